// Row-0 writer, last-row reduction, finalisation and the narrow-boundary
// kernel (arXiv 2608.13110, Sec. 3.1, Algorithm 1).
#include "misc_kernels.cuh"

#include <algorithm>

namespace tb {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {  // a*b + c
    return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}

__device__ __forceinline__ float2 cmac2m(float2 g0, float2 a, float2 g1, float2 b) {
    float2 r;
    r.x = fmaf(g0.x, a.x, fmaf(-g0.y, a.y, fmaf(g1.x, b.x, -g1.y * b.y)));
    r.y = fmaf(g0.x, a.y, fmaf(g0.y, a.x, fmaf(g1.x, b.y, g1.y * b.x)));
    return r;
}

__device__ __forceinline__ int rescale_exp_m(float m) {
    if (!(m > 0.0f) || !isfinite(m)) return 0;
    int e;
    frexpf(m, &e);
    return max(-100, min(100, -e));
}

__device__ __forceinline__ void flush_max_m(float m, uint32_t* dst) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) atomicMax(dst, __float_as_uint(m));
}

// ---------------------------------------------------------------------------
// Row 0 (B <- pi[1]): B_0[s] = a0[s_0] prod_(p>=1) M_p[s_p, s_(p-1)] E_x[s_(h-1)],
// factored as low[s_low] * mid[s_(k-1)][s_mid] * top[x][s_(k+m-1)][s_top].
// One chunk = the 2^k entries sharing their high bits.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) init_kernel(const InitParams p) {
    const int64_t cmask = ((int64_t)1 << p.chunk_shift) - 1;
    const int nk = 1 << p.k;
    float runmax = 0.0f;
    int64_t cur_b = -1;
    for (int64_t g = blockIdx.x; g < p.nchunks; g += gridDim.x) {
        const int64_t b = g >> p.chunk_shift;
        const int64_t c = g & cmask;
        if (b != cur_b) {
            if (cur_b >= 0) flush_max_m(runmax, p.maxs + cur_b * p.sstride);
            runmax = 0.0f;
            cur_b = b;
        }
        const int x = p.bits[b * p.n] ? 1 : 0;
        const int64_t sm = c & (((int64_t)1 << p.m) - 1);
        const int64_t st = c >> p.m;
        const int bm = (int)((sm >> (p.m - 1)) & 1);
        const float2 tv = p.topt[(((int64_t)(x * 2 + bm)) << p.top) + st];
        const float2 g0 = cmul(p.mid[sm], tv);
        const float2 g1 = cmul(p.mid[((int64_t)1 << p.m) + sm], tv);
        float2* dst = p.B + b * p.b_stride + (c << p.k);
        for (int e = threadIdx.x; e < nk; e += blockDim.x) {
            const float2 v = cmul(p.low[e], ((e >> (p.k - 1)) & 1) ? g1 : g0);
            dst[e] = v;
            runmax = fmaxf(runmax, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
    }
    if (cur_b >= 0) flush_max_m(runmax, p.maxs + cur_b * p.sstride);
}

cudaError_t launch_init(const InitParams& p, int grid, cudaStream_t st) {
    init_kernel<<<grid, 256, 0, st>>>(p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Last row: psi = sum_s B[s] V[s], V[s] = top[x][s_top] . mid[s_mid] . low[s_low]
// (row vector . 2x2 . column vector). FP32 within a chunk, FP64 across chunks
// and blocks; partial sums in a fixed order (deterministic).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double2 block_sum_d2(double2 v, double2* red) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    double2 s = make_double2(0.0, 0.0);
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) { s.x += red[i].x; s.y += red[i].y; }
    return s;  // valid in thread 0
}

// The 2^k column vectors (64 KB) are staged once per CTA, which then works off
// many partial sums: with one CTA per partial sum the staging read twice the
// bytes of the boundary itself (n=30, d=40, 32 bitstrings, 8192 chunks:
// 0.246 ms at 1.1 TB/s -> 0.070 ms, zero chunks left out; n=28, d=42, 16
// bitstrings, none zero: 0.244 -> 0.074 ms, 3.6 TB/s).
__global__ void __launch_bounds__(REDUCE_THREADS) reduce_kernel(const __grid_constant__ ReduceParams p) {
    extern __shared__ float4 slow[];  // [2^k]: both components of a column vector
    __shared__ double2 red[2][REDUCE_THREADS / 32];
    const int nk = 1 << p.k;
    const uint32_t lane = threadIdx.x & 31u, col = tile_col(p.skip, lane);
    for (int i = threadIdx.x; i < nk; i += blockDim.x) slow[i] = reinterpret_cast<const float4*>(p.low)[i];
    grid_release();
    grid_wait();
    __syncthreads();
    const int64_t nchunks = (int64_t)1 << p.chunk_shift;
    const int64_t mmask = ((int64_t)1 << p.m) - 1;
    int turn = 0;
    for (int part = blockIdx.x; part < p.nbatch * p.blocks_per_b; part += gridDim.x, turn ^= 1) {
        const int b = part / p.blocks_per_b;
        const int j = part - b * p.blocks_per_b;
        const int x = p.bits[(int64_t)b * p.n + p.n - 1] ? 1 : 0;
        const int s = rescale_exp_m(__uint_as_float(p.maxs[b * p.sstride + p.slot]));
        if (j == 0 && threadIdx.x == 0) p.exps[b * p.sstride + p.slot + 1] = s;
        const double sc = ldexp(1.0, s);
        double ar = 0.0, ai = 0.0;
        for (int64_t u = j; u < nchunks; u += p.blocks_per_b) {
            const int64_t c = tile_of_warp(p.skip.base, col, lane, (uint32_t)u);
            const int64_t sm = c & mmask, stp = c >> p.m;
            const float2* tv = p.topt + ((((int64_t)x << p.top) + stp) << 1);
            const float2* md = p.mid + (sm << 2);
            const float2 r0 = cfma(tv[1], md[2], cmul(tv[0], md[0]));
            const float2 r1 = cfma(tv[1], md[3], cmul(tv[0], md[1]));
            const float2* src = p.B + (int64_t)b * p.b_stride + (c << p.k);
            float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
            // 16 independent loads in flight per thread, then the products
            for (int e0 = threadIdx.x; e0 < nk; e0 += 16 * REDUCE_THREADS) {
                float2 v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int e = e0 + i * REDUCE_THREADS;
                    v[i] = e < nk ? __ldcs(src + e) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const int e = e0 + i * REDUCE_THREADS;
                    if (e < nk) {
                        const float4 w = slow[e];
                        a0 = cfma(v[i], make_float2(w.x, w.y), a0);
                        a1 = cfma(v[i], make_float2(w.z, w.w), a1);
                    }
                }
            }
            const float2 cv = cfma(r1, a1, cmul(r0, a0));
            ar += (double)cv.x;
            ai += (double)cv.y;
        }
        // two scratch rows: a row is written again only after the next sum's barrier
        const double2 tot = block_sum_d2(make_double2(ar * sc, ai * sc), red[turn]);
        if (threadIdx.x == 0) p.partials[part] = tot;
    }
}

cudaError_t launch_reduce(const ReduceParams& p, int nsm, cudaStream_t st) {
    const int smem = (2 << p.k) * (int)sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(reduce_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::min(p.nbatch * p.blocks_per_b, 3 * nsm);  // three CTAs of 64 KB per SM
    return launch_after(reduce_kernel, grid, REDUCE_THREADS, smem, st, p);
}

// psi_b = (sum of its partials) * 2^-(sum of its rescaling exponents).
__global__ void finalize_kernel(const FinalizeParams p) {
    grid_wait();
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int l = threadIdx.x & 31;
    if (b >= p.nbatch) return;
    double sr = 0.0, si = 0.0;
    for (int i = l; i < p.blocks_per_b; i += 32) {
        const double2 v = p.partials[(int64_t)b * p.blocks_per_b + i];
        sr += v.x;
        si += v.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, off);
        si += __shfl_xor_sync(0xffffffffu, si, off);
    }
    int e = 0;  // |exponent| <= 100 per slot
    for (int i = l; i < p.nslots; i += 32) e += p.exps[b * p.sstride + i];
    const long long S = __reduce_add_sync(0xffffffffu, e);
    if (l == 0) {
        const int Si = (int)max(-1000000LL, min(1000000LL, S));
        p.out[2 * b] = scalbn(sr, -Si);
        p.out[2 * b + 1] = scalbn(si, -Si);
    }
}

// ---- log-XEB (Sec. 5.2, normalized log-XEB estimator) -----------------------
// F = gamma + n ln 2 + (1/N) sum_i ln |amp_i|^2, entirely in FP64 on the
// device. One CTA: thread t sums the terms i = t, t + 1024, ... in index
// order, then a fixed binary tree adds the 1024 partial sums, so the result
// does not depend on scheduling. A zero amplitude contributes -inf.
constexpr int XEB_THREADS = 1024;

__global__ void __launch_bounds__(XEB_THREADS) log_xeb_kernel(const double2* amp, int64_t nb, int n, double* out) {
    __shared__ double part[XEB_THREADS];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < nb; i += XEB_THREADS) {
        const double2 a = amp[i];
        s += log(fma(a.x, a.x, a.y * a.y));
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = XEB_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double gamma = 0.57721566490153286060651209;  // Euler's constant
        out[0] = gamma + (double)n * 0.69314718055994530941723212 + part[0] / (double)nb;
    }
}

cudaError_t launch_log_xeb(const double2* amp, int64_t nb, int n, double* out, cudaStream_t st) {
    log_xeb_kernel<<<1, XEB_THREADS, 0, st>>>(amp, nb, n, out);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeParams& p, cudaStream_t st) {
    const int warps = 4;
    return launch_after(finalize_kernel, (p.nbatch + warps - 1) / warps, 32 * warps, 0, st, p);
}

// ---------------------------------------------------------------------------
// Narrow boundaries (h <= 12): one CTA per bitstring runs the whole sweep, row
// 0, every paired step of rows 1..n-2 in order, the last-row contraction, with
// the boundary on chip. Every step evaluates, for both of its outputs,
//   re = fma(g0r, ar, fma(-g0i, ai, fma(g1r, br, -g1i br))), a = in[s=0], b = in[s=1]
// (and im alike), whatever the layout below.
// ---------------------------------------------------------------------------

// Window bits at width h. few: the bitstrings fit one CTA per SM, so the length
// of one sweep counts (fewer entries per thread, more warps); otherwise the
// FP32 pipe counts (more steps per window). Measured with 1 / 128 / 256 / 512 / 2048
// bitstrings at n = 45 (us): width 10 with RW = 2 62 / 62 / 82 / 137 / 432, 3 86 / 105 /
// 105 / 128 / 395; width 11 with RW = 2 100 / 101 / 161 / 312 / 1055, 3 88 / 111 / 136 /
// 255 / 810; width 12 with RW = 3 142 / 144 / 250 / 485 / 1649, 4 142 / 180 / 239 / 488 /
// 1782. At width 9 RW = 3 took 105 instead of 59 with one bitstring; at width 8 it
// would leave half a warp.
constexpr int narrow_rw(int h, bool few) { return h <= 10 ? 2 : h == 11 ? (few ? 2 : 3) : (few ? 3 : 4); }
constexpr int narrow_threads(int h, bool few) { return h < 8 ? 32 : 1 << (h - narrow_rw(h, few) - 1); }

// --- 8 <= h <= 12: register windows ----------------------------------------
// A thread holds 2^(RW+1) entries in registers: RW consecutive address bits
// (the window) and one spectator bit v whose two values share a packed pair
// (paired FP32 FMA, coefficients broadcast). The steps whose targets lie in
// the window are register arithmetic; the boundary goes through shared memory
// only when the window moves. The targets walk 0..h-1 and back, so the windows
// at the two ends serve the steps before and after the turn: per two rows four
// windows (h = 12, RW = 4: 8 + 4 + 8 + 4 steps) where every single step used
// to read and write shared memory behind a barrier. What bounds it: FP32 issue
// (8 FMA per entry and step) once every SM has two warps per scheduler, the
// chain of window moves and steps below that. n = 45, us for 1 / 256 / 2048
// bitstrings, one step per barrier -> this form: width 8 144 / 154 / 457 ->
// 49 / 49 / 109, width 10 236 / 279 / 1235 -> 62 / 82 / 432, width 11
// 360 / 456 / 2355 -> 97 / 136 / 809, width 12 599 / 818 / 4775 -> 142 / 240 / 1782.
// Power-of-two rescaling (exact) at every turn, folded into the next window's
// first coefficients. Two things about that want gates near a unit scale: a
// coefficient times the scale may leave FP32's range although its products do not
// (growth by 2^80, then a gate of 2^-80), and a turn window runs two rows' steps
// without a rescale. WIDE, for plans with other gates (Plan::wide_range), scales the
// entries as the next window loads them and rescales between the rows of a turn
// window too. A form of its own: scaling entries alone cost the ordinary plans 10 %
// at width 8 and 8 % at width 10 with one bitstring.
template <int H, int RW>
struct Narrow {
    static constexpr int T = 1 << (H - RW - 1);  // threads
    static constexpr int NK = 1 << RW;           // packed pairs per thread
    static constexpr int NW = (T + 31) / 32;
    static_assert(H > 2 * RW, "a window between the two turn windows takes the rescale");
    // spectator bit of the window [lo, lo + RW): neither in it nor next to it,
    // and not among the lowest bits, which the lanes hold
    static constexpr int vbit(int lo) { return lo + RW + 1 <= H - 1 ? H - 1 : lo - 2; }
    // shared-memory slot: 16 lanes that differ in the four lowest address bits
    // outside any window fall into 16 different 8-byte banks
    static constexpr uint32_t swz(uint32_t a) { return a ^ ((a >> RW) & 15u); }
    // thread bits fill the address bits other than the window's and v, ascending
    __device__ static __forceinline__ uint32_t thread_addr(int lo, uint32_t t) {
        const int v = vbit(lo), below = v < lo ? v : lo;
        uint32_t a = t & ((1u << below) - 1u);
        t >>= below;
        if (v < lo) {  // bit lo - 1 above v
            a |= (t & 1u) << (lo - 1);
            t >>= 1;
        }
        return a | (t << (lo + RW));
    }
};

constexpr int NARROW_CF = 24;  // packed coefficients per step: [c][g00r g00i -g00i g01r .. -g11i]

__device__ __forceinline__ float2 nfma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

template <int N>
__device__ __forceinline__ void narrow_cf(float2 (&c)[N], const float2* src) {
    const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float4 q = s4[i];
        c[2 * i] = make_float2(q.x, q.y);
        c[2 * i + 1] = make_float2(q.z, q.w);
    }
}

// Step on register bit K; CK: control register bit, -1: cf holds the block of
// this thread's control value (or the step has no control).
template <bool SC, int NK, int K, int CK>
__device__ __forceinline__ void narrow_step(float2 (&P)[NK], float2 (&Q)[NK], const float2* cf, float s) {
#pragma unroll
    for (int cv = 0; cv < (CK >= 0 ? 2 : 1); ++cv) {
        float2 c[12];
        narrow_cf(c, cf + 12 * cv);
        if constexpr (SC) {
#pragma unroll
            for (int i = 0; i < 12; ++i) c[i] = __fmul2_rn(c[i], make_float2(s, s));
        }
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            if (k & (1 << K)) continue;
            if (CK >= 0 && ((k >> (CK < 0 ? 0 : CK)) & 1) != cv) continue;
            const int k1 = k | (1 << K);
            const float2 aP = P[k], aQ = Q[k], bP = P[k1], bQ = Q[k1];
            P[k] = nfma2(c[0], aP, nfma2(c[2], aQ, nfma2(c[3], bP, __fmul2_rn(c[5], bQ))));
            Q[k] = nfma2(c[0], aQ, nfma2(c[1], aP, nfma2(c[3], bQ, __fmul2_rn(c[4], bP))));
            P[k1] = nfma2(c[6], aP, nfma2(c[8], aQ, nfma2(c[9], bP, __fmul2_rn(c[11], bQ))));
            Q[k1] = nfma2(c[6], aQ, nfma2(c[7], aP, nfma2(c[9], bQ, __fmul2_rn(c[10], bP))));
        }
    }
}

// SC: the coefficients of the first step carry the rescale s.
// Forward targets T0 .. T0+N-1 (register bits of the window at lo); cf: the
// row's coefficients, step of target t at cf + t * NARROW_CF.
template <bool SC, int NK, int LO, int T0, int N>
__device__ __forceinline__ void narrow_fwd(float2 (&P)[NK], float2 (&Q)[NK], const float2* cf, uint32_t addr, float s) {
    if constexpr (N > 0) {
        const float2* c = cf + T0 * NARROW_CF;
        if constexpr (T0 == LO) {
            if (T0 > 0 && ((addr >> (T0 > 0 ? T0 - 1 : 0)) & 1u)) c += 12;
            narrow_step<SC, NK, 0, -1>(P, Q, c, s);
        } else {
            narrow_step<SC, NK, T0 - LO, T0 - LO - 1>(P, Q, c, s);
        }
        narrow_fwd<false, NK, LO, T0 + 1, N - 1>(P, Q, cf, addr, 1.0f);
    }
}

// Reversed targets T0, T0-1, .. (N of them); step of target t at cf + (H-1-t) * NARROW_CF.
template <bool SC, int NK, int RW, int H, int LO, int T0, int N>
__device__ __forceinline__ void narrow_rev(float2 (&P)[NK], float2 (&Q)[NK], const float2* cf, uint32_t addr, float s) {
    if constexpr (N > 0) {
        const float2* c = cf + (H - 1 - T0) * NARROW_CF;
        if constexpr (T0 == LO + RW - 1) {
            if (T0 < H - 1 && ((addr >> (T0 + 1)) & 1u)) c += 12;
            narrow_step<SC, NK, T0 - LO, -1>(P, Q, c, s);
        } else {
            narrow_step<SC, NK, T0 - LO, T0 - LO + 1>(P, Q, c, s);
        }
        narrow_rev<false, NK, RW, H, LO, T0 - 1, N - 1>(P, Q, cf, addr, 1.0f);
    }
}

template <int H, int RW, bool WIDE>
struct NarrowRun {
    using W = Narrow<H, RW>;
    static constexpr int NK = W::NK, T = W::T;
    static constexpr int ROW_CF = H * NARROW_CF;       // a row's packed coefficients
    static constexpr int CYCLE = 2 * H * 8;            // raw coefficients of two rows
    static constexpr int PRE = (CYCLE + T - 1) / T;    // of which a thread stages this many
    // The last row's FP64 sum has one grouping for both forms, so that an amplitude
    // does not depend on how many bitstrings share the call: T0 sums (the threads of
    // the many-bitstring form) of STRANDS strided sums each, a thread's own there and
    // one per thread here when this form has more threads.
    static constexpr int T0 = narrow_threads(H, false), STRANDS = narrow_threads(H, true) / T0, OWN = STRANDS * T0 / T;
    static_assert(T == T0 || OWN == 1, "a thread holds all strands of its sum or one of them");
    float2* Bs;
    float2* cf;     // [2 buffers][2 rows][H][NARROW_CF]
    float* red;     // [2][NW]
    const SmallParams& p;
    const uint8_t* xb;
    uint32_t t;
    long long S;
    float2 pre[PRE];

    __device__ __forceinline__ void sync() const {
        if constexpr (T <= 32) __syncwarp(T == 32 ? 0xffffffffu : (1u << T) - 1u);
        else asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
    }
    // coefficients of rows 2 cyc and 2 cyc + 1: global memory -> registers -> shared memory
    __device__ __forceinline__ void fetch(int cyc) {
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int w = i * T + (int)t, st = 2 * H * cyc + (w >> 3);
            if (w < CYCLE && st < p.nrows * H) {
                const int q = p.xq[st];
                pre[i] = p.steps[st].g[q >= 0 && xb[q] ? 1 : 0][w & 7];
            }
        }
    }
    __device__ __forceinline__ void stage(int cyc) {
        float2* dst = cf + (cyc & 1) * 2 * ROW_CF;
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int w = i * T + (int)t;
            if (w < CYCLE) {
                float2* o = dst + (w >> 3) * NARROW_CF + 3 * (w & 7);
                o[0] = make_float2(pre[i].x, pre[i].x);
                o[1] = make_float2(pre[i].y, pre[i].y);
                o[2] = make_float2(-pre[i].y, -pre[i].y);
            }
        }
    }
    template <int LO>
    __device__ __forceinline__ uint32_t addr() const { return W::thread_addr(LO, t); }
    template <int LO>
    __device__ __forceinline__ void load(float2 (&P)[NK], float2 (&Q)[NK]) const {
        const uint32_t b = W::swz(addr<LO>());
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const float2 lo = Bs[b ^ W::swz((uint32_t)k << LO)];
            const float2 hi = Bs[b ^ W::swz((uint32_t)k << LO) ^ W::swz(1u << W::vbit(LO))];
            P[k] = make_float2(lo.x, hi.x);
            Q[k] = make_float2(lo.y, hi.y);
        }
    }
    template <int LO>
    __device__ __forceinline__ void store(const float2 (&P)[NK], const float2 (&Q)[NK]) const {
        const uint32_t b = W::swz(addr<LO>());
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            Bs[b ^ W::swz((uint32_t)k << LO)] = make_float2(P[k].x, Q[k].x);
            Bs[b ^ W::swz((uint32_t)k << LO) ^ W::swz(1u << W::vbit(LO))] = make_float2(P[k].y, Q[k].y);
        }
    }
    // this turn's maximum, for the scale every thread takes after the next sync
    __device__ __forceinline__ void put_max(float m, int turn) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if ((t & 31) == 0) red[(turn & 1) * W::NW + (t >> 5)] = m;
    }
    __device__ __forceinline__ float reg_max(const float2 (&P)[NK], const float2 (&Q)[NK]) const {
        float m = 0.0f;
#pragma unroll
        for (int k = 0; k < NK; ++k)
            m = fmaxf(m, fmaxf(fmaxf(fabsf(P[k].x), fabsf(P[k].y)), fmaxf(fabsf(Q[k].x), fabsf(Q[k].y))));
        return m;
    }
    __device__ __forceinline__ float take_scale(int turn) {
        float m = 0.0f;
#pragma unroll
        for (int i = 0; i < W::NW; ++i) m = fmaxf(m, red[(turn & 1) * W::NW + i]);
        const int s = rescale_exp_m(m);
        S += s;
        return ldexpf(1.0f, s);
    }
    __device__ __forceinline__ static void scale_by(float2 (&P)[NK], float2 (&Q)[NK], float s) {
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            P[k] = __fmul2_rn(P[k], make_float2(s, s));
            Q[k] = __fmul2_rn(Q[k], make_float2(s, s));
        }
    }
    // WIDE: rescale in registers, between the two rows of a turn window
    __device__ __forceinline__ void rescale_row(float2 (&P)[NK], float2 (&Q)[NK], int& turn) {
        if constexpr (WIDE) {
            put_max(reg_max(P, Q), ++turn);
            sync();
            scale_by(P, Q, take_scale(turn));
        }
    }
    // targets of the middle windows, RW at a time; SC: the first one is rescaled
    template <bool SC, int T0>
    __device__ __forceinline__ void mid_fwd(const float2* c, float s) {
        if constexpr (T0 < H - RW) {
            constexpr int N = (H - RW - T0) < RW ? (H - RW - T0) : RW;
            float2 P[NK], Q[NK];
            load<T0>(P, Q);
            if constexpr (SC && WIDE) scale_by(P, Q, s);
            narrow_fwd<SC && !WIDE, NK, T0, T0, N>(P, Q, c, addr<T0>(), s);
            store<T0>(P, Q);
            sync();
            mid_fwd<false, T0 + N>(c, 1.0f);
        }
    }
    template <bool SC, int T0>
    __device__ __forceinline__ void mid_rev(const float2* c, float s) {
        if constexpr (T0 >= RW) {
            constexpr int N = (T0 - RW + 1) < RW ? (T0 - RW + 1) : RW;
            constexpr int LO = T0 - RW + 1;
            float2 P[NK], Q[NK];
            load<LO>(P, Q);
            if constexpr (SC && WIDE) scale_by(P, Q, s);
            narrow_rev<SC && !WIDE, NK, RW, H, LO, T0, N>(P, Q, c, addr<LO>(), s);
            store<LO>(P, Q);
            sync();
            mid_rev<false, T0 - N>(c, 1.0f);
        }
    }

    __device__ void run(int b, double2* redd) {
        constexpr int N = 1 << H, TOP = H - RW;
        const int x0 = xb[0] ? 1 : 0;
        float m = 0.0f;
        fetch(0);
        for (int e = (int)t; e < N; e += T) {
            const float2 v = cmul(p.init_low[e], p.init_top[x0 * 2 + ((e >> (H - 1)) & 1)]);
            Bs[W::swz((uint32_t)e)] = v;
            m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
        stage(0);
        put_max(m, 0);
        sync();
        int row = 0, turn = 0;
        float s = take_scale(0);
        if (p.nrows > 0) {
            float2 P[NK], Q[NK];
            load<0>(P, Q);
            scale_by(P, Q, s);
            for (int cyc = 0;; ++cyc) {
                const float2* c = cf + (cyc & 1) * 2 * ROW_CF;
                fetch(cyc + 1);
                narrow_fwd<false, NK, 0, 0, RW>(P, Q, c, 0u, 1.0f);
                put_max(reg_max(P, Q), ++turn);
                store<0>(P, Q);
                sync();
                s = take_scale(turn);
                mid_fwd<true, RW>(c, s);
                load<TOP>(P, Q);
                narrow_fwd<false, NK, TOP, TOP, RW>(P, Q, c, addr<TOP>(), 1.0f);
                if (++row == p.nrows) {
                    put_max(reg_max(P, Q), ++turn);
                    store<TOP>(P, Q);
                    break;
                }
                rescale_row(P, Q, turn);
                narrow_rev<false, NK, RW, H, TOP, H - 1, RW>(P, Q, c + ROW_CF, 0u, 1.0f);
                put_max(reg_max(P, Q), ++turn);
                store<TOP>(P, Q);
                stage(cyc + 1);
                sync();
                s = take_scale(turn);
                mid_rev<true, H - RW - 1>(c + ROW_CF, s);
                load<0>(P, Q);
                narrow_rev<false, NK, RW, H, 0, RW - 1, RW>(P, Q, c + ROW_CF, addr<0>(), 1.0f);
                if (++row == p.nrows) {
                    put_max(reg_max(P, Q), ++turn);
                    store<0>(P, Q);
                    break;
                }
                rescale_row(P, Q, turn);
            }
            sync();
            s = take_scale(turn);
        }
        const int xl = xb[p.n - 1] ? 1 : 0;
        double ar[OWN] = {}, ai[OWN] = {};
        for (int e0 = (int)t; e0 < N; e0 += OWN * T) {
#pragma unroll
            for (int g = 0; g < OWN; ++g) {
                const int e = e0 + g * T;
                const float2 z = Bs[W::swz((uint32_t)e)];
                const float2 v = cmul(make_float2(z.x * s, z.y * s), p.red_low[2 * e + xl]);
                ar[g] += (double)v.x;
                ai[g] += (double)v.y;
            }
        }
#pragma unroll
        for (int g = 1; g < OWN; ++g) { ar[0] += ar[g]; ai[0] += ai[g]; }
        if constexpr (T > T0) {  // the other strands, through the coefficients' memory (no step is left)
            double2* strand = reinterpret_cast<double2*>(cf);
            if (t >= T0) strand[t - T0] = make_double2(ar[0], ai[0]);
            sync();
            if (t < T0)
#pragma unroll
                for (int g = 1; g < STRANDS; ++g) {
                    const double2 o = strand[(g - 1) * T0 + t];
                    ar[0] += o.x;
                    ai[0] += o.y;
                }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            ar[0] += __shfl_xor_sync(0xffffffffu, ar[0], off);
            ai[0] += __shfl_xor_sync(0xffffffffu, ai[0], off);
        }
        if (t < T0 && (t & 31) == 0) redd[t >> 5] = make_double2(ar[0], ai[0]);
        sync();
        if (t == 0) {
            double2 tot = redd[0];
            for (int i = 1; i < T0 / 32; ++i) { tot.x += redd[i].x; tot.y += redd[i].y; }
            const int Si = (int)max(-1000000LL, min(1000000LL, S));
            p.out[2 * b] = scalbn(tot.x, -Si);
            p.out[2 * b + 1] = scalbn(tot.y, -Si);
        }
    }
};

// --- h <= 7: one warp, address bits 0..4 on the lanes, the rest in registers --
// A step on a lane bit takes the partner's entry by shuffle. Each lane loads the
// coefficient rows of its own outputs a group of rows ahead, with the output
// bits already in registers, so a row waits for its own chain and not for a
// chain of loads (width 4, 64 bitstrings: 8.1 -> 5.0 us at n = 12, 25.4 -> 12.4
// us at n = 45; width 7, n = 45: 47 -> 32 us; a CTA and a barrier per step took
// longer than either).
template <int H>
__device__ void narrow_warp(const SmallParams& p, int b) {
    constexpr int LB = H < 5 ? H : 5, R = H > 5 ? 1 << (H - 5) : 1;
    constexpr int D = H <= 4 ? 4 : H == 5 ? 3 : H == 6 ? 2 : 1;  // rows per group
    const uint32_t lane = threadIdx.x & 31u;
    const uint8_t* xb = p.bits + (int64_t)b * p.n;
    const bool live = lane < (1u << LB);
    uint32_t xm[4];  // output bits 0..127
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int q = 32 * j + (int)lane;
        xm[j] = __ballot_sync(0xffffffffu, q < p.n && xb[q < p.n ? q : 0] != 0);
    }
    auto xbit = [&](int q) -> int {
        if (q >= 128) return xb[q] ? 1 : 0;
        const uint32_t lo = q & 32 ? xm[1] : xm[0], hi = q & 32 ? xm[3] : xm[2];
        return (int)((q & 64 ? hi : lo) >> (q & 31) & 1u);
    };
    // Coefficients of a group of rows: for every target, this lane's output
    // rows. A register target or control needs more than one: [register control
    // or target value][2 entries]. Only the step on the highest bit depends on
    // an output bit, its row's.
    constexpr int NC = R > 1 ? 4 : 1;
    float4 cur[D][H][NC], nxt[D][H][NC];
    auto fetch = [&](int row0, float4 (&o)[D][H][NC]) {
#pragma unroll
        for (int r = 0; r < D; ++r) {
            const int row = row0 + r;
            if (row >= p.nrows) return;
            const bool fwd = (row & 1) == 0;  // row 0 here is the circuit's row 1
#pragma unroll
            for (int tg = 0; tg < H; ++tg) {
                const int st = row * H + (fwd ? tg : H - 1 - tg);
                // 8-byte loads: a caller's workspace need not be aligned to 16
                const float2* g = p.steps[st].g[tg == H - 1 ? xbit(row + 1) : 0];
                const int ct = fwd ? tg - 1 : tg + 1;  // control bit (outside 0..H-1: none)
                const bool cin = ct >= 0 && ct < H;
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const int ap = tg < LB ? (int)(lane >> tg & 1u) : (i & 1);
                    const int c = !cin ? 0 : ct < LB ? (int)(lane >> (ct < 0 ? 0 : ct) & 1u) : (i >> 1);
                    const float2 g0 = g[c * 4 + ap * 2], g1 = g[c * 4 + ap * 2 + 1];
                    o[r][tg][i] = make_float4(g0.x, g0.y, g1.x, g1.y);
                }
            }
        }
    };
    fetch(0, cur);
    float2 v[R];
    const int x0 = xbit(0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t e = (lane & ((1u << LB) - 1u)) | ((uint32_t)r << LB);
        v[r] = live ? cmul(p.init_low[e], p.init_top[x0 * 2 + ((e >> (H - 1)) & 1)]) : make_float2(0.f, 0.f);
    }
    long long S = 0;
    auto rescale = [&]() {
        float m = 0.0f;
#pragma unroll
        for (int r = 0; r < R; ++r) m = fmaxf(m, fmaxf(fabsf(v[r].x), fabsf(v[r].y)));
        // non-negative floats compare like their bits
        const int s = rescale_exp_m(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m))));
        const float sc = ldexpf(1.0f, s);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = make_float2(v[r].x * sc, v[r].y * sc);
        S += s;
    };
    rescale();
    auto out = [](float4 g, float2 a, float2 bb) {
        return cmac2m(make_float2(g.x, g.y), a, make_float2(g.z, g.w), bb);
    };
    auto step = [&](int tg, int ct, const float4 (&g)[NC]) {
        if (tg < LB) {
            const bool hi = (lane >> tg & 1u) != 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float2 o;
                o.x = __shfl_xor_sync(0xffffffffu, v[r].x, 1 << tg);
                o.y = __shfl_xor_sync(0xffffffffu, v[r].y, 1 << tg);
                const int c = (ct >= LB && ct < H) ? (r >> (ct - LB)) & 1 : 0;  // register control
                v[r] = out(g[NC > 1 ? 2 * c : 0], hi ? o : v[r], hi ? v[r] : o);
            }
        } else {
            const int K = tg - LB;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (r & (1 << K)) continue;
                const int r1 = (r | (1 << K)) & (R - 1);
                const int c = (ct >= LB && ct < H) ? (r >> (ct - LB)) & 1 : 0;
                const float2 a = v[r], bb = v[r1];
                v[r] = out(g[NC > 1 ? 2 * c : 0], a, bb);
                v[r1] = out(g[NC > 1 ? 2 * c + 1 : 0], a, bb);
            }
        }
    };
    for (int row0 = 0; row0 < p.nrows; row0 += D) {
        fetch(row0 + D, nxt);
#pragma unroll
        for (int r = 0; r < D; ++r) {
            if (row0 + r >= p.nrows) break;
            if (((row0 + r) & 1) == 0) {
#pragma unroll
                for (int tg = 0; tg < H; ++tg) step(tg, tg - 1, cur[r][tg]);
            } else {
#pragma unroll
                for (int tg = H - 1; tg >= 0; --tg) step(tg, tg + 1, cur[r][tg]);
            }
            rescale();
        }
#pragma unroll
        for (int r = 0; r < D; ++r)
#pragma unroll
            for (int tg = 0; tg < H; ++tg)
#pragma unroll
                for (int i = 0; i < NC; ++i) cur[r][tg][i] = nxt[r][tg][i];
    }
    const int xl = xbit(p.n - 1);
    double ar = 0.0, ai = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t e = (lane & ((1u << LB) - 1u)) | ((uint32_t)r << LB);
        const float2 w = live ? cmul(v[r], p.red_low[2 * e + xl]) : make_float2(0.f, 0.f);
        ar += (double)w.x;
        ai += (double)w.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ar += __shfl_xor_sync(0xffffffffu, ar, off);
        ai += __shfl_xor_sync(0xffffffffu, ai, off);
    }
    if (lane == 0) {
        const int Si = (int)max(-1000000LL, min(1000000LL, S));
        p.out[2 * b] = scalbn(ar, -Si);
        p.out[2 * b + 1] = scalbn(ai, -Si);
    }
}

constexpr int narrow_smem(int h, bool few) {  // boundary, coefficients, reduction scratch of every warp
    return h < 8 ? 0 : (8 << h) + 2 * 2 * h * NARROW_CF * 8 + (narrow_threads(h, false) / 32) * 16 +
                           (narrow_threads(h, few) / 32) * 8;
}

template <int H, bool FEW, bool WIDE>
__device__ __forceinline__ void narrow_sweep(const SmallParams& p, int b, uint8_t* smem) {
    if constexpr (H < 8) {
        if (threadIdx.x < 32) narrow_warp<H>(p, b);
    } else {
        using R = NarrowRun<H, narrow_rw(H, FEW), WIDE>;
        static_assert(R::T >= 32 && R::T0 >= 32, "whole warps");
        static_assert((R::T - R::T0) * 16 <= 2 * 2 * R::ROW_CF * 8, "strands fit the coefficients' memory");
        if (threadIdx.x >= R::T) return;
        float2* Bs = reinterpret_cast<float2*>(smem);
        float2* cf = Bs + (1 << H);
        double2* redd = reinterpret_cast<double2*>(cf + 2 * 2 * R::ROW_CF);  // [T0 / 32], then red [2][NW]
        R r{Bs, cf, reinterpret_cast<float*>(redd + R::T0 / 32), p, p.bits + (int64_t)b * p.n, threadIdx.x, 0, {}};
        r.run(b, redd);
    }
}

template <int H, bool FEW, bool WIDE>
__global__ void __launch_bounds__(narrow_threads(H, FEW)) narrow_kernel(const __grid_constant__ SmallParams p) {
    extern __shared__ __align__(16) uint8_t nsm[];
    narrow_sweep<H, FEW, WIDE>(p, blockIdx.x, nsm);
}

// Several narrow plans in one launch: block i evaluates bitstring
// i - first_block of the item whose block range holds i.
constexpr int NARROW_MULTI_THREADS = 128;
static_assert(narrow_threads(12, false) <= NARROW_MULTI_THREADS && narrow_threads(11, false) <= NARROW_MULTI_THREADS &&
                  narrow_threads(10, false) <= NARROW_MULTI_THREADS, "one CTA size for every width");
__global__ void __launch_bounds__(NARROW_MULTI_THREADS) narrow_multi_kernel(const SmallItem* items, int nitems) {
    extern __shared__ __align__(16) uint8_t nsm[];
    int lo = 0, hi = nitems - 1;
    const int64_t blk = blockIdx.x;
    while (lo < hi) {  // last item with first_block <= blk
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].first_block <= blk) lo = mid;
        else hi = mid - 1;
    }
    const SmallParams p = items[lo].p;
    const int b = (int)(blk - items[lo].first_block);
    switch (p.h) {
        case 1: narrow_sweep<1, false, false>(p, b, nsm); break;
        case 2: narrow_sweep<2, false, false>(p, b, nsm); break;
        case 3: narrow_sweep<3, false, false>(p, b, nsm); break;
        case 4: narrow_sweep<4, false, false>(p, b, nsm); break;
        case 5: narrow_sweep<5, false, false>(p, b, nsm); break;
        case 6: narrow_sweep<6, false, false>(p, b, nsm); break;
        case 7: narrow_sweep<7, false, false>(p, b, nsm); break;
        case 8: p.wide ? narrow_sweep<8, false, true>(p, b, nsm) : narrow_sweep<8, false, false>(p, b, nsm); break;
        case 9: p.wide ? narrow_sweep<9, false, true>(p, b, nsm) : narrow_sweep<9, false, false>(p, b, nsm); break;
        case 10: p.wide ? narrow_sweep<10, false, true>(p, b, nsm) : narrow_sweep<10, false, false>(p, b, nsm); break;
        case 11: p.wide ? narrow_sweep<11, false, true>(p, b, nsm) : narrow_sweep<11, false, false>(p, b, nsm); break;
        case 12: p.wide ? narrow_sweep<12, false, true>(p, b, nsm) : narrow_sweep<12, false, false>(p, b, nsm); break;
        default: break;
    }
}

cudaError_t launch_small_multi(const SmallItem* d_items, int nitems, int64_t nblocks, int hmax, cudaStream_t st) {
    int smem = 0;
    for (int h = 1; h <= hmax; ++h) smem = std::max(smem, narrow_smem(h, false));
    narrow_multi_kernel<<<(unsigned)nblocks, NARROW_MULTI_THREADS, smem, st>>>(d_items, nitems);
    return cudaGetLastError();
}

template <int H, bool WIDE>
cudaError_t launch_form(const SmallParams& p, cudaStream_t st) {
    if (p.nb <= p.nsm) narrow_kernel<H, true, WIDE><<<p.nb, narrow_threads(H, true), narrow_smem(H, true), st>>>(p);
    else narrow_kernel<H, false, WIDE><<<p.nb, narrow_threads(H, false), narrow_smem(H, false), st>>>(p);
    return cudaGetLastError();
}

template <int H>
cudaError_t launch_narrow(const SmallParams& p, cudaStream_t st) {
    if constexpr (H >= 8) {  // narrower boundaries rescale after every row as they are
        if (p.wide) return launch_form<H, true>(p, st);
    }
    return launch_form<H, false>(p, st);
}

cudaError_t launch_small(const SmallParams& p, cudaStream_t st) {
    switch (p.h) {
        case 1: return launch_narrow<1>(p, st);
        case 2: return launch_narrow<2>(p, st);
        case 3: return launch_narrow<3>(p, st);
        case 4: return launch_narrow<4>(p, st);
        case 5: return launch_narrow<5>(p, st);
        case 6: return launch_narrow<6>(p, st);
        case 7: return launch_narrow<7>(p, st);
        case 8: return launch_narrow<8>(p, st);
        case 9: return launch_narrow<9>(p, st);
        case 10: return launch_narrow<10>(p, st);
        case 11: return launch_narrow<11>(p, st);
        case 12: return launch_narrow<12>(p, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tb
