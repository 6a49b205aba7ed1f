// ppf_bwd_unfused.cuh -- the adjoint of the PFB for every shape the forward
// plans (C = 32 .. 4096 and 3 * 2^k, T up to 64, any input type), as three
// passes over a g_y scratch in device memory.  The fused backward kernel
// (ppf_bwd.cuh) covers C in [64, 512] with T <= 16; outside that its carried
// rows and its G/x batches no longer fit one SM, so the three sums of the
// adjoint (same convention as ppf_bwd.cuh, PyTorch's conjugate Wirtinger
// gradient, G = grad_Y):
//   g_y = F^H G                                   (unnormalised inverse DFT)
//   grad_x[r][c] = sum_{t<T} h[t][c] g_y[r-t][c]  (transposed FIR, Alg. 1)
//   grad_h[t][c] = sum_s Re(conj(g_y[s][c]) x[s+t][c])
// (g_y[s] = 0 outside 0 <= s < S) run as separate kernels:
//   1. the forward kernels with one unit tap and conjugated input and output
//      (conj(F conj(.))) on the rows of G, g_y rows to the scratch (C = 512, 65536
//      rows: 85 us; 120 with a kernel of its own that copied rows in and out
//      between CTA-wide stages);
//   2. pfb_bwd_grad_kernel<IN>: both other sums from one pass over g_y, one
//      thread per channel, a window of kAdjL rows of g_y in registers, rows,
//      samples and taps through a TMA ring; per-part partial sums of grad_h
//      reduced in a fixed order by pfb_bwd_reduce_kernel (deterministic).
// HBM traffic per raw sample is about G 8 + g_y 8 (write) + g_y 8 + grad_x 8 + x;
// the halo re-reads come from L2.
#pragma once

#include "ppf_fwd.cuh"
#include "ppf_tmap.h"

namespace ppf {

// Pass 1 at C = 32, where no forward kernel conjugates: 256 rows of G at a time
// through shared memory, the DFT stages in their inverse mode.  args.in: G,
// args.out: g_y (n_spectra*C per stream, strides as for the forward).
template <int C>
struct IdftShape {
    static constexpr int NT = 256;
    static constexpr int B = 8192 / C;
    static constexpr int YBYTES = B * C * 8;
    static constexpr int SMEM = YBYTES + tw_size(C) * 8;
};

template <int C>
__global__ void __launch_bounds__(IdftShape<C>::NT) pfb_bwd_idft_kernel(FwdArgs a) {
    using S = IdftShape<C>;
    constexpr int NT = S::NT, B = S::B, NST = fft_stages(C);
    extern __shared__ __align__(128) unsigned char smem[];
    float2* ybuf = reinterpret_cast<float2*>(smem);
    float2* tw_s = reinterpret_cast<float2*>(smem + S::YBYTES);
    const int tid = threadIdx.x;
    for (int i = tid; i < tw_size(C); i += NT) tw_s[i] = a.tw[i];
    float4* y4 = reinterpret_cast<float4*>(ybuf);
    BatchShare share((a.n_spectra + B - 1) / B, a.n_streams, blockIdx.x, gridDim.x);
    long long strm, lo, hi;
    while (share.next(strm, lo, hi)) {
        const float4* src = reinterpret_cast<const float4*>(static_cast<const float2*>(a.in) + (size_t)strm * a.in_stride);
        float4* dst = reinterpret_cast<float4*>(static_cast<float2*>(a.out) + (size_t)strm * a.out_stride);
        for (long long k = lo; k < hi; ++k) {
            const long long s0 = k * B;
            const int rows = (int)(a.n_spectra - s0 < B ? a.n_spectra - s0 : B);
            const long long base = s0 * (C / 2);            // float4 index of the batch's first row
            __syncthreads();   // the previous batch's rows have been stored (and the twiddles copied)
            for (int i = tid; i < B * C / 2; i += NT)
                y4[i] = (i < rows * (C / 2)) ? __ldcs(src + base + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
            // inverse mode: the last stage leaves g_y rows in natural order in ybuf, then synchronises
            static_for<NST>([&](auto p) {
                fft_stage<C, B, NT, decltype(p)::value, OUT_CF32, true, 0, true>(ybuf, tw_s, nullptr, 0, 0, 0);
            });
            for (int i = tid; i < rows * (C / 2); i += NT) dst[base + i] = y4[i];
        }
    }
}

// grad_x and the tap correlation in one pass over g_y.  A CTA owns NCT channels
// (one per consumer thread) and a share of the tiles of kAdjL raw rows of all
// streams.  For the tile at raw row r0 a window of kAdjL rows of g_y lives in
// registers; step u (tap t = T-1-u) has rows r0 + j - t, j = 0 .. kAdjL-1, in it,
// so both sums need no other operand:
//   grad_x[r0+j] += h[t] g_y[r0+j-t]                  (kAdjL packed FMAs)
//   grad_h[t]    += sum_j Re(conj(g_y[r0+j-t]) x[r0+j])  (kAdjL packed FMAs)
// then the oldest row leaves the window and row r0 + kAdjL - t enters.  The sum
// over j is added to the thread's column of a [T][NCT] table in shared memory,
// written out once per CTA (partial sums, reduced in a fixed order later).
// A producer warp keeps a ring of chunks filled with boxes of tensor maps: 8
// rows of g_y with 8 rows of x (the window and the tile's samples), then 8
// rows of g_y with 8 taps.  Rows outside a stream read as zeros; ENDS, the form for
// short streams, leaves out the steps that see nothing else (AdjSteps).
// Bound by FP32 issue (2 T packed FMAs per sample, 1.0 clock per sample and SM at
// T = 32; it takes 2.2, 52 % of the FMA pipe) and for few taps by HBM.  The two
// kernels it replaces read g_y once each, the halo five times from L2 (tiles
// of 8 rows), and spent as many instructions on staging as on FMAs: C = 512,
// T = 32, int8, 65536 spectra 457 -> 236 us; the whole adjoint (GS/s) C = 512
// T = 64 33 -> 60, C = 1024 T = 8 FP32 98 -> 128, C = 32 T = 8 50 -> 99.
constexpr int kAdjL = 16;    // raw rows per tile
constexpr int kAdjRC = 8;    // rows (and taps) per chunk
constexpr int kAdjNS = 3;    // ring slots

struct AdjArgs {
    float2* gx;              // grad_x, n_raw*C per stream, streams contiguous (GX)
    float* partials;         // gridDim.x rows of TM*C partial sums (GH)
    int* err;
    long long n_spectra, n_streams;
    int C, T, TM;
    int flags;               // FwdFlags (testing aid)
};

// The steps of a tile: taps t1, t1 - 1, .., n of them.  All T, or (ENDS) the ones whose
// window r0 - t .. r0 - t + kAdjL-1, for the tile at raw row r0, meets rows 0 .. S-1 of
// the stream (at least one does).
struct AdjSteps {
    int t1, n;
    __device__ __forceinline__ explicit AdjSteps(int T) : t1(T - 1), n(T) {}
    __device__ __forceinline__ AdjSteps(long long r0, long long S, int T) {
        t1 = r0 + kAdjL < T ? (int)r0 + kAdjL - 1 : T - 1;
        n = t1 + 1 - (r0 >= S ? (int)(r0 - S) + 1 : 0);
    }
};

struct AdjMaps {
    CUtensorMap g, x, taps;
};

template <int IN, int NCT>
struct AdjShape {
    static constexpr int NT = NCT + 32;
    static constexpr int MINB = NCT == 128 ? 3 : NCT == 64 ? 5 : 8;  // CTAs per SM: at most 16 warps of 128 registers
    static constexpr int BIN = InTraits<IN>::bytes;
    static constexpr int GB = kAdjRC * NCT * 8;                      // a chunk's rows of g_y
    static constexpr int XB = kAdjRC * NCT * (BIN > 4 ? BIN : 4);    // its rows of x, or its taps
    static constexpr int CHUNKB = GB + XB;
    static constexpr int BAR_OFF = kAdjNS * CHUNKB;
    static constexpr int GH_OFF = BAR_OFF + 64;
    static constexpr int smem(int T) { return GH_OFF + T * NCT * 4; }
};

template <int IN, int NCT, bool GX, bool GH, bool ENDS>
__global__ void __launch_bounds__(AdjShape<IN, NCT>::NT, AdjShape<IN, NCT>::MINB)
pfb_bwd_grad_kernel(AdjArgs a, const __grid_constant__ CUtensorMap g_map, const __grid_constant__ CUtensorMap x_map,
                    const __grid_constant__ CUtensorMap tap_map) {
    using S = AdjShape<IN, NCT>;
    using u64 = unsigned long long;
    constexpr int L = kAdjL, RC = kAdjRC, NS = kAdjNS, BIN = S::BIN;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::BAR_OFF);     // [NS] chunk landed
    uint64_t* empty = full + NS;                                          // [NS] every consumer warp is done with it
    volatile int* sdead = reinterpret_cast<volatile int*>(full + 2 * NS);
    uint64_t* inj = full + 2 * NS + 1;                                    // never completed (testing aid)
    float* ghs = reinterpret_cast<float*>(smem + S::GH_OFF);              // [T][NCT]

    grid_dependency_wait();                                               // launched by launch_early
    const int tid = threadIdx.x, lane = tid & 31;
    const int status = tid == 0 ? *static_cast<volatile int*>(a.err) : 0; // requested here, needed below
    const int c0 = blockIdx.y * NCT;
    const int T = a.T;
    const long long n_raw = a.n_spectra + T - 1;
    const long long tiles = (n_raw + L - 1) / L;
    const int nch = L / RC + (T + RC - 1) / RC;
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NCT / 32);
        }
        mbar_init(inj, 1);
        fence_mbar_init();
        *sdead = 0;
    }
    if (GH && tid < NCT)
        for (int t = 0; t < T; ++t) ghs[t * NCT + tid] = 0.f;
    // the status word is set: the inverse DFT (or an earlier launch) gave up, g_y
    // may not have been written
    const bool failed = __syncthreads_or(status != 0);

    BatchShare share(tiles, a.n_streams, blockIdx.x, gridDim.x);
    long long strm, lo, hi;
    if (failed) {            // grad_x becomes NaN, as grad_h does in the reduction
        if (GX && tid < NCT) {
            const float nan = __int_as_float(0x7fc00000);
            while (share.next(strm, lo, hi)) {
                float2* out = a.gx + (size_t)strm * n_raw * a.C + c0 + tid;
                const long long end = hi * L < n_raw ? hi * L : n_raw;
                for (long long r = lo * L; r < end; ++r) out[(size_t)r * a.C] = make_float2(nan, nan);
            }
        }
        return;
    }
    // chunk use g sits in slot g mod NS and completes phase g / NS of its barriers
    int slot = 0;
    uint32_t phase = 0;
    auto advance = [&] {
        if (++slot == NS) {
            slot = 0;
            phase ^= 1;
        }
    };
    if (tid >= NCT) {
        // ------------------------------------------------ producer warp
        long long issued = 0;
        bool ok = true;
        while (ok && share.next(strm, lo, hi)) {
            for (long long k = lo; ok && k < hi; ++k) {
                const AdjSteps st = ENDS ? AdjSteps(k * L, a.n_spectra, T) : AdjSteps(T);
                for (int c = 0; c < (ENDS ? L / RC + (st.n + RC - 1) / RC : nch); ++c) {
                    if (issued >= NS) ok = mbar_wait_bounded_or(&empty[slot], phase ^ 1, kWaitLimitNs, sdead);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (lane == 0) {
                        unsigned char* dst = smem + slot * S::CHUNKB;
                        fence_proxy_async_smem();
                        const int u = (c - L / RC) * RC;             // the chunk's first step
                        const bool first = u < 0;
                        mbar_expect_tx(&full[slot], S::GB + (first ? (GH ? RC * NCT * BIN : 0) : RC * NCT * 4));
                        tma_load_box3(dst, &g_map, c0, (int)(k * L) - (ENDS ? st.t1 : T - 1) + c * RC, (int)strm, &full[slot]);
                        if (!first) tma_load_box2(dst + S::GB, &tap_map, c0, ENDS ? st.t1 + 1 - RC - u : T - RC - u, &full[slot]);
                        else if (GH) tma_load_box3(dst + S::GB, &x_map, c0, (int)(k * L) + c * RC, (int)strm, &full[slot]);
                    }
                    __syncwarp();
                    ++issued;
                    advance();
                }
            }
        }
        if (!ok && lane == 0 && !*sdead) {
            atomicExch(a.err, 1);
            *sdead = 1;
        }
        // leave only after every copy of this CTA has landed
        for (long long i = 0; i < NS && i < issued; ++i) {
            if (slot == 0) {
                slot = NS;
                phase ^= 1;
            }
            --slot;
            mbar_wait_bounded(&full[slot], phase, kWaitLimitNs);
        }
        return;
    }

    // ---------------------------------------------------- consumer warps
    auto wait_full = [&] {
        if (mbar_try_wait(&full[slot], phase) || *sdead) return;
        if (!mbar_wait_bounded(&full[slot], phase, kWaitLimitNs)) {
            atomicExch(a.err, 1);
            *sdead = 1;
        }
    };
    auto release = [&] {
        __syncwarp();
        if (lane == 0) mbar_arrive_cta(&empty[slot]);
        advance();
    };
    if (tid == 0 && (a.flags & FWD_INJECT_TIMEOUT) && !mbar_wait_bounded(inj, 0, kInjectedWaitNs)) {
        atomicExch(a.err, 1);
        *sdead = 1;
    }
    while (share.next(strm, lo, hi)) {
        for (long long k = lo; k < hi; ++k) {
            const long long r0 = k * L;
            u64 acc[GX ? L : 1], win[L], xs[GH ? L : 1];
            if constexpr (GX) {
#pragma unroll
                for (int j = 0; j < L; ++j) acc[j] = 0ull;
            }
            auto load_g = [&](int i, u64& w) {
                w = *reinterpret_cast<const u64*>(smem + slot * S::CHUNKB + (i * NCT + tid) * 8);
            };
#pragma unroll
            for (int c = 0; c < L / RC; ++c) {
                wait_full();
#pragma unroll
                for (int i = 0; i < RC; ++i) {
                    load_g(i, win[c * RC + i]);
                    if constexpr (GH) {
                        const float2 v = load_one_smem<IN>(smem + slot * S::CHUNKB + S::GB + (i * NCT + tid) * BIN);
                        xs[c * RC + i] = pk2(v.x, v.y);
                    }
                }
                release();
            }
            const AdjSteps st = ENDS ? AdjSteps(r0, a.n_spectra, T) : AdjSteps(T);
            auto steps = [&](auto edge_tag) {
                // EDGE (FP32 input): some rows lie outside the stream, and an inf or NaN
                // sample must not meet their zeros
                [[maybe_unused]] constexpr bool EDGE = decltype(edge_tag)::value != 0;
#pragma unroll 1
                for (int tb = 0; tb < (ENDS ? st.n : T); tb += L) {
#pragma unroll
                    for (int blk = 0; blk < L / RC; ++blk) {
                        const int u0 = tb + blk * RC;
                        if (u0 >= (ENDS ? st.n : T)) break;
                        wait_full();
#pragma unroll
                        for (int i = 0; i < RC; ++i) {
                            const int w = blk * RC + i;              // window slot of the oldest row
                            const int t = ENDS ? st.t1 - u0 - i : T - 1 - u0 - i;
                            if (ENDS ? u0 + i >= st.n : t < 0) break;
                            if constexpr (GX) {
                                const float hv = *reinterpret_cast<const float*>(smem + slot * S::CHUNKB + S::GB +
                                                                                 ((RC - 1 - i) * NCT + tid) * 4);
                                const u64 h = pk2(hv, hv);
#pragma unroll
                                for (int j = 0; j < L; ++j) ffma2(acc[j], h, win[(j + w) % L]);
                            }
                            if constexpr (GH) {
                                u64 p0 = 0ull, p1 = 0ull;
#pragma unroll
                                for (int j = 0; j < L; ++j) {
                                    u64 x = xs[j];
                                    if constexpr (EDGE && NCT < 128) {
                                        // (a stream of 2^31 rows would not fit the device)
                                        if ((unsigned)((int)r0 - t + j) >= (unsigned)a.n_spectra) continue;
                                    } else if constexpr (EDGE) {
                                        const long long s = r0 + j - t;
                                        if (s < 0 || s >= a.n_spectra) x = 0ull;
                                    }
                                    ffma2(j & 1 ? p1 : p0, win[(j + w) % L], x);
                                }
                                const float2 p = upk2(add2(p0, p1));
                                ghs[t * NCT + tid] += p.x + p.y;
                            }
                            load_g(i, win[w]);
                        }
                        release();
                    }
                }
            };
            // EDGE's checks make a tile two to six times as long, so with 128 channels
            // they wait for an inf or NaN sample at the ends of a stream (with fewer the
            // search cost as much: C = 32, T = 8 -2 %)
            bool odd = false;
            if constexpr (GH && IN == IN_CF32) {
                odd = r0 < T - 1 || r0 + L > a.n_spectra;
                if constexpr (NCT == 128) {
                    if (odd) {
                        odd = false;
#pragma unroll
                        for (int j = 0; j < L; ++j) {
                            const float2 v = upk2(xs[j]);
                            odd |= !(fabsf(v.x) < INFINITY) | !(fabsf(v.y) < INFINITY);
                        }
                        odd = __any_sync(0xffffffffu, odd);
                    }
                }
            }
            if (GH && IN == IN_CF32 && odd) steps(ic<1>{});
            else steps(ic<0>{});
            // a wait gave up: this warp stores nothing more (the producer and the
            // other warps leave the same way)
            if (__any_sync(0xffffffffu, *sdead != 0)) return;
            if constexpr (GX) {
                float2* out = a.gx + ((size_t)strm * n_raw + r0) * a.C + c0 + tid;
#pragma unroll
                for (int j = 0; j < L; ++j)
                    if (r0 + j < n_raw) __stcs(out + (size_t)j * a.C, upk2(acc[j]));
            }
        }
    }
    if constexpr (GH) {
        float* part = a.partials + (size_t)blockIdx.x * a.TM * a.C + c0 + tid;
        for (int t = 0; t < T; ++t) part[(size_t)t * a.C] = ghs[t * NCT + tid];
    }
}

}  // namespace ppf
