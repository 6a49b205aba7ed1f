// ppf_fwd_longtap.cuh -- fused PFB forward kernel for many taps (T = 17..64).
//
// With many taps the T-1 halo rows a batch of output spectra shares with the
// previous batch (the overlap of neighbouring blocks, Sec. 3.2) no longer fit
// in registers, and for 32-bit input not in shared memory either (63 rows of
// 4 KB at C = 512).  So each batch of B output spectra streams all B + T - 1 raw
// rows it needs through a TMA ring in chunks of 8 rows: the rows new to the
// batch come from HBM, the halo rows from L2, where the previous batches of
// the same CTA just brought them (L2 -> SM traffic is (B + T - 1) / B times the
// input).
//
// FIR (Alg. 1): a thread owns one channel and the batch's B outputs, taps
// outermost: a window of B rows lives in registers; tap t adds h[t] x[j + t] to
// output j for all B outputs, then the dead row t is replaced by row t + B (slot
// (j + t) mod B holds row j + t).  Each FMA is a packed (re, im) x (h, h) pair.
// B = 32: per tap a thread spends 32 FMAs on one row load and one tap load, both
// from shared memory.  C = 512 is filtered in two passes of 256 channels, so
// that accumulators and window (128 registers) stay in registers with all the
// SM's 8 consumer warps on one CTA.  A warp of its own feeds the ring, taps and
// rows: it waits for a slot's "empty" barrier (every consumer warp is done
// with it) and requests the next chunk, so no consumer waits for another
// inside the FIR.  A chunk is two boxes of tensor maps (8 rows, and 8 taps, of
// the pass's channels): as one bulk copy per row of 1 - 2 KB the ring could not
// keep up (about 100 clocks per copy; 2.9 instead of 2.4 clocks per sample and SM at
// C = 512, T = 64, FP32).  The filtered batch then goes through the same warp-local
// DFT stages (Eq. 2) as the carry kernel, 16 spectra at a time.
//
// Bound by FP32 issue: T packed FMAs per sample, 1.0 clock per sample and SM at
// T = 64; the FIR takes 1.8 there with two warps per scheduler, the DFT 0.6.
// Against the form it replaces (channel pairs, batches of 16, taps and rows
// requested by consumer threads; GS/s, 2^27 samples): C = 512 FP32 T = 64 90 ->
// 136, T = 32 133 -> 188; int8 98 -> 141, 159 -> 206; C = 128 FP32 T = 32 114 -> 204;
// C = 64 int8 T = 40 139 -> 178.  Also tried: taps through registers 8 ahead
// (the loads' latency shows: 58 GS/s at T = 64), in two sets of 8 registers
// (spills: 116), refills by the last warp off a slot (73).
#pragma once

#include "ppf_fwd_carry.cuh"
#include "ppf_launch.h"
#include "ppf_tmap.h"

namespace ppf {

// Rows come as boxes of a tensor map of (channel, row, stream), whose strides have
// to be multiples of one another.  Streams that lie no whole number of rows
// apart have no such map: their rows are copied one by one (ROWS, a form of its
// own: beside the boxes in one kernel it cost 1.5 % at C = 512, T = 64, FP32).
inline bool longtap_boxes(const FwdArgs& a, int C) { return a.n_streams == 1 || a.in_stride % C == 0; }

// DIV = 1: batches of 32 outputs.  DIV = 2: of 16, for calls too short to give
// every SM a batch of 32; the same arithmetic per output.
template <int C, int IN, int DIV = 1>
struct LongShape {
    static constexpr int NCT = C < 256 ? C : 256;                    // consumer threads: one channel each per pass
    static constexpr int NPASS = C / NCT;
    static constexpr int NT = NCT + 32;                              // and the producer warp
    static constexpr int NWARP = NCT / 32;
    static constexpr int MINB = 256 / NCT;                           // CTAs per SM
    static constexpr int B = 32 / DIV;                               // output spectra per batch
    static constexpr int BIN = InTraits<IN>::bytes;
    static constexpr int RC = 8;                                     // rows (and taps) per ring chunk
    static constexpr int SPW = 16 / (NWARP > 0 ? NWARP : 1);         // spectra per warp in the DFT of 16
    static constexpr int YBYTES = B * C * 8;
    static constexpr int TWBYTES = tw_size(C) * 8;
    static constexpr int TAPB = RC * NCT * 4;                        // a chunk: 8 taps, then 8 rows
    static constexpr int ROWB = NCT * BIN;                           // one pass's channels of a row
    static constexpr int CHUNKB = TAPB + RC * ROWB;
    static constexpr int RING_OFF = (YBYTES + TWBYTES + 127) / 128 * 128;
    static constexpr int CAP = (228 * 1024) / MINB - 1024 - 256;
    static constexpr int NS0 = (CAP - RING_OFF) / (CHUNKB + 16);
    static constexpr int NS = NS0 > 8 ? 8 : NS0;                     // ring slots
    static constexpr int BAR_OFF = RING_OFF + NS * CHUNKB;           // NS full + NS empty + 1 + flag
    static constexpr int SMEM = BAR_OFF + 8 * (2 * NS + 2);
    static constexpr bool OK = C >= 64 && C <= 512 && SPW >= 1 && SPW * NWARP == 16 && warp_fft_ok(C, SPW) &&
                               NS >= 3 && SMEM <= CAP;
};

template <int C, int IN, int OUT, int DIV = 1, bool ROWS = false>
__global__ void __launch_bounds__(LongShape<C, IN, DIV>::NT, LongShape<C, IN, DIV>::MINB)
pfb_fwd_longtap_kernel(FwdArgs args, const __grid_constant__ CUtensorMap in_map, const __grid_constant__ CUtensorMap tap_map) {
    using S = LongShape<C, IN, DIV>;
    using u64 = unsigned long long;
    constexpr int NCT = S::NCT, B = S::B, BIN = S::BIN, RC = S::RC, NS = S::NS, NPASS = S::NPASS;
    constexpr int NST = fft_stages(C);
    constexpr int OB = OUT == OUT_CF32 ? 8 : 4;
    static_assert(S::OK, "shape not supported by the long-tap kernel");
    extern __shared__ __align__(128) unsigned char smem[];
    float2* ybuf = reinterpret_cast<float2*>(smem);
    float2* tw_s = reinterpret_cast<float2*>(smem + S::YBYTES);
    unsigned char* ring = smem + S::RING_OFF;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::BAR_OFF);    // [NS] chunk landed
    uint64_t* empty = full + NS;                                         // [NS] every consumer warp is done with it
    uint64_t* inj = full + 2 * NS;                                       // never completed (testing aid)
    volatile int* sdead = reinterpret_cast<volatile int*>(full + 2 * NS + 1);   // a wait gave up
    volatile int* sgone = sdead + 1;                                     // what the consumers go by: one value a batch

    if constexpr (DIV > 1 || ROWS) grid_dependency_wait();   // launched by launch_early
    const int tid = threadIdx.x, lane = tid & 31;
    const long long n_spectra = args.n_spectra;
    const int T = args.T;                        // 17 .. 64
    const long long n_raw = n_spectra + T - 1;
    const long long nbt = (n_spectra + B - 1) / B;
    // chunks per pass: the window's B rows, then 8 taps with the 8 rows they bring in
    const int nch = B / RC + (T + RC - 1) / RC;

    for (int i = tid; i < tw_size(C); i += S::NT) tw_s[i] = args.tw[i];
    if (tid == 0) {
        for (int i = 0; i < NS; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], S::NWARP);
        }
        mbar_init(inj, 1);
        fence_mbar_init();
        *sdead = 0;
    }
    __syncthreads();

    BatchShare share(nbt, args.n_streams, blockIdx.x, gridDim.x);
    long long strm, lo, hi;
    // Chunk uses are counted over the whole kernel: use g sits in slot g mod NS
    // and completes phase g / NS of its barriers, across passes, batches and
    // the stream segments of the CTA's share.
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
                for (int p = 0; ok && p < NPASS; ++p) {
                    for (int c = 0; c < nch; ++c) {
                        if (issued >= NS) ok = mbar_wait_bounded_or(&empty[slot], phase ^ 1, kWaitLimitNs, sdead);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) break;
                        const int t0 = (c - B / RC) * RC;            // the chunk's first tap
                        unsigned char* dst = ring + slot * S::CHUNKB;
                        if constexpr (ROWS) {
                            // a row per lane; rows past the stream are left as they are: no stored output reads them
                            const long long r = k * B + c * RC, left = n_raw - r;
                            const int rows = left < 0 ? 0 : left < RC ? (int)left : RC;
                            if (lane == 0) mbar_expect_tx(&full[slot], (t0 >= 0 ? S::TAPB : 0) + rows * S::ROWB);
                            __syncwarp();
                            if (lane < rows) {
                                fence_proxy_async_smem();
                                tma_load_1d(dst + S::TAPB + lane * S::ROWB,
                                            static_cast<const unsigned char*>(args.in) +
                                                (size_t)(strm * args.in_stride + (r + lane) * C + p * NCT) * BIN,
                                            S::ROWB, &full[slot]);
                            }
                        }
                        if (lane == 0) {
                            fence_proxy_async_smem();
                            if constexpr (!ROWS) {
                                mbar_expect_tx(&full[slot], t0 >= 0 ? S::CHUNKB : S::CHUNKB - S::TAPB);
                                // rows past the stream are filled with zeros
                                tma_load_box3(dst + S::TAPB, &in_map, p * NCT, (int)(k * B + c * RC), (int)strm, &full[slot]);
                            }
                            if (t0 >= 0) tma_load_box2(dst, &tap_map, p * NCT, t0, &full[slot]);
                        }
                        __syncwarp();
                        ++issued;
                        advance();
                    }
                }
            }
        }
        if (!ok && lane == 0 && !*sdead) {
            atomicExch(args.err, 1);
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
    // the chunk in the current slot has landed
    auto wait_full = [&] {
        if (mbar_try_wait(&full[slot], phase) || *sdead) return;
        if (!mbar_wait_bounded(&full[slot], phase, kWaitLimitNs)) {
            atomicExch(args.err, 1);
            *sdead = 1;
        }
    };
    auto release = [&] {
        __syncwarp();
        if (lane == 0) mbar_arrive_cta(&empty[slot]);
        advance();
    };
    auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NCT) : "memory"); };
    if (tid == 0 && (args.flags & FWD_INJECT_TIMEOUT) && !mbar_wait_bounded(inj, 0, kInjectedWaitNs)) {
        atomicExch(args.err, 1);
        *sdead = 1;
    }
    sync();
    while (share.next(strm, lo, hi)) {
        void* out = static_cast<unsigned char*>(args.out) + (size_t)strm * args.out_stride * OB;
        for (long long k = lo; k < hi; ++k) {
#pragma unroll 1
            for (int p = 0; p < NPASS; ++p) {
                // --------------------------------------------------- FIR
                u64 acc[B], win[B];
#pragma unroll
                for (int j = 0; j < B; ++j) acc[j] = 0ull;
                auto load_row = [&](const unsigned char* rows, int i, u64& w) {
                    const float2 v = load_one_smem<IN>(rows + i * NCT * BIN);
                    w = pk2(v.x, v.y);
                };
#pragma unroll
                for (int c = 0; c < B / RC; ++c) {
                    wait_full();
                    const unsigned char* rows = ring + slot * S::CHUNKB + S::TAPB + tid * BIN;
#pragma unroll
                    for (int i = 0; i < RC; ++i) load_row(rows, i, win[c * RC + i]);
                    release();
                }
#pragma unroll 1
                for (int tb = 0; tb < T; tb += B) {
#pragma unroll
                    for (int blk = 0; blk < B / RC; ++blk) {
                        const int t0 = tb + blk * RC;
                        if (t0 >= T) break;
                        wait_full();
                        const float* tp = reinterpret_cast<const float*>(ring + slot * S::CHUNKB) + tid;
                        const unsigned char* rows = ring + slot * S::CHUNKB + S::TAPB + tid * BIN;
                        // tap t: its row's last use is output 0, then row t + B takes the slot
                        auto tap = [&](int i, bool row) {
                            const int u = blk * RC + i;
                            const float hv = tp[i * NCT];
                            const u64 h = pk2(hv, hv);
                            ffma2(acc[0], h, win[u]);
                            if (row) load_row(rows, i, win[u]);
#pragma unroll
                            for (int j = 1; j < B; ++j) ffma2(acc[j], h, win[(j + u) % B]);
                        };
                        if (t0 + RC <= T) {
                            // of the last block's rows, the last is not used
#pragma unroll
                            for (int i = 0; i < RC; ++i) tap(i, true);
                        } else {
#pragma unroll
                            for (int i = 0; i < RC - 1; ++i)
                                if (t0 + i < T) tap(i, t0 + i < T - 1);
                        }
                        release();
                    }
                }
                if (p == 0) sync();   // every warp is done with the previous batch's rows
#pragma unroll
                for (int j = 0; j < B; ++j) ybuf[j * C + p * NCT + tid] = upk2(acc[j]);
            }
            if (tid == 0) *sgone = *sdead;
            sync();
            // A CTA that gave up stores nothing and leaves, with the producer: before the
            // DFT at C = 512, after it elsewhere, where each left the kernel as fast
            // as without the exit (the other way -1.8 % at C = 512, T = 64, FP32, and
            // -3 % at C = 128, T = 17, through code generation)
            const bool gone = *sgone != 0;
            if (NPASS > 1 && gone) return;
            // ------------------------------------------------------- FFT
            const long long vhi = NPASS == 1 && gone ? 0 : n_spectra;
#pragma unroll 1
            for (int q = 0; q < B / 16; ++q) {
                static_for<NST>([&](auto st) {
                    fft_stage<C, 16, NCT, decltype(st)::value, OUT, true, S::SPW>(ybuf + q * 16 * C, tw_s, out,
                                                                                  k * B + q * 16, 0, vhi);
                });
            }
            if (NPASS == 1 && vhi == 0) return;
        }
    }
}

// Tensor maps of a launch: the streams' samples as (channel, row, stream) in
// boxes of 8 rows of NCT channels (the first stream's only where the rows come
// one by one), and the plan's tap table (64 rows).
inline cudaError_t longtap_maps(const FwdArgs& a, int C, int bin, int nct, CUtensorMap* in_map, CUtensorMap* tap_map) {
    const unsigned long long n_raw = a.n_spectra + a.T - 1, row = (unsigned long long)C * bin;
    const bool one = a.n_streams == 1 || !longtap_boxes(a, C);
    const cudaError_t ce = make_tmap(in_map, a.in, bin, C, n_raw, row, one ? 1 : a.n_streams,
                                     one ? n_raw * row : a.in_stride * bin, nct, 8);
    return ce != cudaSuccess ? ce : make_tmap(tap_map, a.taps, 4, C, 64, C * 4ull, 0, 0, nct, 8);
}

template <int C, int IN, int OUT, int DIV>
inline cudaError_t longtap_launch(const FwdArgs& a, int grid, cudaStream_t st) {
    using S = LongShape<C, IN, DIV>;
    CUtensorMap in_map, tap_map;
    cudaError_t ce = longtap_maps(a, C, S::BIN, S::NCT, &in_map, &tap_map);
    if (ce != cudaSuccess) return ce;
    if (!longtap_boxes(a, C)) {
        constexpr auto k = &pfb_fwd_longtap_kernel<C, IN, OUT, DIV, true>;
        ce = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
        return ce != cudaSuccess ? ce : launch_early(k, grid, S::NT, S::SMEM, st, a, in_map, tap_map);
    }
    if constexpr (DIV > 1) {
        return launch_early(pfb_fwd_longtap_kernel<C, IN, OUT, DIV>, grid, S::NT, S::SMEM, st, a, in_map, tap_map);
    } else {
        pfb_fwd_longtap_kernel<C, IN, OUT, DIV><<<grid, S::NT, S::SMEM, st>>>(a, in_map, tap_map);
        return cudaPeekAtLastError();
    }
}

}  // namespace ppf
