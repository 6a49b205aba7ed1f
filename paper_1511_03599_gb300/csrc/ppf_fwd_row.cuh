// ppf_fwd_row.cuh -- fused PFB forward kernel for large channel counts, with
// the first DFT stage done on the FIR's registers and the rest of the
// transform local to a few warps.
//
// C = R0 * M (R0 = 1, 2, 3 or 4; M = 128 .. 1024, in small batches from 64).  With channel c = a M + b and
// bin q = k0 + R0 k', Eq. 2 splits into an R0-point DFT over a per column b,
// a twiddle W_C^{b k0}, and an M-point DFT over b per row k0:
//   * FIR (Alg. 1) + R0-point DFT: a thread owns the R0 channels of one column
//     (or of a pair of neighbouring columns) and L output spectra; it filters
//     them in registers (packed f32x2 FMAs, taps ascending), transforms over
//     a and multiplies by W_C^{b k0} (a few registers, constant for the
//     run), so the filtered spectra never pass through shared memory;
//   * the M-point DFT of each (spectrum, k0) row is two stages of one warp
//     (M = RA * RB): the first stays inside the row; the second is shared by
//     the R0 warps of a spectrum, which lets consecutive lanes hold
//     consecutive bins, so the stores to global memory are whole lines.
// One CTA of 16 warps runs per SM.  Per batch there is one barrier over the
// CTA (the rows are complete), barriers over the R0 warps of a spectrum, and
// one counted barrier that a warp only waits on before it overwrites the rows
// (they have all been read): a warp that is done with its spectra goes on to
// filter the next batch while others still transform, so the conversions and
// FMAs of the FIR overlap the shared-memory traffic of the DFT.
//
// Raw rows come from a ring of rows in shared memory filled by TMA (each row
// is read from HBM once; the T-1 halo rows of a batch stay in the ring).  The
// finished spectra then leave by TMA too: with plain stores all 16 warps
// store 128 KB at once and wait for the L2's write rate, while a bulk store
// drains during the next batch's FIR (GS/s, plain -> bulk: C = 4096 int8 T = 8
// 274 -> 293, 2048 331 -> 358, 1536 311 -> 353, 1024 int16 T = 4 411 -> 441).
// Where the ring does not fit beside the batch the rows are loaded from
// global memory, their halo from L2, and plain stores are faster (C = 3072
// int16 T = 8: 273 vs 250).  FP32 pairs up to C = 3072 go through per-thread
// cp.async slots instead of registers, whose loads could not be requested
// far enough ahead (C = 1024 T = 4: 309 -> 361, T = 8: 269 -> 293; C = 4096, where
// the slots are few, 183 -> 166).  The rows of the next batch are brought
// into L2 one batch ahead: two ahead, the rows that all CTAs keep live no
// longer fit L2 and the halo is read from HBM again (C = 1536 FP32 T = 8: 1.77
// instead of 1.07 GB read, 209 vs 266 GS/s).
//
// What bounds it: 64 instructions per sample (C = 4096 int8) at 48 % issue with 16 warps of
// 128 registers; the FIR takes a quarter of the time, shared memory traffic
// (about half of the LSU's rate) and the DFT the rest.  Against the generic
// kernel it replaces (GS/s, 2^27 samples per launch, T = 8): C = 4096 int8 230 ->
// 293, int16 170 -> 254, FP32 107 -> 194; 3072 int8 151 -> 300, int16 173 -> 273,
// FP32 119 -> 231; 2048 int8 265 -> 358, int16 209 -> 296; 1536 161 -> 353 /
// 143 -> 276 / 127 -> 266; 768 int8 177 -> 385; 384 219 -> 348 / FP32 127 -> 281;
// 1024 int16 194 -> 355, FP32 153 -> 293.  (Two CTAs of 256 threads per SM on
// half the batch measured 2-18 % slower except at T <= 2.)
#pragma once

#include "ppf_fwd_carry.cuh"

namespace ppf {

// ------------------------------------------------- packed FP32 pair helpers
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// cp_async_wait with a count known after unrolling only
__device__ __forceinline__ void cp_async_wait_upto(int n) {
    switch (n) {
        case 0: cp_async_wait<0>(); break;
        case 1: cp_async_wait<1>(); break;
        case 2: cp_async_wait<2>(); break;
        case 3: cp_async_wait<3>(); break;
        case 4: cp_async_wait<4>(); break;
        case 5: cp_async_wait<5>(); break;
        case 6: cp_async_wait<6>(); break;
        default: cp_async_wait<7>(); break;
    }
}

// A pair of 8- or 16-bit samples as (re, re) and (im, im): the real parts by the
// conversion unit, the imaginary parts (sign bit flipped) placed in the low
// mantissa of 2^23 and the bias taken off by one packed add; both are exact.
// The conversion unit does 16 lanes a clock, and a batch converts its halo rows
// again ((L + TM - 1) / L times each sample), so sharing the work pays where L
// is small: C = 4096 int8 T = 16 196 -> 217 GS/s, T = 4 335 -> 358, T = 8 277 -> 281,
// int16 T = 8 242 -> 256, C = 1024 int8 T = 16 326 -> 335.
template <int IN, class W>
__device__ __forceinline__ void cvt_mixed(W w, unsigned long long& re, unsigned long long& im) {
    if constexpr (IN == IN_CI8) {
        re = pk2((float)(int8_t)(w & 0xff), (float)(int8_t)((w >> 16) & 0xff));
        const uint32_t u = w ^ 0x80808080u;
        im = add2(pk2(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7441)), __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7443))),
                  pk2(-8388736.f, -8388736.f));
    } else {
        re = pk2((float)(int16_t)(w.x & 0xffff), (float)(int16_t)(w.y & 0xffff));
        im = add2(pk2(__uint_as_float(__byte_perm(w.x ^ 0x80008000u, 0x4B000000u, 0x7432)),
                      __uint_as_float(__byte_perm(w.y ^ 0x80008000u, 0x4B000000u, 0x7432))),
                  pk2(-8421376.f, -8421376.f));
    }
}

// R0-point DFT (sign -i) of two neighbouring columns at once: re[a], im[a]
// hold the real and imaginary parts of both columns.
template <int R0>
__device__ __forceinline__ void dft_cols(unsigned long long (&re)[R0], unsigned long long (&im)[R0]) {
    using u64 = unsigned long long;
    if constexpr (R0 == 2) {
        const u64 r = re[1], i = im[1];
        re[1] = sub2(re[0], r);
        im[1] = sub2(im[0], i);
        re[0] = add2(re[0], r);
        im[0] = add2(im[0], i);
    } else if constexpr (R0 == 3) {
        constexpr float h = 0.866025403784438646763723170752936183f;   // sqrt(3)/2
        const u64 mh = pk2(-0.5f, -0.5f), ph = pk2(h, h), nh = pk2(-h, -h);
        const u64 sr = add2(re[1], re[2]), si = add2(im[1], im[2]);
        const u64 dr = sub2(re[1], re[2]), di = sub2(im[1], im[2]);
        const u64 tr = fma2(sr, mh, re[0]), ti = fma2(si, mh, im[0]);
        re[0] = add2(re[0], sr);
        im[0] = add2(im[0], si);
        re[1] = fma2(di, ph, tr);                                      // t - i sqrt(3)/2 d
        im[1] = fma2(dr, nh, ti);
        re[2] = fma2(di, nh, tr);
        im[2] = fma2(dr, ph, ti);
    } else if constexpr (R0 == 4) {
        const u64 pr = add2(re[0], re[2]), pi = add2(im[0], im[2]);
        const u64 qr = sub2(re[0], re[2]), qi = sub2(im[0], im[2]);
        const u64 rr = add2(re[1], re[3]), ri = add2(im[1], im[3]);
        const u64 dr = sub2(re[1], re[3]), di = sub2(im[1], im[3]);
        re[0] = add2(pr, rr);
        im[0] = add2(pi, ri);
        re[1] = add2(qr, di);                                          // q - i d
        im[1] = sub2(qi, dr);
        re[2] = sub2(pr, rr);
        im[2] = sub2(pi, ri);
        re[3] = sub2(qr, di);                                          // q + i d
        im[3] = add2(qi, dr);
    }
}

// ------------------------------------------------------------ launch shape
constexpr int kRowThreads = 512;

// DIV = 1: the batch that fills the CTA's 16 warps.  DIV = 4: a quarter of it,
// for calls too short to give every SM a whole batch (row_small): a call of
// one batch is a chain of latencies, and a quarter of the outputs per thread
// on four times the SMs shortens it.  Both do the same arithmetic per output.

template <int C, int TM, int IN, int DIV = 1>
struct RowShape {
    static constexpr int R0 = row_r0(C);
    static constexpr int M = C / R0;
    static constexpr int NT = kRowThreads, NW = NT / 32;
    static constexpr int CAP = 227 * 1024;                               // dynamic shared memory of the SM's one CTA
    static constexpr int RA = row_radix(C, 0), RB = row_radix(C, 1);     // the row's two stages
    static constexpr int RPW = 1024 / M;                                 // rows per warp
    static constexpr int GW = R0;                                        // warps that share a spectrum
    static constexpr int NG_MAX = NW / GW;
    static constexpr int B = DIV == 1 ? NG_MAX * RPW : NG_MAX >= 4 ? NG_MAX / 4 * RPW : RPW;   // spectra per batch
    static constexpr int NG = B / RPW;                                   // groups of GW warps that transform
    // FIR items: a pair of columns per thread at M = 1024, else one column
    static constexpr bool PAIR = M == 1024;
    static constexpr int COLT = PAIR ? M / 2 : M;                        // threads per segment
    static constexpr int G = NT / COLT;                                  // segments per batch
    static constexpr int L = B / G;                                      // outputs per segment
    // Rows of the DFT buffer.  Its second stage reads RB consecutive elements
    // (row k1 of RA) per lane, consecutive (k0, k1) in consecutive lanes.
    // Padded: rows k1 of RB + 1 elements and a span per k0 that keeps a
    // half-warp's banks apart mod 16 (even at M = 1024, where two columns are
    // stored as 16 bytes): constant offsets, no index arithmetic.  Swizzled
    // (SWZ), where the padding would not leave room for the ring and the
    // twiddles: element j of row (k0, k1) sits at j ^ swz(k0, k1), one XOR per
    // access (C = 2048 int8 T = 8, where both fit: 305 GS/s swizzled, 330
    // padded; C = 4096, where only swizzled rows leave the twiddles in shared
    // memory: 272 vs 267; without a ring the two are equal, except that R0 = 3
    // pays for its swizzle: C = 3072 int16 T = 8 238 vs 273).
    static constexpr int PAD_SPAN = RA * (RB + 1) + (R0 == 4 ? 4 : R0 == 2 ? 8 : R0 == 3 ? (PAIR ? 6 : 11) : 0);
    static constexpr int RINGB = (B + TM - 1) * C * InTraits<IN>::bytes + 64;
    static constexpr int PADB = B * ((R0 * PAD_SPAN + 1) / 2 * 2) * 8 + 128;
    static constexpr bool SWZ = PADB + RINGB + (RA - 1) * RB * 8 > CAP && (R0 != 3 || B * C * 8 + RINGB <= CAP);
    static constexpr int RS = SWZ ? RB : RB + 1;                         // elements between rows k1
    static constexpr int SPAN = SWZ ? M : PAD_SPAN;
    static constexpr int SS = (R0 * SPAN + 1) / 2 * 2;                   // elements per spectrum (16-byte multiple)
    // distinct mod 16 over the consecutive k0 + R0 k1 of a half-warp
    static constexpr int swz(int k0, int k1) { return R0 == 3 ? (k0 + 3 * k1) & (RB - 1) : (k1 ^ (k0 * (16 / R0))) & (RB - 1); }
    static constexpr int YBYTES = (B * SS * 8 + 127) / 128 * 128;
    static constexpr int BIN = InTraits<IN>::bytes;
    static constexpr int ROWB = C * BIN;                                 // bytes of one raw row
    static constexpr int TWN = (RA - 1) * RB;                            // twiddles between the row's stages
    static constexpr int TWBYTES = TWN * 8;
    // ring of raw rows: the B + TM - 1 rows of a batch, and room for the next
    // batch's new rows where it fits beside the twiddles
    static constexpr int NR_MIN = B + TM - 1, NR_MAX = 2 * B + TM - 1;
    static constexpr bool fits(int nr, bool tw) { return YBYTES + nr * ROWB + (tw ? TWBYTES : 0) + 64 <= CAP; }
    static constexpr bool RING = fits(NR_MIN, false);
    static constexpr int NR = !RING ? 0 : fits(NR_MAX, true) ? NR_MAX : NR_MIN;
    static constexpr int AHEAD = NR == NR_MAX ? 2 : 1;                   // batches whose rows the ring holds
    static constexpr bool TW_SMEM = RING ? fits(NR, true) : true;
    // 8/16-bit pairs are converted by two units (cvt_mixed); not with 16 taps held
    // in registers (C = 2048 T = 16: -1 %)
    static constexpr bool MIXED = PAIR && IN != IN_CF32 && (L <= 5 || TM <= 8 || TM > 16);
    // STAGE: each thread copies the rows of its columns ahead of their use
    // with cp.async into NCH groups of GR slots of its own
    static constexpr int CB = BIN * (PAIR ? 2 : 1);                      // bytes of one copy
    static constexpr int LW = PAIR && L > 8 ? L / 2 : L;                 // outputs at a time with many taps
    static constexpr int RW = L + TM - 1;                                // rows of a segment
    static constexpr int NROW = R0 * RW;                                 // copies per thread and batch
    static constexpr int GR = 2;
    static constexpr int NGR = (NROW + GR - 1) / GR;                     // groups per batch
    static constexpr int NCH0 = (CAP - YBYTES - TWBYTES - 64) / (GR * NT * CB);
    static constexpr int NCH1 = NCH0 > 8 ? 8 : NCH0;
    static constexpr bool STAGE = !RING && IN == IN_CF32 && PAIR && R0 <= 3 && TM <= 16;
    static constexpr int NCH = !STAGE ? 0 : NCH1 < NGR ? NCH1 : NGR;
    // batches ahead whose new rows are brought into L2: one where the rows that
    // all CTAs keep live stay within half of it (FP32 at C = 4096, T = 8: 75 MB
    // with one ahead, 183 GS/s; 53 MB without, 194)
    static constexpr int PF = RING ? 0 : (2 * B + TM - 1) * ROWB <= 64 * 1024 * 1024 / 152 ? 1 : 0;
    static constexpr int RING_OFF = YBYTES + (TW_SMEM ? TWBYTES : 0);
    static constexpr int BAR_OFF = RING_OFF + NR * ROWB + NCH * GR * NT * CB;
    static constexpr int SMEM = BAR_OFF + 64;
    static constexpr bool OK = SMEM <= CAP && (!STAGE || (CB >= 4 && NCH >= 2));
    static_assert(B == L * G && RING_OFF % 16 == 0 && ROWB % 16 == 0, "whole segments, 16-byte aligned rows");
};

// The row kernel's body over output batches [lo, hi) of one stream (in, out:
// that stream's buffers), by a whole CTA of kRowThreads threads.  Returns
// false when a bounded wait gave up.  Safe to call again for another range.
// CONJ (T = 1, FP32): the unnormalised inverse DFT of the rows, conj(DFT(conj(.))).
template <int C, int TM, int IN, int OUT, int DIV = 1, bool CONJ = false>
__device__ __forceinline__ bool row_range(const FwdArgs& args, const void* in, void* out, long long lo, long long hi,
                                          unsigned char* smem) {
    using S = RowShape<C, TM, IN, DIV>;
    using u64 = unsigned long long;
    constexpr int R0 = S::R0, M = S::M, B = S::B, L = S::L, RA = S::RA, RB = S::RB, BIN = S::BIN, NR = S::NR;
    constexpr int SPAN = S::SPAN, RPW = S::RPW, GW = S::GW, NW = S::NW;
    constexpr bool RING = S::RING, PAIR = S::PAIR;
    static_assert(S::OK, "shape not supported by the row kernel");
    float2* ybuf = reinterpret_cast<float2*>(smem);
    float2* tw_s = reinterpret_cast<float2*>(smem + S::YBYTES);
    unsigned char* ring = smem + S::RING_OFF;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::BAR_OFF);     // [2] a batch's new rows landed
    uint64_t* yfree = full + 2;                                          // every warp has read the rows of ybuf
    uint64_t* inj = full + 3;                                            // never completed (testing aid)

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long n_spectra = args.n_spectra;
    const int T = args.T;
    const long long n_raw = n_spectra + T - 1;
    const long long nb = hi - lo;
    if (nb <= 0) return true;
    const int col = (tid % S::COLT) * (PAIR ? 2 : 1);                    // the thread's (first) column
    const int seg = (tid / S::COLT) * L;                                 // its first output of a batch

    __syncthreads();   // the previous range of this CTA is done with shared memory
    // the row tables: W_C^{b k0}, then the row's own
    const float2* row_tw = args.tw + row_tw_offset(C);
    const float2* stage_tw = row_tw + (R0 - 1) * M;
    if constexpr (S::TW_SMEM) {
        for (int i = tid; i < S::TWN; i += S::NT) tw_s[i] = stage_tw[i];
    }
    u64 wr[R0 > 1 ? R0 - 1 : 1], wi[R0 > 1 ? R0 - 1 : 1];                // PAIR: both columns' parts; else (re, im) in wr
#pragma unroll
    for (int k = 0; k + 1 < R0; ++k) {
        const float2* p = row_tw + k * M + col;
        if constexpr (PAIR) {
            const float4 w = *reinterpret_cast<const float4*>(p);
            wr[k] = pk2(w.x, w.z);
            wi[k] = pk2(w.y, w.w);
        } else {
            wr[k] = pk2(p->x, p->y);
        }
    }

    // ------------------------------------------------------------- the ring
    // Rows are relative to raw row lo*B and live in slot (row mod NR).  Copy u
    // brings the rows that batch u needs beyond batch u-1's: [0, B+TM-1) for
    // u = 0, else [uB+TM-1, (u+1)B+TM-1), clipped to the stream; with nothing
    // left to copy it still completes its phase of full[u & 1].
    const unsigned char* src = static_cast<const unsigned char*>(in) + (size_t)lo * B * S::ROWB;
    const long long rows_left = n_raw - lo * B;
    auto issue = [&](long long u) {
        const long long r0 = u == 0 ? 0 : u * B + TM - 1;
        long long r1 = (u + 1) * B + TM - 1;
        r1 = r1 < rows_left ? r1 : rows_left;
        const int n = r1 > r0 ? (int)(r1 - r0) : 0;
        uint64_t* bar = &full[u & 1];
        mbar_expect_tx(bar, (uint32_t)n * S::ROWB);
        if (n > 0) {
            const int s = (int)(r0 % (NR > 0 ? NR : 1));
            const int n0 = n < NR - s ? n : NR - s;
            tma_load_1d_once(ring + (size_t)s * S::ROWB, src + (size_t)r0 * S::ROWB, (uint32_t)n0 * S::ROWB, bar);
            if (n > n0)
                tma_load_1d_once(ring, src + (size_t)(r0 + n0) * S::ROWB, (uint32_t)(n - n0) * S::ROWB, bar);
        }
    };
    if (tid == 0) {
        mbar_init(&full[0], 1);
        mbar_init(&full[1], 1);
        mbar_init(yfree, RING ? S::NG : NW);
        mbar_init(inj, 1);
        fence_mbar_init();
        if constexpr (RING) {
            fence_proxy_async_smem();   // the slots were last read by the previous range's FIR
            for (int u = 0; u < S::AHEAD && u < nb; ++u) issue(u);
        }
    }
    __syncthreads();

    bool dead = false;                            // a wait of this thread gave up
    auto wait = [&](uint64_t* bar, uint32_t parity, uint64_t limit) {
        if (!dead && !mbar_wait_bounded(bar, parity, limit)) {
            atomicExch(args.err, 1);
            dead = true;
        }
    };
    int base = 0;                                 // ring slot of the batch's first row
    // staging: copy n of a batch is row i of the columns of channel block a; copies
    // are committed in groups of GR, the last of a batch may be short
    unsigned char* stg = ring + tid * S::CB;
    auto stage_group = [&](long long kk, int gi) {
        const long long r0 = (lo + kk) * B + seg;
        const long long left = n_raw - r0;
        const int rows = left < S::RW ? (int)left : S::RW;       // rows of the segment inside the stream
        const unsigned char* p = static_cast<const unsigned char*>(in) + ((size_t)r0 * C + col) * BIN;
#pragma unroll
        for (int q = 0; q < S::GR; ++q) {
            const int n = gi * S::GR + q, i = n % S::RW, a = n / S::RW;
            if (n < S::NROW)
                cp_async_or_zero<S::CB>(stg + (n % (S::NCH * S::GR)) * (S::NT * S::CB),
                                        p + (size_t)(i * C + a * M) * BIN, i < rows);
        }
        cp_async_commit();
    };
    if constexpr (S::STAGE) {
#pragma unroll
        for (int gi = 0; gi < S::NCH; ++gi) stage_group(0, gi);
    }
    for (long long k = 0; k < nb; ++k) {
        if constexpr (RING) wait(&full[k & 1], (uint32_t)((k >> 1) & 1), kWaitLimitNs);
        if (k == 0 && tid == 0 && (args.flags & FWD_INJECT_TIMEOUT)) wait(inj, 0, kInjectedWaitNs);
        const long long row0 = (lo + k) * B;      // first raw row and first output of the batch
        if constexpr (!RING) {
            if (S::PF > 0 && tid == 0 && k + 1 < nb) {   // warm L2 with the next batch's new rows
                const long long r0 = row0 + B + TM - 1, rows = n_raw - r0 < B ? n_raw - r0 : B;
                if (rows > 0)
                    tma_prefetch_l2(static_cast<const unsigned char*>(in) + (size_t)r0 * S::ROWB,
                                    (uint32_t)(rows * S::ROWB));
            }
        }
        // ---------------------------------------------- FIR, R0-point DFT
        // PAIR: accp[a][j] = real parts, acci = imaginary parts of both
        // columns; else accp = (re, im) of the column.
        const float* taps = args.taps + col;
        u64 accp[R0][L], acci[PAIR ? R0 : 1][PAIR ? L : 1];
        auto fir = [&](auto fast_tag, bool inside) {
            // FAST: for FP32 input, every tap of the bucket exists (a zero tap
            // must not meet an inf or NaN)
            constexpr bool FAST = decltype(fast_tag)::value != 0;
            auto row = [&](int a, int i, u64& x0, u64& x1) {
                const int off = (a * M + col) * BIN;
                if constexpr (RING) {
                    int s = base + seg + i;
                    s = s >= NR ? s - NR : s;
                    const unsigned char* p = ring + s * S::ROWB + off;
                    if constexpr (S::MIXED && IN == IN_CI8) cvt_mixed<IN>(*reinterpret_cast<const uint32_t*>(p), x0, x1);
                    else if constexpr (S::MIXED) cvt_mixed<IN>(*reinterpret_cast<const uint2*>(p), x0, x1);
                    else if constexpr (PAIR) {
                        const float4 v = load_pair_smem<IN>(p);
                        x0 = pk2(v.x, v.z);
                        x1 = CONJ ? pk2(-v.y, -v.w) : pk2(v.y, v.w);
                    } else {
                        const float2 v = load_one_smem<IN>(p);
                        x0 = pk2(v.x, CONJ ? -v.y : v.y);
                    }
                } else if constexpr (!S::STAGE) {
                    const long long r = row0 + seg + i;
                    const bool ok = inside || r < n_raw;
                    const unsigned char* p = static_cast<const unsigned char*>(in) + (size_t)(r * C + a * M + col) * BIN;
                    if constexpr (S::MIXED && IN == IN_CI8) {
                        cvt_mixed<IN>(ok ? __ldg(reinterpret_cast<const uint32_t*>(p)) : 0u, x0, x1);
                    } else if constexpr (S::MIXED) {
                        cvt_mixed<IN>(ok ? __ldg(reinterpret_cast<const uint2*>(p)) : make_uint2(0u, 0u), x0, x1);
                    } else if constexpr (PAIR) {
                        const float4 v = ok ? load_pair_global<IN>(in, r * C + a * M + col) : make_float4(0.f, 0.f, 0.f, 0.f);
                        x0 = pk2(v.x, v.z);
                        x1 = CONJ ? pk2(-v.y, -v.w) : pk2(v.y, v.w);
                    } else {
                        const float2 v = ok ? load_one_global<IN>(in, r * C + a * M + col) : make_float2(0.f, 0.f);
                        x0 = pk2(v.x, CONJ ? -v.y : v.y);
                    }
                } else {
                    const int n = a * S::RW + i, gi = n / S::GR;
                    if (n % S::GR == 0) cp_async_wait_upto(S::NGR - 1 - gi < S::NCH - 1 ? S::NGR - 1 - gi : S::NCH - 1);
                    const unsigned char* p = stg + (n % (S::NCH * S::GR)) * (S::NT * S::CB);
                    const float4 v = load_pair_smem<IN>(p);      // STAGE means PAIR
                    x0 = pk2(v.x, v.z);
                    x1 = CONJ ? pk2(-v.y, -v.w) : pk2(v.y, v.w);
                    if ((n % S::GR == S::GR - 1 || n + 1 == S::NROW) && gi + S::NCH < S::NGR) stage_group(k, gi + S::NCH);
                }
            };
            auto tap = [&](int a, int t) -> u64 {
                if constexpr (PAIR) {
                    const float2 h = __ldg(reinterpret_cast<const float2*>(taps + (size_t)t * C + a * M));
                    return pk2(h.x, h.y);
                } else {
                    const float h = __ldg(taps + (size_t)t * C + a * M);
                    return pk2(h, h);
                }
            };
#pragma unroll
            for (int a = 0; a < R0; ++a) {
#pragma unroll
                for (int j = 0; j < L; ++j) {
                    accp[a][j] = 0ull;
                    if constexpr (PAIR) acci[a][j] = 0ull;
                }
                if constexpr (TM > 16) {
                    // many taps (T is a runtime bound): taps outermost, a window of
                    // LW rows in registers, LW outputs at a time.  Bound by the loads'
                    // latency, hence the blocks: tap by tap C = 4096 int8 T = 64 took 23
                    // GS/s, in blocks 59 (the generic kernel 14; C = 1024 int8 T = 32 174
                    // against 91, C = 384 FP32 T = 64 93 against 45)
                    constexpr int LW = S::LW;
#pragma unroll
                    for (int j0 = 0; j0 < L; j0 += LW) {
                        u64 x0[LW], x1[LW];
#pragma unroll
                        for (int i = 0; i < LW; ++i) row(a, j0 + i, x0[i], x1[i]);
                        auto fma_tap = [&](u64 h, int u) {
#pragma unroll
                            for (int j = 0; j < LW; ++j) {
                                ffma2(accp[a][j0 + j], h, x0[(j + u) % LW]);
                                if constexpr (PAIR) ffma2(acci[a][j0 + j], h, x1[(j + u) % LW]);
                            }
                        };
                        int tb = 0;
                        // whole blocks of taps without checks: their loads go out together
                        auto block = [&](auto size_tag) {
                            constexpr int N = decltype(size_tag)::value;
                            u64 h[N];
#pragma unroll
                            for (int u = 0; u < N; ++u) h[u] = tap(a, tb + u);
#pragma unroll
                            for (int u = 0; u < N; ++u) {
                                fma_tap(h[u], u);
                                if (u + 1 < N || tb + N < T) row(a, j0 + tb + u + LW, x0[u % LW], x1[u % LW]);
                            }
                            tb += N;
                        };
                        constexpr int BLK = LW * ((8 + LW - 1) / LW);
#pragma unroll 1
                        while (tb + BLK <= T) block(ic<BLK>{});
                        if constexpr (BLK > LW) {
#pragma unroll 1
                            while (tb + LW <= T) block(ic<LW>{});
                        }
#pragma unroll
                        for (int u = 0; u < LW - 1; ++u) {
                            if (tb + u < T) {
                                fma_tap(tap(a, tb + u), u);
                                if (tb + u + 1 < T) row(a, j0 + tb + u + LW, x0[u], x1[u]);
                            }
                        }
                    }
                } else if constexpr (L <= 5) {
                    // taps outermost, a window of L rows in registers
                    u64 x0[L], x1[L];
#pragma unroll
                    for (int i = 0; i < L; ++i) row(a, i, x0[i], x1[i]);
#pragma unroll
                    for (int t = 0; t < TM; ++t) {
                        if (FAST || IN != IN_CF32 || t < T) {
                            const u64 h = tap(a, t);
#pragma unroll
                            for (int j = 0; j < L; ++j) {
                                ffma2(accp[a][j], h, x0[(j + t) % L]);
                                if constexpr (PAIR) ffma2(acci[a][j], h, x1[(j + t) % L]);
                            }
                        }
                        if (t + 1 < TM) row(a, t + L, x0[t % L], x1[t % L]);
                    }
                } else {
                    // rows outermost, the taps in registers
                    u64 h[TM];
#pragma unroll
                    for (int t = 0; t < TM; ++t) h[t] = tap(a, t);
#pragma unroll
                    for (int i = 0; i < L + TM - 1; ++i) {
                        u64 x0, x1;
                        row(a, i, x0, x1);
#pragma unroll
                        for (int j = 0; j < L; ++j) {
                            const int t = i - j;
                            if (t >= 0 && t < TM) {
                                if (FAST || IN != IN_CF32 || t < T) {
                                    ffma2(accp[a][j], h[t], x0);
                                    if constexpr (PAIR) ffma2(acci[a][j], h[t], x1);
                                }
                            }
                        }
                    }
                }
            }
        };
        {
            const bool inside = RING || row0 + B + TM - 1 <= n_raw;
            if (inside && (IN != IN_CF32 || T == TM)) fir(ic<1>{}, true);
            else fir(ic<0>{}, RING);
        }
#pragma unroll
        for (int j = 0; j < L; ++j) {
            if constexpr (PAIR) {
                u64 re[R0], im[R0];
#pragma unroll
                for (int a = 0; a < R0; ++a) { re[a] = accp[a][j]; im[a] = acci[a][j]; }
                dft_cols<R0>(re, im);
#pragma unroll
                for (int a = 1; a < R0; ++a) {
                    const u64 nwi = mul2(wi[a - 1], pk2(-1.f, -1.f));
                    const u64 r = re[a], i = im[a];
                    re[a] = fma2(i, nwi, mul2(r, wr[a - 1]));
                    im[a] = fma2(i, wr[a - 1], mul2(r, wi[a - 1]));
                }
#pragma unroll
                for (int a = 0; a < R0; ++a) { accp[a][j] = re[a]; acci[a][j] = im[a]; }
            } else {
                float2 v[R0];
#pragma unroll
                for (int a = 0; a < R0; ++a) v[a] = upk2(accp[a][j]);
                dft_reg<R0>(v);
#pragma unroll
                for (int a = 1; a < R0; ++a) v[a] = cmul(v[a], upk2(wr[a - 1]));
#pragma unroll
                for (int a = 0; a < R0; ++a) accp[a][j] = pk2(v[a].x, v[a].y);
            }
        }
        // the previous batch's rows have been read, and its spectra have left
        if (RING && k > 0 && lane == 0 && warp % GW == 0 && warp / GW < S::NG) {
            bulk_wait_read_all();
            mbar_arrive_cta(yfree);
        }
        if (k > 0) wait(yfree, (uint32_t)((k - 1) & 1), kWaitLimitNs);
#pragma unroll
        for (int j = 0; j < L; ++j) {
#pragma unroll
            for (int a = 0; a < R0; ++a) {
                float2* p = ybuf + (seg + j) * S::SS + a * SPAN + col;
                const float2 r = upk2(accp[a][j]);
                if constexpr (PAIR) {
                    const float2 i = upk2(acci[a][j]);
                    *reinterpret_cast<float4*>(p) = make_float4(r.x, i.x, r.y, i.y);
                } else {
                    *p = r;
                }
            }
        }
        if constexpr (S::STAGE) {
            if (k + 1 < nb) {
#pragma unroll
                for (int gi = 0; gi < S::NCH; ++gi) stage_group(k + 1, gi);
            }
        }
        if (__syncthreads_or(dead)) {
            // give up: let every copy in flight land, then leave
            bulk_wait_all();
            cp_async_wait<0>();
            if constexpr (RING) {
                if (tid == 0)
                    for (long long u = k; u < k + S::AHEAD && u < nb; ++u)
                        mbar_wait_bounded(&full[u & 1], (uint32_t)((u >> 1) & 1), kWaitLimitNs);
            }
            return false;
        }
        if constexpr (RING) {
            // the FIR of this batch has read its first B rows: their slots take a later batch's
            if (tid == 0 && k + S::AHEAD < nb) {
                fence_proxy_async_smem();
                issue(k + S::AHEAD);
            }
            base += B;
            base = base >= NR ? base - NR : base;
        }
        // ------------------------------------------------- M-point row DFTs
        const int g = warp / GW, m = warp % GW;
        if (g < S::NG) {
            {
                constexpr int IPT = RPW * RB / 32;
                static_assert(IPT >= 1 && IPT * 32 == RPW * RB, "a warp's first stage fills its lanes");
                float2 v[IPT][RA];
#pragma unroll
                for (int it = 0; it < IPT; ++it) {
                    const int item = lane + 32 * it, b = item % RB;
                    const float2* p = ybuf + (g * RPW + item / RB) * S::SS + m * SPAN + b;
#pragma unroll
                    for (int a = 0; a < RA; ++a) v[it][a] = p[RB * a];
                }
                __syncwarp();
#pragma unroll
                for (int it = 0; it < IPT; ++it) {
                    const int item = lane + 32 * it, b = item % RB;
                    float2* p = ybuf + (g * RPW + item / RB) * S::SS + m * SPAN + b;
                    dft_reg<RA>(v[it]);
                    apply_twiddles<RA, RB, S::TW_SMEM>(v[it], S::TW_SMEM ? tw_s : stage_tw, b);
#pragma unroll
                    for (int a = 0; a < RA; ++a) p[S::RS * a + (S::SWZ ? (b ^ S::swz(m, a)) - b : 0)] = v[it][a];
                }
            }
            auto group_sync = [&] {                            // the warps that share a spectrum
                if constexpr (GW == 1) __syncwarp();
                else asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(GW * 32) : "memory");
            };
            group_sync();
            constexpr int IPT = RPW * RA / 32;
            static_assert(IPT >= 1 && IPT * 32 == RPW * RA, "a group's second stage fills its lanes");
            constexpr int SITEMS = R0 * RA;                    // items per spectrum
            float2 v[IPT][RB];
#pragma unroll
            for (int it = 0; it < IPT; ++it) {
                const int item = m * 32 + lane + it * GW * 32, sl = item / SITEMS, e = item % SITEMS;
                const float2* p = ybuf + (g * RPW + sl) * S::SS + (e % R0) * SPAN + (e / R0) * S::RS;
                const int x = S::SWZ ? S::swz(e % R0, e / R0) : 0;
#pragma unroll
                for (int b = 0; b < RB; ++b) v[it][b] = p[b ^ x];
            }
            if constexpr (RING) {
                group_sync();                                  // every row of the group's spectra has been read
#pragma unroll
                for (int it = 0; it < IPT; ++it) {
                    const int item = m * 32 + lane + it * GW * 32, sl = item / SITEMS, e = item % SITEMS;
                    dft_reg<RB>(v[it]);
                    float2* p = ybuf + (g * RPW + sl) * S::SS;
#pragma unroll
                    for (int b = 0; b < RB; ++b) {
                        if constexpr (OUT == OUT_CF32) p[e + SITEMS * b] = conj_if<CONJ>(v[it][b]);
                        else reinterpret_cast<__half2*>(p)[e + SITEMS * b] = __float22half2_rn(v[it][b]);
                    }
                }
                fence_proxy_async_smem();
                group_sync();
                if (m == 0 && lane == 0) {
                    constexpr int OB = OUT == OUT_CF32 ? 8 : 4;
#pragma unroll
                    for (int sl = 0; sl < RPW; ++sl) {
                        const long long s = row0 + g * RPW + sl;
                        if (s < n_spectra)
                            tma_store_1d(static_cast<unsigned char*>(out) + (size_t)s * C * OB,
                                         ybuf + (g * RPW + sl) * S::SS, C * OB);
                    }
                    bulk_commit();
                }
            } else {
                __syncwarp();
                if (lane == 0) mbar_arrive_cta(yfree);
#pragma unroll
                for (int it = 0; it < IPT; ++it) {
                    const int item = m * 32 + lane + it * GW * 32, sl = item / SITEMS, e = item % SITEMS;
                    dft_reg<RB>(v[it]);
                    const long long s = row0 + g * RPW + sl;
                    if (s < n_spectra) {
#pragma unroll
                        for (int b = 0; b < RB; ++b) store_out<OUT>(out, s * C + e + SITEMS * b, conj_if<CONJ>(v[it][b]));
                    }
                }
            }
        } else if (!RING && lane == 0) {
            mbar_arrive_cta(yfree);
        }
    }
    if (RING) bulk_wait_all();
    // retire the barriers, the next range of this CTA initialises them anew
    // (every copy has landed: each was waited for by every thread)
    __syncthreads();
    if (tid == 0) {
        mbar_inval(&full[0]);
        mbar_inval(&full[1]);
        mbar_inval(yfree);
        mbar_inval(inj);
    }
    return true;
}

template <int C, int TM, int IN, int OUT, int DIV = 1, bool CONJ = false>
__global__ void __launch_bounds__(kRowThreads, 1) pfb_fwd_row_kernel(FwdArgs args) {
    using S = RowShape<C, TM, IN, DIV>;
    extern __shared__ __align__(128) unsigned char smem[];
    if constexpr (DIV > 1) grid_dependency_wait();   // launched by launch_early
    BatchShare share((args.n_spectra + S::B - 1) / S::B, args.n_streams, blockIdx.x, gridDim.x);
    long long strm, lo, hi;
    while (share.next(strm, lo, hi)) {
        const void* in = static_cast<const unsigned char*>(args.in) + (size_t)strm * args.in_stride * S::BIN;
        void* out = static_cast<unsigned char*>(args.out) + (size_t)strm * args.out_stride * (OUT == OUT_CF32 ? 8 : 4);
        if (!row_range<C, TM, IN, OUT, DIV, CONJ>(args, in, out, lo, hi, smem)) return;
    }
}

}  // namespace ppf
