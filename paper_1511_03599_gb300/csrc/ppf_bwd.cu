// ppf_bwd.cu -- instantiates the fused PFB adjoint kernels (complex int8 /
// int16 / FP32 input, C in {64, 128, 256, 512}, tap buckets up to 16 where
// the batch holds the halo) and the runtime-shape passes of the unfused
// adjoint, and exports their lookups and launches.
#include <algorithm>

#include "ppf_bwd.cuh"
#include "ppf_bwd_unfused.cuh"
#include "ppf_internal.h"

namespace ppf {

template <int C, int TM, int IN>
static bool make_bwd(BwdEntry* e) {
    const BwdInfo i = bwd_info<C, TM, IN>();
    if (i.fn == nullptr) return false;
    *e = BwdEntry{i.threads, i.batch, i.smem, i.fn, &bwd_launch<C, TM, IN>};
    return true;
}

template <int C, int IN>
static bool bwd_by_tm(int tm, BwdEntry* e) {
    switch (tm) {
        case 1: return make_bwd<C, 1, IN>(e);
        case 2: return make_bwd<C, 2, IN>(e);
        case 4: return make_bwd<C, 4, IN>(e);
        case 8: return make_bwd<C, 8, IN>(e);
        case 16: return make_bwd<C, 16, IN>(e);
        default: return false;
    }
}

template <int C>
static bool bwd_by_in(int tm, int in, BwdEntry* e) {
    switch (in) {
        case IN_CI8: return bwd_by_tm<C, IN_CI8>(tm, e);
        case IN_CI16: return bwd_by_tm<C, IN_CI16>(tm, e);
        case IN_CF32: return bwd_by_tm<C, IN_CF32>(tm, e);
        default: return false;
    }
}

bool bwd_lookup(int C, int tm, int in, BwdEntry* e) {
    switch (C) {
        case 64: return bwd_by_in<64>(tm, in, e);
        case 128: return bwd_by_in<128>(tm, in, e);
        case 256: return bwd_by_in<256>(tm, in, e);
        case 512: return bwd_by_in<512>(tm, in, e);
        default: return false;
    }
}

cudaError_t bwd_reduce(const float* partials, int nparts, int T, int TM, int C, const int* err, float* grad_h,
                       cudaStream_t st) {
    const int TC = T * C;
    return launch_early(pfb_bwd_reduce_kernel, (TC + 31) / 32, dim3(32, kReduceLanes), 0, st, partials, nparts, TC, TM * C,
                        err, grad_h);
}

template <int IN, int NCT, bool GX, bool GH, bool ENDS>
static cudaError_t grad_launch(const AdjArgs& a, const AdjMaps& m, int parts, cudaStream_t st) {
    using S = AdjShape<IN, NCT>;
    constexpr auto k = &pfb_bwd_grad_kernel<IN, NCT, GX, GH, ENDS>;
    const int smem = S::smem(GH ? a.T : 0);
    const cudaError_t ce = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::smem(PPF_MAX_TAPS));
    if (ce != cudaSuccess) return ce;
    return launch_early(k, dim3(parts, a.C / NCT), S::NT, smem, st, a, m.g, m.x, m.taps);
}

// Streams of few rows, most of whose tiles hold an end, leave out the steps that meet
// no row of theirs (calls per s, without -> with: C = 512, T = 64, int8, 400 streams of
// 9 rows 4290 -> 9560, 50 of 100 rows 12200 -> 12900, 50 of 800 rows 2850 -> 2870; FP32, 10 of
// 400 rows 19100 -> 18700); for longer ones the bounds cost up to 1.5 %.
template <int IN, int NCT, bool GX, bool GH>
static cudaError_t grad_by_length(const AdjArgs& a, const AdjMaps& m, int parts, cudaStream_t st) {
    return a.n_spectra < 4ll * a.T ? grad_launch<IN, NCT, GX, GH, true>(a, m, parts, st)
                                   : grad_launch<IN, NCT, GX, GH, false>(a, m, parts, st);
}

template <int IN, int NCT>
static cudaError_t grad_by_sums(const AdjArgs& a, const AdjMaps& m, int parts, cudaStream_t st) {
    if (a.gx == nullptr) return grad_by_length<IN, NCT, false, true>(a, m, parts, st);
    if (a.partials == nullptr) return grad_by_length<IN_CI8, NCT, true, false>(a, m, parts, st);   // x is not read
    return grad_by_length<IN, NCT, true, true>(a, m, parts, st);
}

template <int IN>
static cudaError_t grad_by_channels(const AdjArgs& a, const AdjMaps& m, int parts, cudaStream_t st) {
    return a.C == 32 ? grad_by_sums<IN, 32>(a, m, parts, st)
         : a.C == 64 ? grad_by_sums<IN, 64>(a, m, parts, st) : grad_by_sums<IN, 128>(a, m, parts, st);
}

// Channels per CTA (every planned C >= 128 is a multiple of 128).
static int grad_channels(int C) { return C < 128 ? C : 128; }

int bwd_grad_parts(int in, int C, int T, int sms, long long n_raw, long long n_streams) {
    const int nct = grad_channels(C), blocks = C / nct;
    // resident CTAs: bounded by registers (AdjShape::MINB) and by the grad_h table
    const int regs = nct == 128 ? 3 : nct == 64 ? 5 : 8;
    const int bytes = (in == IN_CF32 ? AdjShape<IN_CF32, 128>::smem(T) : AdjShape<IN_CI8, 128>::smem(T)) / 128 * nct + 1024;
    const int fit = 228 * 1024 / bytes;
    const long long tiles = n_streams * ((n_raw + kAdjL - 1) / kAdjL);
    const long long parts = std::max(1ll, (long long)sms * std::max(1, std::min(regs, fit)) / blocks);
    return (int)std::min(parts, tiles);
}

cudaError_t bwd_grad(int in, const AdjArgs& a, const float2* gy, const void* x, const float* taps, int parts,
                     cudaStream_t st) {
    AdjMaps m;
    const int nct = grad_channels(a.C), bin = in == IN_CI8 ? 2 : in == IN_CI16 ? 4 : 8;
    const unsigned long long C = a.C, S = a.n_spectra, n_raw = S + a.T - 1;
    cudaError_t ce = make_tmap(&m.g, gy, 8, C, S, C * 8, a.n_streams, S * C * 8, nct, kAdjRC);
    if (ce == cudaSuccess) ce = make_tmap(&m.x, x, bin, C, n_raw, C * bin, a.n_streams, n_raw * C * bin, nct, kAdjRC);
    if (ce == cudaSuccess) ce = make_tmap(&m.taps, taps, 4, C, a.TM, C * 4, 0, 0, nct, kAdjRC);
    if (ce != cudaSuccess) return ce;
    switch (in) {
        case IN_CI8: return grad_by_channels<IN_CI8>(a, m, parts, st);
        case IN_CI16: return grad_by_channels<IN_CI16>(a, m, parts, st);
        case IN_CF32: return grad_by_channels<IN_CF32>(a, m, parts, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace ppf
