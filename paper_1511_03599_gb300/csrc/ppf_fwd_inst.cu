// ppf_fwd_inst.cu -- instantiates the fused forward kernel for one channel
// count C (compiled once per C with -DPPF_C=<C>) over every tap bucket,
// input type and output type, and the inverse DFT of the unfused adjoint,
// and exports the lookups used by the C ABI.
#include "ppf_bwd_unfused.cuh"
#include "ppf_fwd.cuh"
#include "ppf_internal.h"

#ifndef PPF_C
#error "compile with -DPPF_C=<channels>"
#endif

#define PPF_CAT2(a, b) a##b
#define PPF_CAT(a, b) PPF_CAT2(a, b)

namespace ppf {

template <int TM, int IN, int OUT>
static bool make_entry(FwdEntry* e) {
    FwdInfo i = fwd_info<PPF_C, TM, IN, OUT>();
    *e = FwdEntry{i.threads, i.batch, i.smem, i.stages, i.tap_bucket, i.variant, i.fn, &fwd_launch<PPF_C, TM, IN, OUT>,
                  i.cluster, 0, 0, nullptr, nullptr, nullptr, nullptr};
    if constexpr (row_small<PPF_C, TM, IN>()) {
        using S = RowShape<PPF_C, TM, IN, 4>;
        e->small_batch = S::B;
        e->small_smem = S::SMEM;
        e->small_fn = reinterpret_cast<const void*>(&pfb_fwd_row_kernel<PPF_C, TM, IN, OUT, 4>);
        e->small_launch = &row_small_launch<PPF_C, TM, IN, OUT>;
        e->small_ctas = 1;
    }
    if constexpr (TM == 64) {
        if constexpr (LongShape<PPF_C, IN>::OK) {
            using S = LongShape<PPF_C, IN, 2>;
            e->small_batch = S::B;
            e->small_smem = S::SMEM;
            e->small_fn = reinterpret_cast<const void*>(&pfb_fwd_longtap_kernel<PPF_C, IN, OUT, 2>);
            e->small_launch = &longtap_launch<PPF_C, IN, OUT, 2>;
            e->small_ctas = S::MINB;
        }
    }
    if constexpr (carry_preferred<PPF_C, TM, IN>()) {
        e->short_fn = reinterpret_cast<const void*>(&pfb_fwd_carry_kernel<PPF_C, TM, IN, OUT, false, true>);
        e->short_launch = &carry_short_launch<PPF_C, TM, IN, OUT>;
    }
    return true;
}

template <int TM, int IN>
static bool by_out(int out, FwdEntry* e) {
    switch (out) {
        case OUT_CF32: return make_entry<TM, IN, OUT_CF32>(e);
        case OUT_CF16: return make_entry<TM, IN, OUT_CF16>(e);
        default: return false;
    }
}

template <int TM>
static bool by_in(int in, int out, FwdEntry* e) {
    switch (in) {
        case IN_CI8: return by_out<TM, IN_CI8>(out, e);
        case IN_CI16: return by_out<TM, IN_CI16>(out, e);
        case IN_CF32: return by_out<TM, IN_CF32>(out, e);
        default: return false;
    }
}

bool PPF_CAT(fwd_lookup_c, PPF_C)(int tm, int in, int out, FwdEntry* e) {
    switch (tm) {
        case 1: return by_in<1>(in, out, e);
        case 2: return by_in<2>(in, out, e);
        case 4: return by_in<4>(in, out, e);
        case 8: return by_in<8>(in, out, e);
        case 16: return by_in<16>(in, out, e);
        case 64: return by_in<64>(in, out, e);   // any T in 17..64 (runtime tap loop)
        default: return false;
    }
}

template <int TM, int IN>
static bool make_fir(FwdEntry* e) {
    FwdInfo i;
    if (!fir_info<PPF_C, TM, IN>(&i)) return false;
    *e = FwdEntry{i.threads, i.batch, i.smem, i.stages, i.tap_bucket, i.variant, i.fn, &fir_launch<PPF_C, TM, IN>, 0,
                  0, 0, nullptr, nullptr, nullptr, nullptr};
    return true;
}

template <int TM>
static bool fir_by_in(int in, FwdEntry* e) {
    switch (in) {
        case IN_CI8: return make_fir<TM, IN_CI8>(e);
        case IN_CI16: return make_fir<TM, IN_CI16>(e);
        case IN_CF32: return make_fir<TM, IN_CF32>(e);
        default: return false;
    }
}

bool PPF_CAT(fir_lookup_c, PPF_C)(int tm, int in, FwdEntry* e) {
    switch (tm) {
        case 1: return fir_by_in<1>(in, e);
        case 2: return fir_by_in<2>(in, e);
        case 4: return fir_by_in<4>(in, e);
        case 8: return fir_by_in<8>(in, e);
        case 16: return fir_by_in<16>(in, e);
        default: return false;
    }
}

template <auto KERNEL, int NT, int SMEM>
static cudaError_t launch_kernel(const FwdArgs& a, int grid, cudaStream_t st) {
    KERNEL<<<grid, NT, SMEM, st>>>(a);
    return cudaPeekAtLastError();
}

template <auto KERNEL, int NT, int SMEM>
static cudaError_t launch_kernel_early(const FwdArgs& a, int grid, cudaStream_t st) {
    return launch_early(KERNEL, grid, NT, SMEM, st, a);
}

// The inverse DFT of the three-pass adjoint: the forward kernels with T = 1 and
// conjugation; the small batches wherever the forward has them.
template <int C>
static bool make_idft(FwdEntry* e) {
    *e = FwdEntry{};
    e->tap_bucket = 1;
    if constexpr (C == 32) {
        using S = IdftShape<C>;
        e->threads = S::NT;
        e->batch = S::B;
        e->smem = S::SMEM;
        e->fn = reinterpret_cast<const void*>(&pfb_bwd_idft_kernel<C>);
        e->launch = &launch_kernel<pfb_bwd_idft_kernel<C>, S::NT, S::SMEM>;
        return true;
    } else {
        if constexpr (carry_preferred<C, 1, IN_CF32>()) {
            using S = CarryShape<C, 1, IN_CF32>;
            constexpr auto k = &pfb_fwd_carry_kernel<C, 1, IN_CF32, OUT_CF32, false, false, true>;
            constexpr auto ks = &pfb_fwd_carry_kernel<C, 1, IN_CF32, OUT_CF32, false, true, true>;
            e->threads = S::NT;
            e->batch = S::B;
            e->smem = S::SMEM;
            e->variant = 4;
            e->fn = reinterpret_cast<const void*>(k);
            e->launch = &launch_kernel<k, S::NT, S::SMEM>;
            e->short_fn = reinterpret_cast<const void*>(ks);
            e->short_launch = &launch_kernel_early<ks, S::NT, S::SMEM>;
        } else {
            using S = RowShape<C, 1, IN_CF32>;
            constexpr auto k = &pfb_fwd_row_kernel<C, 1, IN_CF32, OUT_CF32, 1, true>;
            e->threads = S::NT;
            e->batch = S::B;
            e->smem = S::SMEM;
            e->variant = 128;
            e->fn = reinterpret_cast<const void*>(k);
            e->launch = &launch_kernel<k, S::NT, S::SMEM>;
        }
        using M = RowShape<C, 1, IN_CF32, 4>;
        constexpr auto km = &pfb_fwd_row_kernel<C, 1, IN_CF32, OUT_CF32, 4, true>;
        e->small_batch = M::B;
        e->small_smem = M::SMEM;
        e->small_fn = reinterpret_cast<const void*>(km);
        e->small_launch = &launch_kernel_early<km, M::NT, M::SMEM>;
        e->small_ctas = 1;
        return true;
    }
}

bool PPF_CAT(idft_lookup_c, PPF_C)(FwdEntry* e) { return make_idft<PPF_C>(e); }

int PPF_CAT(fwd_twiddle_count_c, PPF_C)() { return tw_total_float2s(PPF_C) > 0 ? tw_total_float2s(PPF_C) : 1; }

void PPF_CAT(fwd_twiddles_c, PPF_C)(float* host_pairs) {
    fill_twiddles<PPF_C>(reinterpret_cast<float2*>(host_pairs));
}

}  // namespace ppf
