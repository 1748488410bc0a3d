// SpMM dispatch by element type and algorithm, and the unvectorised kernel.
#include "spmm_kernels.cuh"

namespace gbsp {

// Units per lane: what covers the row, at most 8 (FP32 sums of at most 16 elements a lane).
template <class EL, int LB>
int launch_units(const SpmmProblem &P, cudaStream_t s) {
    using namespace spmm_detail;
    // (single elements: up to 64, in E4M3 also past 192)
    constexpr int ES = (int)sizeof(typename EL::stored), UE = LB / ES;
    constexpr int TMAX = UE >= 8 || (UE == 1 && ES > 1) ? 2 : UE >= 4 ? 4 : 8;
    const int units = P.N / UE;
    const dim3 grid((P.M + 7) / 8);
    if (units <= 32)
        spmm_unit_kernel<EL, LB, 1><<<grid, 256, 0, s>>>(P);
    else if (units <= 64 || TMAX == 2)
        spmm_unit_kernel<EL, LB, 2><<<grid, 256, 0, s>>>(P);
    else if constexpr (UE == 1)
        spmm_unit_kernel<EL, LB, TMAX><<<grid, 256, 0, s>>>(P);
    else if (units <= 128 || TMAX == 4)
        spmm_unit_kernel<EL, LB, TMAX < 4 ? TMAX : 4><<<grid, 256, 0, s>>>(P);
    else
        spmm_unit_kernel<EL, LB, TMAX><<<grid, 256, 0, s>>>(P);
    count_launches(1);
    return check_launch("spmm units");
}

template <class EL, int U, int T>
int launch_elements(const SpmmProblem &P, cudaStream_t s) {
    spmm_detail::spmm_scalar_kernel<EL, U, T><<<dim3((P.M + 7) / 8), 256, 0, s>>>(P);
    count_launches(1);
    return check_launch("spmm scalar");
}

// The unvectorised kernels, by what the rows' alignment allows (lb bytes a load) and what was measured on 30,011
// x 41,017 (20 and 205 entries a row, even and Zipf), 4,000 x 41,017 (1,500), 200,000 x 3,000 (100), 3,000 x 3,000
// (200) and 20,000 x 250,000 (60, clustered):
// - rows averaging under 16 entries (or not said): one entry at a time.  200,000 x 3,000, 6 entries a row,
//   N = 101: 85 us against 117 for the units.
// - wide loads that leave half of the lanes without one are halved: E4M3 N = 24 to 120 from 8 bytes 1.4 to 2.8
//   times as fast; the others level or better.
// - 65 to 96 single elements: three columns a lane, four entries in flight, 0.67 to 0.88 of the units' time (four
//   columns), 0.82 to 1.10 of one at a time's (the lower end on Zipf rows).
// - more of them: FP32 four columns and entries, 0.81 to 1.05 of the units' time; E4M3 up to 128 the same, 0.89 to
//   1.02 (one at a time takes 0.78 to 0.99 of theirs on even rows, 1.03 to 1.07 on Zipf ones).  E4M3 up to 192
//   three columns one at a time, 0.64 to 0.89 of the units' time; BF16 four columns one at a time, up to 128 0.66
//   to 0.98, past that 0.68 to 0.85 (1.02 on Zipf rows).  E4M3 past 192 the units: one at a time takes 0.73 to 0.91
//   of their time on even rows and 1.13 on Zipf ones.
template <class EL>
int launch_unvectorised(const SpmmProblem &P, cudaStream_t s) {
    constexpr int ES = (int)sizeof(typename EL::stored);
    if (P.nnz < 16LL * P.M) return launch_elements<EL, 1, 4>(P, s);
    int lb = unit_bytes(P.B, P.ldb, P.N, ES);
    while (lb > ES && P.N * ES < 16 * lb) lb /= 2;
    if (lb == ES && P.N > 64) {
        if (P.N <= 96) return launch_elements<EL, 4, 3>(P, s);
        if constexpr (ES == 2) return launch_elements<EL, 1, 4>(P, s);
        if constexpr (ES != 2)
            if (ES == 4 || P.N <= 128) return launch_elements<EL, 4, 4>(P, s);
        if constexpr (ES == 1)
            if (P.N <= 192) return launch_elements<EL, 1, 3>(P, s);
    }
    if constexpr (ES <= 1)
        if (lb == 1) return launch_units<EL, 1>(P, s);
    if constexpr (ES <= 2)
        if (lb == 2) return launch_units<EL, 2>(P, s);
    return lb == 4 ? launch_units<EL, 4>(P, s) : launch_units<EL, 8>(P, s);
}

template <class EL>
int launch_spmm_typed(const SpmmProblem &P, int variant, int vecs, int unroll, int ctas_per_sm, cudaStream_t s) {
    if (variant == GBSP_VARIANT_SCALAR) return launch_unvectorised<EL>(P, s);
    if (variant == GBSP_VARIANT_MERGE) return launch_spmm_algo<EL, GBSP_VARIANT_MERGE>(P, vecs, unroll, ctas_per_sm, s);
    if (variant == GBSP_VARIANT_ROWGROUP)
        return launch_spmm_algo<EL, GBSP_VARIANT_ROWGROUP>(P, vecs, unroll, ctas_per_sm, s);
    return launch_spmm_algo<EL, GBSP_VARIANT_ROWSPLIT>(P, vecs, unroll, ctas_per_sm, s);
}

int launch_spmm(const SpmmProblem &p, int variant, int vecs, int unroll, int ctas_per_sm, cudaStream_t s) {
    switch (p.dtype) {
        case GBSP_F32: return launch_spmm_typed<F32>(p, variant, vecs, unroll, ctas_per_sm, s);
        case GBSP_BF16: return launch_spmm_typed<BF16>(p, variant, vecs, unroll, ctas_per_sm, s);
        case GBSP_E4M3: return launch_spmm_typed<E4M3>(p, variant, vecs, unroll, ctas_per_sm, s);
    }
    return fail(GBSP_ERR_UNSUPPORTED, "spmm: dtype %d", p.dtype);
}

}  // namespace gbsp
