// SpMM dispatch by element type and algorithm, and the unvectorised kernel.
#include "spmm_kernels.cuh"

namespace gbsp {

// Units per lane: what covers the row, at most 8 (FP32 sums of at most 16 elements a lane).
template <class EL, int LB>
int launch_scalar(const SpmmProblem &P, cudaStream_t s) {
    using namespace spmm_detail;
    constexpr int UE = LB / (int)sizeof(typename EL::stored), TMAX = UE >= 8 ? 2 : UE >= 4 ? 4 : 8;
    const int units = P.N / UE;
    const dim3 grid((P.M + 7) / 8);
    if (units <= 32)
        spmm_unit_kernel<EL, LB, 1><<<grid, 256, 0, s>>>(P);
    else if (units <= 64 || TMAX == 2)
        spmm_unit_kernel<EL, LB, 2><<<grid, 256, 0, s>>>(P);
    else if (units <= 128 || TMAX == 4)
        spmm_unit_kernel<EL, LB, TMAX < 4 ? TMAX : 4><<<grid, 256, 0, s>>>(P);
    else
        spmm_unit_kernel<EL, LB, TMAX><<<grid, 256, 0, s>>>(P);
    count_launches(1);
    return check_launch("spmm scalar");
}

template <class EL>
int launch_spmm_typed(const SpmmProblem &P, int variant, int vecs, int unroll, int ctas_per_sm, cudaStream_t s) {
    if (variant == GBSP_VARIANT_SCALAR) {
        // rows averaging under 16 entries (or not said): 200,000 x 3,000, 6 entries a row, N = 101: 85 us
        // against 117 for the units; and 65 to 128 single BF16 elements a row: 287 us against 299 on 30,011 x
        // 41,017, N = 101
        constexpr int ES = (int)sizeof(typename EL::stored);
        const int lb = unit_bytes(P.B, P.ldb, P.N, ES);
        if (P.nnz < 16LL * P.M || (ES == 2 && lb == 2 && P.N > 64 && P.N <= 128)) {
            spmm_detail::spmm_scalar_kernel<EL><<<dim3((P.M + 7) / 8, 1), 256, 0, s>>>(P);
            count_launches(1);
            return check_launch("spmm scalar");
        }
        if constexpr (ES <= 1)
            if (lb == 1) return launch_scalar<EL, 1>(P, s);
        if constexpr (ES <= 2)
            if (lb == 2) return launch_scalar<EL, 2>(P, s);
        return lb == 4 ? launch_scalar<EL, 4>(P, s) : launch_scalar<EL, 8>(P, s);
    }
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
