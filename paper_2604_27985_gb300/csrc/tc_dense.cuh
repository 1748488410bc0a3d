// Densified tensor-core path: A's 128 x 64 tiles are expanded into shared memory and multiplied
// whole (tc_dense.cu).
#pragma once

#include "tc_ptx.cuh"

namespace gbsp {
namespace dense {

constexpr int kRows = 128;  // rows of a block (the MMA's M)
constexpr int kCols = 64;   // columns of a tile: 128 bytes of BF16, one swizzle atom

inline int64_t row_blocks(int64_t M) { return (M + kRows - 1) / kRows; }
inline int64_t ent_count(int64_t nnz) { return nnz + 4; }
inline int64_t col_tiles(int64_t K) { return (K + kCols - 1) / kCols; }

// A's stored entries regrouped by tile, block after block (a block's entries keep the CSR range
// of its rows): ent[e] = BF16 value << 16 | byte offset in the swizzled tile, and
// tptr[b * (col_tiles + 1) + t] = first entry of tile t of row block b.  bad[b] is 1 where a
// row of the block has column indices that are not strictly increasing or not in [0, K), and
// the block's entries are then not written.
// ent is 16-byte aligned and has room for ent_count(nnz) words (whole 16-byte pieces are read).
struct Tiles {
    uint32_t *ent;
    int32_t *tptr;
    int32_t *bad;
    int32_t *chunk;  // per row block: log2 of the tiles of an SpMM accumulator, up to 128 features | past them << 4
    int32_t *pos;  // ent[e]'s CSR position, or null
};

// Microseconds that a call's scratch costs beside its kernels: what the pool does not keep is mapped anew after
// every synchronisation (1.2 GB 0.4 ms, 1.9 GB 1.7, 3.4 GB 4.3, 4.0 GB 5.3; a little less is counted, since not
// every call is followed by one).
inline double scratch_us(int64_t bytes) {
    return bytes > (int64_t)kPoolKeep ? 1.6e-6 * (double)(bytes - (int64_t)kPoolKeep) : 0.0;
}

// Whether the regrouping is possible for these sizes (entry positions are 32-bit and run up to 2,048 past
// the last entry), and whether it is worth it.
bool tiles_fit(int64_t M, int64_t K, int64_t nnz);
// (dense_nnz: the entries that a plan's 16 x 8 blocks would hold)
bool spmm_pays(int64_t M, int64_t K, int64_t N, int64_t nnz, int64_t dense_nnz);
// ... for a plan, whose N is not known yet: at 256 features, in accuracy at 512 if not.
bool spmm_may_pay(int64_t M, int64_t K, int64_t nnz, int64_t dense_nnz);
// ... also where the regrouping is part of every call, against the CSR kernels.
bool spmm_pays_unplanned(int64_t M, int64_t K, int64_t N, int64_t nnz);

// (vals may be null where pos is not: the words then hold no values)
int launch_bin(const int32_t *rowptr, const int32_t *colidx, const uint16_t *vals, int64_t M, int64_t K, int64_t nnz,
               Tiles t, cudaStream_t s);
// C = A B for N a multiple of 8 and 16-byte aligned B rows: every block of rows on the tensor
// cores, then the marked ones (by t.bad when given, by a value that is not finite or by a wait
// that ran out) again on the CUDA cores from p's CSR arrays.  marks: mark_count ints of scratch.
// err, when given, records a wait that ran out (withhold >= 0: block 0 never loads that tile).
inline int64_t mark_count(int64_t M, int64_t N) { return row_blocks(M) * ((N + 255) / 256); }
int launch_spmm(const SpmmProblem &p, Tiles t, int32_t *marks, int *err, int withhold, cudaStream_t s);


// out[p] = svals[p] <X_i, Y_j> for every entry of the regrouped pattern (t.pos given): the whole
// product of 128 X rows and 64 Y rows per tile on the tensor cores, read at the entries.  Kd of at
// most sddmm_max_kd elements, Kd and the leading dimensions multiples of 16 bytes, 16-byte aligned X
// and Y.  err records a wait that ran out; without it (E4M3, Kd <= 256) the blocks marked in t.bad are
// computed again on the CUDA cores.
inline int64_t sddmm_max_kd(bool fp8) { return fp8 ? 512 : 256; }
bool sddmm_pays(int64_t M, int64_t K, int64_t Kd, int64_t nnz, bool fp8);
bool sddmm_pays_unplanned(int64_t M, int64_t K, int64_t Kd, int64_t nnz);  // (E4M3 X and Y)
int launch_sddmm(const SddmmProblem &p, Tiles t, int *err, int withhold, cudaStream_t s);

}  // namespace dense
}  // namespace gbsp
