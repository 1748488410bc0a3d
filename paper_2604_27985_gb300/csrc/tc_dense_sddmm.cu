// Dense-tile SDDMM on the tensor cores: out[p] = s_p <X_i, Y_j>.
//
// At 10% of entries a CSR kernel gathers one Y row per entry (512 bytes at Kd = 256 in BF16: 13.7 GB
// on 16,384^2) while the whole product X Y^T is 137 GFLOP, 73 us at the measured cuBLAS rate.  A
// CTA keeps 128 X rows in shared memory, streams Y 64 rows at a time by TMA, multiplies them with
// tcgen05.mma (M = 128 X rows, N = 64 Y rows) and reads the tile's stored entries out of the result:
// TMEM to shared memory (16-byte chunks swizzled by row), then each entry's word times its value,
// to its CSR position.  The product's other cells are never looked at, so X and Y rows meet only
// where an entry is stored, whatever they hold.
//
// The tensor core's accumulation is not rounded to nearest, so Kd is cut into four parts with an
// accumulator each, added in FP32: error against 64 bits at Kd = 256 in BF16 8.1e-8 (the 16 x 8
// blocks' one accumulator and their CSR residual together 1.7e-7, the CSR kernel 6.1e-8), in
// E4M3 3.0e-8 (4.7e-8, 4.5e-8), where value and scales are applied with one rounding.
//
// 16,384^2 at 90%, half in dense blocks, Kd = 256: BF16 on a plan 637 -> 215 us, where the MMAs alone
// (N = 64 reads A's rows from shared memory for little work: 92 clocks each) take 152; E4M3 without
// a plan 804 -> 446 with the regrouping's 172 (260 here: fewer MMA steps, more instructions per entry).  On the way: 328 us with the tile coordinates by
// 64-bit division in every warp, 245 without.
#include <mutex>

#include "sddmm_kernels.cuh"
#include "tc_dense.cuh"

namespace gbsp {
namespace dense {
namespace {

using namespace gbsp::tc;

constexpr int kGroups = 2;                  // groups of warps, each with a TMEM and a staging buffer
constexpr int kGroupWarps = 8;              // a warp reads 32 rows x 32 columns of a tile
constexpr int kGroupThreads = 32 * kGroupWarps;
constexpr int kThreads = (kGroupWarps * kGroups + 2) * 32;
constexpr int kStageBytes = kRows * kCols * 4;  // a tile's FP32 results
constexpr int kPer = 4;                     // entries per thread of a tile loaded ahead
constexpr int kParts = 4;                   // accumulators of a tile: 64 TMEM columns each
constexpr int kAhead = 8;                   // tiles of a group between the L2 prefetch of entries and their load
constexpr int kMaxSmem = 227 * 1024;
// Shared memory that leaves L1 some 64 KB where it can: the entries' values are gathered through L1
// (each miss holds a line), and with 224 KB taken the kernel spent a third of its time on them
// (16,384^2 at 90%, Kd = 256: 266 us with three Y stages, 212 with two).
constexpr int kSmemGoal = 164 * 1024;
constexpr int kMaxStages = 8;

struct SdArgs {
    Tiles t;
    const float *svals;
    float *out;
    const float *x_scale, *y_scale;
    int M, Ny, nkt;
    int64_t tiles;   // row blocks x column tiles, shared evenly and in order among the CTAs
    int kb;          // 128-byte blocks of an X or Y row
    int stages;      // Y tiles held or on their way
    int *err;
    int withhold;
};

// One word of a run of about 64 / density bytes that the next tiles go on with: the miss brings 256
// bytes to L2.
__device__ __forceinline__ float ld_run(const float *p) {
    float v;
    asm volatile("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ void add(float (&x)[16], const float (&y)[16]) {
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        const float2 v = __fadd2_rn(make_float2(x[j], x[j + 1]), make_float2(y[j], y[j + 1]));
        x[j] = v.x;
        x[j + 1] = v.y;
    }
}

// (v + ev) * x * y rounded once, ev being the rounding error of v: the three roundings of v * (x * y)
// are most of the E4M3 form's error (16,384^2 at 90%, Kd = 256: 4.57e-8 with them, 3.0e-8 so; the CSR
// kernel has 4.55e-8, and the whole call takes 447 us against 439).  v * (x * y) itself where something is
// not finite and for a zero's sign.
__device__ __forceinline__ float scaled(float v, float ev, float x, float y) {
    const float p = __fmul_rn(x, y), plain = __fmul_rn(v, p);
    const float exact = __fmaf_rn(v, p, __fmaf_rn(v, __fmaf_rn(x, y, -p), __fmul_rn(ev, p)));
    return fabsf(exact) > 0.f && fabsf(exact) < __int_as_float(0x7f800000) ? exact : plain;
}

template <int V>
struct Int { static constexpr int value = V; };

// Where a CTA's tile i lies: row block b, column tile kt (steps forward without a division).
struct At {
    int i, b, kt;
    __device__ __forceinline__ void step(int by, int nkt) {
        i += by;
        kt += by;
        while (kt >= nkt) {
            kt -= nkt;
            ++b;
        }
    }
};

template <bool FP8>
__global__ void __launch_bounds__(kThreads, 1) sddmm_kernel(const __grid_constant__ CUtensorMap tmX,
                                                            const __grid_constant__ CUtensorMap tmY, const SdArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int xbytes = a.kb * kRows * 128, ybytes = a.kb * kCols * 128;
    uint8_t *ys = smem + xbytes;
    uint8_t *staging = ys + a.stages * ybytes;
    float *scales = reinterpret_cast<float *>(staging + kGroups * kStageBytes);  // E4M3: a group's X and Y scales
    uint64_t *xfull = reinterpret_cast<uint64_t *>(scales + (FP8 ? kGroups * (kRows + kCols) : 0));
    uint64_t *xfree = xfull + 1;             // the last MMA on the X rows is done
    uint64_t *yfull = xfree + 1;             // a Y tile landed
    uint64_t *yfree = yfull + kMaxStages;    // ... and its MMAs are done
    uint64_t *dfull = yfree + kMaxStages;    // a group's accumulators are complete
    uint64_t *dfree = dfull + kGroups;       // ... and read
    uint32_t *tslot = reinterpret_cast<uint32_t *>(dfree + kGroups);
    int *failed = reinterpret_cast<int *>(tslot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t f0 = a.tiles * blockIdx.x / gridDim.x, f1 = a.tiles * (blockIdx.x + 1) / gridDim.x;
    const int n = (int)(f1 - f0), nkt = a.nkt;
    const At first{0, (int)(f0 / nkt), (int)(f0 % nkt)};

    if (tid == 0) {
        mbar_init(xfull, 1);
        mbar_init(xfree, 1);
        for (int s = 0; s < a.stages; ++s) {
            mbar_init(&yfull[s], 1);
            mbar_init(&yfree[s], 1);
        }
        for (int g = 0; g < kGroups; ++g) {
            mbar_init(&dfull[g], 1);
            mbar_init(&dfree[g], kGroupWarps);
        }
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tslot, kGroups * kParts * kCols);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = *tslot;

    if (warp < kGroupWarps * kGroups) {
        const int g = warp / kGroupWarps, q = warp & 3, half = (warp >> 2) & 1, t = tid % kGroupThreads;
        const uint8_t *st = staging + g * kStageBytes;
        const uint32_t tlane = taddr + ((uint32_t)(32 * q) << 16) + g * kParts * kCols + half * (kCols / 2);
        const int row = 32 * q + lane;  // of the block: this thread's TMEM lane
        float *own = scales + g * (kRows + kCols);  // thread t: the scale of X row t or of Y row t - 128
        float scale = 1.f;                          // ... for the tile after this one
        float *mine = reinterpret_cast<float *>(staging + g * kStageBytes) + row * kCols;
        bool ok = true;
        // A tile's words and positions are loaded two turns ahead and its values one: each is a
        // trip to HBM (about a microsecond) or, for the first two, to L2 after a prefetch.
        struct Ent {
            int e0, e1;
            uint32_t w[kPer];
            int p[kPer];
        };
        auto bounds = [&](const At &at, int &e0, int &e1) {
            const int32_t *tp = a.t.tptr + (int64_t)at.b * (nkt + 1) + at.kt;
            e0 = __ldg(tp);
            e1 = __ldg(a.t.bad + at.b) ? e0 : __ldg(tp + 1);  // (a block that was not regrouped has no entries here)
        };
        At at = first, ahead = first, far = first;  // the tile worked on, loaded, brought to L2
        at.step(g, nkt);
        ahead.step(g, nkt);
        far.step(g + kAhead * kGroups, nkt);
        int b0 = 0, b1 = 0, q0 = 0, q1 = 0;  // bounds of those two tiles, loaded a turn before their use
        auto more = [&]() {
            b0 = b1 = q0 = q1 = 0;
            if (ahead.i < n) bounds(ahead, b0, b1);
            if (t == 0 && far.i < n) bounds(far, q0, q1);
            ahead.step(kGroups, nkt);
            far.step(kGroups, nkt);
        };
        auto load = [&](Ent &x) {
            x.e0 = b0;
            x.e1 = b1;
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                const int e = x.e0 + t + kGroupThreads * j;
                x.w[j] = e < x.e1 ? __ldcs(a.t.ent + e) : 0;
                x.p[j] = e < x.e1 ? __ldcs(a.t.pos + e) : -1;
            }
            if (q1 > q0) {
                q0 &= ~3;
                prefetch_l2(a.t.ent + q0, ((q1 - q0) * 4 + 15) & ~15);
                prefetch_l2(a.t.pos + q0, ((q1 - q0) * 4 + 15) & ~15);
            }
            more();
        };
        auto values = [&](const Ent &x, float (&s)[kPer]) {
#pragma unroll
            for (int j = 0; j < kPer; ++j) s[j] = x.p[j] >= 0 ? ld_run(a.svals + x.p[j]) : 0.f;
        };
        Ent now, next, after;
        float s[kPer], snext[kPer];
        auto scale_of = [&](const At &x) {
            const int r = x.b * kRows + t, c = x.kt * kCols + t - kRows;
            if (t < kRows) return x.i < n && r < a.M ? __ldg(a.x_scale + r) : 1.f;
            return x.i < n && t < kRows + kCols && c < a.Ny ? __ldg(a.y_scale + c) : 1.f;
        };
        if (FP8) scale = scale_of(at);
        more();
        load(now);
        load(next);
        load(after);
        values(now, s);
        values(next, snext);
        for (int turn = 0; at.i < n; at.step(kGroups, nkt), ++turn) {
            ok = __all_sync(FULL, mbar_wait(&dfull[g], turn & 1));
            ok = bar_all(1 + g, kGroupThreads, ok);  // (the group is also done with the last tile's staging)
            if (!ok) break;
            if (FP8) {
                if (t < kRows + kCols) own[t] = scale;
                At then = at;
                then.step(kGroups, nkt);
                scale = scale_of(then);
            }
            fence_after_sync();
#pragma unroll
            for (int k = 0; k < kCols / 2; k += 16) {
                float d[16];
                tmem_ld16(tlane + k, d);
#pragma unroll
                for (int part = 1; part < kParts; ++part) {
                    float r[16];
                    tmem_ld16(tlane + part * kCols + k, r);
                    add(d, r);
                }
                // the image of the BF16 tile, two bytes per byte: an entry's place is its word's
#pragma unroll
                for (int j = 0; j < 16; j += 8) {
                    float4 *to = reinterpret_cast<float4 *>(mine + ((((half * 32 + k + j) >> 3) ^ (row & 7)) << 3));
                    to[0] = make_float4(d[j], d[j + 1], d[j + 2], d[j + 3]);
                    to[1] = make_float4(d[j + 4], d[j + 5], d[j + 6], d[j + 7]);
                }
            }
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dfree[g]);
            ok = bar_all(1 + g, kGroupThreads, ok);  // every row of the tile is staged
            auto emit = [&](uint32_t w, int p, float sv) {
                const float d = *reinterpret_cast<const float *>(st + (w & 0xffffu) * 2);
                float v = __fmul_rn(sv, d);
                if (FP8) {
                    const int r = (w >> 7) & 127, c = (((w >> 4 ^ r) & 7) << 3) + ((w >> 1) & 7);
                    v = scaled(v, __fmaf_rn(sv, d, -v), own[r], own[kRows + c]);
                }
                a.out[p] = v;
            };
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (now.p[j] >= 0) emit(now.w[j], now.p[j], s[j]);
            for (int e = now.e0 + t + kGroupThreads * kPer; e < now.e1; e += kGroupThreads) {
                const int p = __ldcs(a.t.pos + e);
                emit(__ldcs(a.t.ent + e), p, __ldg(a.svals + p));
            }
            now = next;
            next = after;
#pragma unroll
            for (int j = 0; j < kPer; ++j) s[j] = snext[j];
            values(next, snext);
            load(after);
        }
        if (!ok) *failed = 1;
    } else if (warp == kGroupWarps * kGroups) {
        if (lane == 0) {
            bool ok = true;
            int xs = 0, ynum = 0;  // X blocks and Y tiles sent for
            int sl = 0, phase = 1;  // Y stage; the parity of its last release
            At at = first;
            for (; at.i < n; at.step(1, nkt)) {
                const int i = at.i;
                if (i == 0 || at.kt == 0) {
                    if (xs > 0 && !mbar_wait(xfree, (xs - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(xfull, xbytes);
                    for (int k = 0; k < a.kb; ++k)
                        tma_load_2d(smem + k * kRows * 128, &tmX, xfull, k * (FP8 ? 128 : 64), at.b * kRows);
                    ++xs;
                }
                if (i >= a.stages && !mbar_wait(&yfree[sl], phase)) {
                    ok = false;
                    break;
                }
                if (i == a.withhold && blockIdx.x == 0) break;  // nothing will complete yfull[sl]
                mbar_expect_tx(&yfull[sl], ybytes);
                for (int k = 0; k < a.kb; ++k)
                    tma_load_2d(ys + sl * ybytes + k * kCols * 128, &tmY, &yfull[sl], k * (FP8 ? 128 : 64), at.kt * kCols);
                ynum = i + 1;
                if (++sl == a.stages) {
                    sl = 0;
                    phase ^= 1;
                }
            }
            if (!ok) *failed = 1;
            // every issued copy lands before the CTA can leave (bounded waits)
            if (xs > 0) mbar_wait(xfull, (xs - 1) & 1);
            for (int i = ynum > a.stages ? ynum - a.stages : 0; i < ynum; ++i)
                mbar_wait(&yfull[i % a.stages], (i / a.stages) & 1);
        }
    } else {
        // FP32 accumulator, A (X rows) and B (Y rows) K-major, M = 128, N = 64; BF16 or E4M3
        constexpr uint32_t kIdesc = (1u << 4) | ((FP8 ? 0u : 1u) << 7) | ((FP8 ? 0u : 1u) << 10) |
                                    ((uint32_t)(kCols >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t ad0 = smem_desc(smem_u32(smem), 16, 1024), bd0 = smem_desc(smem_u32(ys), 16, 1024);
        const bool one = elect_one();
        bool ok = true;
        int xs = 0;
        int sl = 0, phase = 0;
        At at = first;
        for (; at.i < n; at.step(1, nkt)) {
            const int i = at.i, g = i % kGroups;
            if (i == 0 || at.kt == 0) {
                ok = __all_sync(FULL, mbar_wait(xfull, xs & 1));
                ++xs;
            }
            if (i >= kGroups) ok = ok && __all_sync(FULL, mbar_wait(&dfree[g], (i / kGroups - 1) & 1));
            ok = ok && __all_sync(FULL, mbar_wait(&yfull[sl], phase));
            if (!ok) break;
            fence_after_sync();
            const uint64_t bd = bd0 + (uint32_t)(sl * ybytes >> 4);
            const uint32_t d = taddr + g * kParts * kCols;
            // kb blocks of four 32-byte steps in kParts parts of kb steps each
            auto issue = [&](auto kbt) {
                constexpr int KB = decltype(kbt)::value;
#pragma unroll
                for (int x = 0; x < 4 * KB; ++x) {
                    const uint64_t ad = ad0 + (uint32_t)(x / 4 * (kRows * 128 >> 4) + x % 4 * 2);
                    const uint64_t bdk = bd + (uint32_t)(x / 4 * (kCols * 128 >> 4) + x % 4 * 2);
                    if constexpr (FP8)
                        mma_e4m3(d + x / KB * kCols, ad, bdk, kIdesc, x % KB ? 1u : 0u);
                    else
                        mma_bf16(d + x / KB * kCols, ad, bdk, kIdesc, x % KB ? 1u : 0u);
                }
            };
            if (one) {
                switch (a.kb) {
                    case 1: issue(Int<1>{}); break;
                    case 2: issue(Int<2>{}); break;
                    case 3: issue(Int<3>{}); break;
                    default: issue(Int<4>{});
                }
                mma_commit(&yfree[sl]);
                mma_commit(&dfull[g]);
                if (i == n - 1 || at.kt == nkt - 1) mma_commit(xfree);
            }
            __syncwarp();
            if (++sl == a.stages) {
                sl = 0;
                phase ^= 1;
            }
        }
        if (!ok && one) *failed = 1;
    }
    __syncwarp();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (warp == 0) tmem_dealloc(taddr, kGroups * kParts * kCols);
    if (tid == 0 && *failed) {
        if (a.err)
            atomicExch(a.err, 1);
        else  // without a plan to report to, the blocks are computed again
            for (int64_t b = f0 / nkt; b * nkt < f1; ++b) a.t.bad[b] = 1;
    }
}

// The blocks marked in bad, from the CSR arrays (E4M3, Kd of at most 256): a warp per row.  Usually
// no block is marked and the CTAs leave at once.
__global__ void __launch_bounds__(256) marked_rows_kernel(const SddmmProblem P, const int32_t *bad) {
    if (!__ldg(bad + blockIdx.x / (kRows / 8))) return;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= P.M) return;
    sddmm_detail::sddmm_segment<E4M3, 16, 1, true>(P, row, __ldg(P.rowptr + row), __ldg(P.rowptr + row + 1),
                                                   threadIdx.x & 31);
}

template <bool FP8>
int launch(const CUtensorMap &mx, const CUtensorMap &my, const SdArgs &a, int ctas, int smem, cudaStream_t s) {
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return fail(GBSP_ERR_UNSUPPORTED, "tc dense sddmm: device ordinal %d", dev);
    std::call_once(once[dev], [] {
        cudaFuncSetAttribute(sddmm_kernel<FP8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    });
    sddmm_kernel<FP8><<<(unsigned)ctas, kThreads, smem, s>>>(mx, my, a);
    count_launches(1);
    return check_launch("tc dense sddmm kernel");
}

int encode(const void *data, int64_t rows, int64_t cols, int64_t ld, bool fp8, int box_rows, CUtensorMap *map) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return fail(GBSP_ERR_CUDA, "tc dense sddmm: cuTensorMapEncodeTiled is not available");
    const int es = fp8 ? 1 : 2;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * es};
    const cuuint32_t box[2] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(data), dims,
            strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return fail(GBSP_ERR_CUDA, "tc dense sddmm: tensor map encoding failed");
    return GBSP_OK;
}

}  // namespace

// Time against time, in microseconds: a CTA takes 0.95 a tile whatever the tile holds and Kd is
// (BF16 and E4M3, 2,048 to 24,000 rows and columns); the plan's blocks and CSR residual, and the
// CSR kernels alone, 12 / 16 / 24 ps per entry at Kd = 64 / 128 / 256.  On 16,384^2 the lines
// cross near 7.5% / 5.5% / 3.7% of entries.
bool sddmm_pays(int64_t M, int64_t K, int64_t Kd, int64_t nnz, bool fp8) {
    // (rows of at least one 128-byte block: a copy's box does not pass the row's width)
    if (M < 2048 || K < 2048 || Kd > sddmm_max_kd(fp8) || Kd < (fp8 ? 128 : 64) ||
        (double)nnz < 0.03 * (double)M * (double)K)
        return false;
    const double tile = 0.95 * (double)(row_blocks(M) * col_tiles(K)) / (double)(sm_count() > 0 ? sm_count() : 1);
    return tile + 8.0 < 0.9e-6 * (double)nnz * (8.0 + 0.062 * (double)Kd);
}

// ... with the regrouping in every call (0.6 ns per entry of a block of rows, a wave of blocks at a
// time; 0.8 with the positions on 16,384^2, where at Kd = 128 the two paths take the same time and whole
// tiles are the more exact one).  E4M3 only: at Kd <= 256 its error is below the CSR kernel's (3.0e-8 against 4.55e-8 on
// 16,384^2 at 90%, Kd = 256), BF16's four steps per part have the larger one
// (8.0e-8 against 6.1e-8).  The E4M3 CSR kernel is bound by its conversions: 16 / 30 ps per entry at
// Kd = 128 / 256.  Where the scratch passes the pool's limit (from 134 million entries on) a tile was measured at
// 1.6 to 2.2 ns an entry: 300 million, calls waited for, Kd = 128 7.7 ms against 4.3 for the row split, Kd = 256
// 7.7 against 8.4; 138 million 2.3 against 2.1 and 2.4 against 3.9.
bool sddmm_pays_unplanned(int64_t M, int64_t K, int64_t Kd, int64_t nnz) {
    if (M < 2048 || K < 2048 || Kd > 256 || Kd < 128 || (double)nnz < 0.03 * (double)M * (double)K) return false;
    const int64_t sms = sm_count() > 0 ? sm_count() : 1, nb = row_blocks(M);
    const double held = (double)nnz / (double)(nb * col_tiles(K)), remap = scratch_us(8 * nnz);
    const double tile = (remap > 0 && held > 560 ? 1.7e-3 * held : 0.95) * (double)(nb * col_tiles(K)) / (double)sms;
    const double bins = (double)((nb + sms - 1) / sms) * 0.6e-3 * (double)nnz / (double)nb;
    return tile + bins + 12.0 + remap < 0.85e-6 * (double)nnz * (2.5 + 0.105 * (double)Kd);
}

int launch_sddmm(const SddmmProblem &p, Tiles t, int *err, int withhold, cudaStream_t s) {
    const bool fp8 = p.dtype == GBSP_E4M3;
    CUtensorMap mx, my;
    int st;
    if ((st = encode(p.X, p.M, p.Kd, p.ldx, fp8, kRows, &mx)) || (st = encode(p.Y, p.N, p.Kd, p.ldy, fp8, kCols, &my)))
        return st;
    const int kb = (int)((p.Kd * (fp8 ? 1 : 2) + 127) / 128);
    SdArgs a{t, p.svals, p.out, p.x_scale, p.y_scale, p.M, p.N, (int)col_tiles(p.N), 0, kb, 0, err, withhold};
    a.tiles = row_blocks(p.M) * a.nkt;
    const int fixed = kb * kRows * 128 + kGroups * kStageBytes + 1024 + 256 +
                      (fp8 ? kGroups * (kRows + kCols) * 4 : 0);
    a.stages = (kSmemGoal - fixed) / (kb * kCols * 128);
    a.stages = a.stages > kMaxStages ? kMaxStages : a.stages < 2 ? 2 : a.stages;
    const int smem = fixed + a.stages * kb * kCols * 128;
    const int ctas = (int)(a.tiles < sm_count() ? a.tiles : sm_count());
    st = fp8 ? launch<true>(mx, my, a, ctas, smem, s) : launch<false>(mx, my, a, ctas, smem, s);
    if (st || err) return st;
    marked_rows_kernel<<<(unsigned)(row_blocks(p.M) * (kRows / 8)), 256, 0, s>>>(p, t.bad);
    count_launches(1);
    return check_launch("tc dense sddmm marked rows");
}

}  // namespace dense
}  // namespace gbsp
