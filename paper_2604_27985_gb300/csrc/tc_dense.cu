// Dense-tile SpMM on the tensor cores for BF16 matrices of a few percent of entries and more.
//
// At 90% sparsity a row split gathers one B row (512 bytes at N = 256) per stored entry from
// L2, 13.7 GB on 16,384^2, while the whole dense product is 137 GFLOP, 73 us at the measured
// cuBLAS rate.  So A is expanded: a CTA takes 128 rows of A and all of (up to 256 columns of)
// B, walks A's columns 64 at a time, scatters a 128 x 64 tile's entries into a zeroed tile in
// shared memory (already in the MMA's K-major 128-byte-swizzled image), loads the 64 B rows by
// TMA and multiplies with tcgen05.mma (M = 128 rows, N = the features, K = 64).
//
// The products of BF16 values are exact; the tensor core cuts each at the accumulator's last bit, so its
// error grows with the entries that one accumulator takes.  So an accumulator in TMEM runs over at most
// 512 columns, in a block of rows with more entries there than suit it (sum_limit) over 256, 128 or
// 64, and the worker warps add it to FP32 sums in registers, two accumulators alternating.  Error
// against 64 bits on 16,384^2 at 90%, uniform: 1.53e-7 with 256 columns per accumulator (where the
// register sums' rounding dominates), 1.28e-7 with 512, 1.50e-7 with 1,024; the CSR kernel has 2.0e-7
// (N = 256), the 16 x 8 blocks over all columns 9.7e-7.  With values and B of one sign an accumulator
// of e entries a row is 1.9e-9 e too small: 512 columns at 10% / 40% of entries 9.6e-8 / 4.5e-7.
//
// The expanded zeros meet B's values: an infinity or NaN in any B row makes NaN in every row
// of C.  Every accumulated value is tested at the end, and a block with one that is not finite
// is computed again from the CSR arrays on the CUDA cores, where only stored entries count.
#include <mutex>

#include "spmm_kernels.cuh"
#include "tc_dense.cuh"

namespace gbsp {

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

namespace dense {
namespace {

using namespace gbsp::tc;

// ---- regrouping -----------------------------------------------------------------------------

constexpr int kColBits = 6;  // log2(kCols)
static_assert(1 << kColBits == kCols, "tiles of 64 columns");
constexpr int kBinThreads = 1024;
constexpr int kLogChunk = 3;  // log2 of the tiles of a TMEM accumulator at most: 512 columns of A
constexpr int kChunk = 1 << kLogChunk;
constexpr int kMaxTiles = 8 * 1024;  // one shared-memory counter per tile of a row block

// Entries [p0, p1) of a row, U chunks of 32 at a time with the next U chunks' loads in flight:
// f(columns, values, first entry of the first chunk, whether every lane holds an entry).  Lanes past
// p1 hold column kNone.
constexpr int kNone = 0x7fffffff;
template <int V>
struct Int { static constexpr int value = V; };
struct true_t { static constexpr bool value = true; };
struct false_t { static constexpr bool value = false; };
template <int U, bool VALS, class F>
__device__ __forceinline__ void for_chunks(const int32_t *colidx, const uint16_t *vals, int p0, int p1, int lane,
                                           F f) {
    int nc[U];
    uint16_t nv[U];
    const int32_t *cp = colidx + p0 + lane;
    const uint16_t *vp = vals + p0 + lane;
    auto load = [&](int left) {  // (left entries of the row from the next block's first one on)
        if (left >= 32 * U) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                nc[u] = __ldg(cp + 32 * u);
                if (VALS) nv[u] = __ldg(vp + 32 * u);
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = 32 * u + lane < left;
                nc[u] = in ? __ldg(cp + 32 * u) : kNone;
                if (VALS) nv[u] = in ? __ldg(vp + 32 * u) : 0;
            }
        }
        cp += 32 * U;
        vp += 32 * U;
    };
    load(p1 - p0);
    for (int base = p0; base < p1; base += 32 * U) {
        int c[U];
        uint16_t v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = nc[u];
            v[u] = VALS ? nv[u] : 0;
        }
        if (base + 32 * U < p1) load(p1 - base - 32 * U);
        if (base + 32 * U <= p1)
            f(c, v, base, true_t{});
        else
            f(c, v, base, false_t{});
    }
}

// One CTA per block of 128 rows, a warp per row: counts the entries per tile, turns the counts into
// offsets and writes each entry's packed word at its tile's cursor (the order inside a tile is
// free: every entry has its own place there).  The two passes read the column indices from HBM
// and again mostly from L2.  Columns ascend, so a tile's count is the sum over rows of where the
// row leaves the tile minus where it enters it; a chunk's run of entries in one tile is placed by
// its first lane's reservation.
// 16,384^2 at 90% (26.8M entries): 107 us, bound by instruction issue (89 per 32 entries); 168 with
// the runs also counted and one chunk in flight.  Three launches over a table of every row's
// entry into every tile, with the whole GPU but no atomics, took 53 + 16 + 69.
template <bool VALS, bool POS>
__global__ void __launch_bounds__(kBinThreads) bin_kernel(const int32_t *__restrict__ rowptr,
                                                          const int32_t *__restrict__ colidx,
                                                          const uint16_t *__restrict__ vals, int M, int K, int nkt,
                                                          Tiles t, int2 limit) {
    constexpr int U = 4;
    extern __shared__ int32_t cnt[];  // nkt counters, then cursors
    __shared__ int32_t warp_sum[32];
    __shared__ int32_t carry, over;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.x, r0 = b * kRows, r1 = min(r0 + kRows, M);
    for (int i = tid; i < nkt; i += kBinThreads) cnt[i] = 0;
    if (tid == 0) carry = over = 0;
    __syncthreads();
    bool good = true;
    for (int r = r0 + warp; r < r1; r += kBinThreads / 32) {
        const int p0 = __ldg(rowptr + r), p1 = __ldg(rowptr + r + 1);
        int last = -1;  // the column before the chunk's first
        for_chunks<U, false>(colidx, nullptr, p0, p1, lane, [&](const int (&c)[U], const uint16_t (&)[U], int base, auto all) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                int prev = __shfl_up_sync(FULL, c[u], 1);
                if (lane == 0) prev = last;
                last = __shfl_sync(FULL, c[u], 31);
                if (!all.value && c[u] == kNone) continue;
                const bool fits = c[u] > prev && c[u] < K;
                good &= fits;
                const int p = base + 32 * u + lane, t1 = c[u] >> kColBits, t0 = prev >> kColBits;
                if (fits && t1 != t0) {
                    atomicSub(&cnt[t1], p);
                    if (t0 >= 0 && t0 < nkt) atomicAdd(&cnt[t0], p);
                }
            }
        });
        if (lane == 0 && p1 > p0) {
            const int c = __ldg(colidx + p1 - 1);
            if (c >= 0 && c < K) atomicAdd(&cnt[c >> kColBits], p1);
        }
    }
    const bool bad = !__syncthreads_and(good);
    const int32_t start = __ldg(rowptr + r0);
    int32_t *tp = t.tptr + (int64_t)b * (nkt + 1);
    for (int base = 0; base < nkt; base += kBinThreads) {
        const int i = base + tid;
        const int v = i < nkt ? cnt[i] : 0;
        int x = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(FULL, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        int before = carry;
        for (int w = 0; w < warp; ++w) before += warp_sum[w];
        if (i < nkt) {
            cnt[i] = start + before + x - v;
            tp[i] = start + before + x - v;
        }
        __syncthreads();
        if (tid == kBinThreads - 1) carry = before + x;
        __syncthreads();
    }
    // bit k of over: some 2^(k + 1) tiles (from a multiple of that on) hold more entries than the narrow
    // form's limit; bit 3 + k: ... the wide form's
    auto first = [&](int i) { return i < nkt ? cnt[i] : start + carry; };
    int mine = 0;
    for (int i = 2 * tid; i < nkt; i += 2 * kBinThreads)
#pragma unroll
        for (int k = 0; k < kLogChunk; ++k) {
            const int held = i % (2 << k) == 0 ? first(i + (2 << k)) - first(i) : 0;
            mine |= (held > limit.x) << k | (held > limit.y) << (kLogChunk + k);
        }
    if (mine) atomicOr(&over, mine);
    __syncthreads();
    if (tid == 0) {
        tp[nkt] = start + carry;
        t.bad[b] = bad ? 1 : 0;
        const int narrow = over & (kChunk - 1), wide = over >> kLogChunk;  // (the lowest bit: how often 512 columns are halved)
        t.chunk[b] = (narrow ? __ffs(narrow) - 1 : kLogChunk) | (wide ? __ffs(wide) - 1 : kLogChunk) << 4;
    }
    if (bad) return;
    const unsigned upto = FULL >> (31 - lane), beyond = ~upto;
    for (int r = r0 + warp; r < r1; r += kBinThreads / 32) {
        const uint32_t row_off = (r - r0) * 128, flip = ((r - r0) & 7) << 4;
        for_chunks<U, VALS>(colidx, vals, __ldg(rowptr + r), __ldg(rowptr + r + 1), lane,
                            [&](const int (&c)[U], const uint16_t (&v)[U], int base, auto all) {
            int first[U], at[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int t1 = c[u] >> kColBits, t0 = __shfl_up_sync(FULL, t1, 1);
                const unsigned heads = __ballot_sync(FULL, t1 != t0) | 1u;
                first[u] = 31 - __clz(heads & upto);
                if (first[u] == lane && (all.value || c[u] != kNone)) {  // (lanes without an entry are a run too)
                    const unsigned after = heads & beyond;
                    at[u] = atomicAdd(&cnt[t1], (after ? __ffs(after) - 1 : 32) - lane) - lane;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int to = __shfl_sync(FULL, at[u], first[u]) + lane;
                const uint32_t off = row_off + (((uint32_t)c[u] << 1 & 0x70u) ^ flip) + ((uint32_t)c[u] << 1 & 0xeu);
                if (all.value || c[u] != kNone) {
                    t.ent[to] = ((uint32_t)v[u] << 16) | off;
                    if (POS) t.pos[to] = base + 32 * u + lane;
                }
            }
        });
    }
}

// ---- product --------------------------------------------------------------------------------

constexpr int kGroups = 4;                      // groups of four warps that expand tiles and drain accumulators
constexpr int kWorkers = 4 * kGroups;
constexpr int kThreads = (kWorkers + 2) * 32;   // + one warp that copies, one that issues MMAs
constexpr int kATileBytes = kRows * kCols * 2;  // 16 KB
constexpr int kSlot = 1072;                     // words of an entry slot (any more come from global memory)
constexpr int kAhead = 3;                       // turns between the L2 prefetch of a tile's entries and their copy

template <int NT>
struct Shape {
    static constexpr int BT = kCols * NT * 2;         // bytes of a tile's B rows
    static constexpr int SB = NT == 256 ? 4 : NT == 128 ? 6 : 8;  // tiles whose B rows are held or on their way
    static constexpr int R = NT == 256 ? 2 : 3;       // entry slots of a group: one is read, the others on their way
    static constexpr int SLOTS = R * kGroups;
    static constexpr int SMEM = kGroups * kATileBytes + SB * BT + SLOTS * (kSlot * 4 + 24) + 1024 + 256;
};

struct Args {
    Tiles t;
    int32_t *marks;  // [feature tile][row block]: 1 where the block is to be computed again
    float *C;
    int64_t ldc;
    int M, N, nkt;
    int vec;  // floats per store: 8 (32-byte aligned C rows), 4 or 1
    int *err;
    int withhold;
};

__device__ __forceinline__ void st_shared_u16(uint32_t addr, uint16_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}
__device__ __forceinline__ void st_shared_zero16(uint32_t addr) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0) : "memory");
}

// grid (row blocks, feature tiles of NT).  What bounds it at N = 256 is the chain around one of
// the four expanded tiles (MMAs done, zero, barrier, scatter, MMAs), 0.46 us a tile against
// 0.34 for the MMAs at cuBLAS's rate.  Sixteen warps expand: a group of four owns an expanded tile
// and takes every fourth, so its chain has four tiles' time.  Measured on 16,384^2 at 90%, half in
// dense blocks, N = 256 (the 16 x 8 blocks + residual kernel before: 415 us): 264 us with two
// groups and entries loaded to registers a tile ahead, 170 with the entries copied to shared
// memory, 150 with four groups, 124 with the entry loop unpredicated, 119 with the MMAs issued
// from a uniform loop, 116 with an accumulator's tiles a constant of that loop.  (Accumulators ended tile by tile,
// by entries counted in the kernel: 143, in the loop's branches.)
template <int NT>
__global__ void __launch_bounds__(kThreads, 1) spmm_kernel(const __grid_constant__ CUtensorMap tmB,
                                                                         const Args a) {
    using SH = Shape<NT>;
    constexpr int S = kGroups, R = SH::R, SB = SH::SB, W = NT / kGroups;  // W: columns of the sums that a thread holds
    const int b = blockIdx.x;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *bring = smem + S * kATileBytes;  // (a group owns one expanded tile, and takes every fourth)
    uint32_t *ring = reinterpret_cast<uint32_t *>(bring + SB * SH::BT);
    int4 *hdr = reinterpret_cast<int4 *>(ring + SH::SLOTS * kSlot);  // per slot: words to skip, words, first, last entry
    uint64_t *full = reinterpret_cast<uint64_t *>(hdr + SH::SLOTS);  // a tile is expanded and its B rows landed
    uint64_t *empty = full + SB;                                         // ... and its MMAs are done
    uint64_t *cdone = empty + SB;                                        // an accumulator is complete
    uint64_t *bfree = cdone + 2;                                         // ... and drained
    uint64_t *efull = bfree + 2;                                         // a ring slot's entries landed
    uint32_t *tslot = reinterpret_cast<uint32_t *>(efull + SH::SLOTS);
    int *failed = reinterpret_cast<int *>(tslot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (a.t.bad && __ldg(a.t.bad + b)) {  // the block's entries were not regrouped
        if (tid == 0) a.marks[blockIdx.y * gridDim.x + b] = 1;
        return;
    }
    const int nst = a.nkt, lg = __ldg(a.t.chunk + b) >> (NT == 256 ? 4 : 0) & 15;  // log2 of an accumulator's tiles
    const int32_t *tp = a.t.tptr + (int64_t)b * (a.nkt + 1);
    const int n0 = blockIdx.y * NT;

    if (tid == 0) {
        for (int s = 0; s < SB; ++s) {
            mbar_init(&full[s], 1 + 4);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&cdone[i], 1);
            mbar_init(&bfree[i], kWorkers);
        }
        for (int i = 0; i < SH::SLOTS; ++i) mbar_init(&efull[i], 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
    }
    if (warp == 0) tmem_alloc(tslot, 2 * NT);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t taddr = *tslot;

    // Sums of the even and of the odd accumulators where the registers allow both, half as many
    // roundings each (error on 16,384^2 at 95%, N = 128: 1.37e-7 with one sum over accumulators of
    // 256 columns, 9.0e-8 with two over 512; the CSR kernel has 9.6e-8)
    constexpr int P = NT == 256 ? 1 : 2;
    float acc[P][W];
#pragma unroll
    for (int k = 0; k < P * W; ++k) acc[k / W][k % W] = 0.f;

    if (warp < kWorkers) {
        const int g = warp >> 2, t = tid & 127;
        const uint32_t tlane = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + g * W;
        const uint32_t at = smem_u32(smem + g * kATileBytes);
        bool ok = true;
        int drained = 0;
        auto drain = [&](int c) {  // adds accumulator c to the sums and frees its buffer
            const int buf = c & 1;
            ok = ok && __all_sync(FULL, mbar_wait(&cdone[buf], (c >> 1) & 1));
            if (!ok) return;
            fence_after_sync();
            auto add = [&](float (&sum)[W]) {
#pragma unroll
                for (int k = 0; k < W; k += 16) {
                    float r[16];
                    tmem_ld16(tlane + buf * NT + k, r);
#pragma unroll
                    for (int j = 0; j < 16; j += 2) {
                        const float2 v =
                            __fadd2_rn(make_float2(sum[k + j], sum[k + j + 1]), make_float2(r[j], r[j + 1]));
                        sum[k + j] = v.x;
                        sum[k + j + 1] = v.y;
                    }
                }
            };
            if (P == 1 || buf == 0)
                add(acc[0]);
            else
                add(acc[P - 1]);
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bfree[buf]);
        };
        // The group's first thread sends for tiles' entries (turn k's go to slot R * g + k % R) once
        // the whole group is past that slot's previous tile: a bulk copy from the 16-byte boundary
        // before the first entry.  A copy from HBM takes about a turn (1.6 us), so the entries
        // are brought to L2 three turns earlier.
        int sent = g, f0 = 0, f1 = 0, q0 = 0, q1 = 0;
        auto bounds = [&]() {  // of the next tile to send for and to bring to L2, a turn ahead
            if (sent < nst) {
                f0 = __ldg(tp + sent);
                f1 = __ldg(tp + sent + 1);
            }
            const int q = sent + kAhead * kGroups;
            q0 = q < nst ? __ldg(tp + q) & ~3 : 0;
            q1 = q < nst ? __ldg(tp + q + 1) : 0;
        };
        auto send = [&]() {
            if (q1 > q0) prefetch_l2(a.t.ent + q0, ((q1 - q0) * 4 + 15) & ~15);
            const int sl = R * g + sent / kGroups % R, skip = f0 & 3;
            const int words = min((f1 - f0 + skip + 3) & ~3, kSlot);
            hdr[sl] = make_int4(skip, f1 > f0 ? min(f1 - f0, kSlot - skip) : 0, f0, f1);
            if (f1 > f0) {
                mbar_expect_tx(&efull[sl], words * 4);
                bulk_load(ring + sl * kSlot, a.t.ent + (f0 - skip), words * 4, &efull[sl]);
            } else {
                mbar_arrive(&efull[sl]);
            }
            sent += kGroups;
            bounds();
        };
        if (t == 0) {
            bounds();
            while (sent < nst && sent < (R - 1) * kGroups) send();
        }
        int i = g;
        for (int turn = 0; i < nst; i += kGroups, ++turn) {
            const int sl = R * g + turn % R;
            if (turn > 0) ok = __all_sync(FULL, mbar_wait(&empty[(i - kGroups) % SB], (i - kGroups) / SB & 1)) && ok;
            if (ok) {
#pragma unroll
                for (int j = 0; j < kATileBytes / 16 / 128; ++j) st_shared_zero16(at + t * 16 + 2048 * j);
            }
            ok = bar_all(1 + g, 128, ok);
            if (!ok) break;
            if (t == 0 && sent < nst) send();
            ok = __all_sync(FULL, mbar_wait(&efull[sl], turn / R & 1));
            const int4 h = ok ? hdr[sl] : make_int4(0, 0, 0, 0);
            const uint32_t *e = ring + sl * kSlot + h.x + t;
            auto put = [&](uint32_t w) { st_shared_u16(at + (w & 0xffffu), (uint16_t)(w >> 16)); };
            int n = h.y;
#pragma unroll 1
            for (; n >= 512; n -= 512, e += 512) {
                const uint32_t w0 = e[0], w1 = e[128], w2 = e[256], w3 = e[384];
                put(w0);
                put(w1);
                put(w2);
                put(w3);
            }
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = t + 128 * j < n ? e[128 * j] : 0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (t + 128 * j < n) put(w[j]);
            for (int x = h.z + h.y + t; x < h.w; x += 128) put(__ldcs(a.t.ent + x));  // past the slot's words
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[i % SB]);
            // Accumulators that ended before this tile need nothing more of this group.  (The MMAs of tile i wait
            // for all groups to drain the accumulator before last, which ended by tile i - 2: a group reaches
            // that after it expanded a tile up to i + 2, for which it needs the MMAs of tiles up to i - 2.)
            while (ok && (drained + 1) << lg <= i) drain(drained++);
        }
        while (ok && drained << lg < nst) drain(drained++);
        if (!ok) {
            *failed = 1;
            if (t == 0)  // copies still on their way land before the CTA can leave
                for (int x = i; x < sent; x += kGroups)
                    mbar_wait(&efull[R * g + x / kGroups % R], x / kGroups / R & 1);
        }
    } else if (warp == kWorkers) {
        if (lane == 0) {
            int issued = 0;
            for (int i = 0; i < nst; ++i) {
                const int s = i % SB;
                if (i >= SB && !mbar_wait(&empty[s], (i / SB - 1) & 1)) {
                    *failed = 1;
                    break;
                }
                if (i == a.withhold && b == 0) break;  // nothing will complete full[s]
                mbar_expect_tx(&full[s], SH::BT);
#pragma unroll
                for (int f = 0; f < NT / 64; ++f)
                    tma_load_2d(bring + s * SH::BT + f * (kCols * 128), &tmB, &full[s], n0 + 64 * f, i * kCols);
                issued = i + 1;
            }
            // every issued copy lands before the CTA can leave (bounded waits)
            for (int i = issued - SB > 0 ? issued - SB : 0; i < issued; ++i) mbar_wait(&full[i % SB], (i / SB) & 1);
        }
    } else {
        // The whole warp walks the loop and one elected lane issues: the descriptors then stay in
        // uniform registers (a loop inside one lane's branch took about 80 clocks per MMA).
        // FP32 accumulator, BF16 A (K-major) and B (MN-major: transpose bit 16), M = 128, N = NT
        constexpr uint32_t kIdesc =
            (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(NT >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t ad0 = smem_desc(smem_u32(smem), 16, 1024), bd0 = smem_desc(smem_u32(bring), kCols * 128, 1024);
        const bool one = elect_one();
        bool ok = true;
        auto products = [&](auto log) {  // (a constant: what the loop tests stays uniform)
            constexpr int LG = decltype(log)::value;
            for (int i = 0; i < nst; ++i) {
                const int s = i % SB, c = i >> LG;
                const bool begins = i % (1 << LG) == 0;
                if (begins && c >= 2) ok = __all_sync(FULL, mbar_wait(&bfree[c & 1], ((c >> 1) - 1) & 1));
                ok = ok && __all_sync(FULL, mbar_wait(&full[s], (i / SB) & 1));
                if (!ok) break;
                fence_after_sync();
                const uint64_t ad = ad0 + (uint32_t)(i % S) * (kATileBytes >> 4), bd = bd0 + (uint32_t)s * (SH::BT >> 4);
                if (one) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        mma_bf16(taddr + (c & 1) * NT, ad + j * 2, bd + j * 128, kIdesc, (!begins || j) ? 1u : 0u);
                    mma_commit(&empty[s]);
                    if ((i + 1) % (1 << LG) == 0 || i == nst - 1) mma_commit(&cdone[c & 1]);
                }
                __syncwarp();
            }
        };
        switch (lg) {
            case 0: products(Int<0>{}); break;
            case 1: products(Int<1>{}); break;
            case 2: products(Int<2>{}); break;
            default: products(Int<kLogChunk>{});
        }
        if (!ok && one) *failed = 1;
    }
    __syncwarp();
    bool fine = true;
    if (warp < kWorkers) {
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if constexpr (P == 2) acc[0][k] += acc[1][k];
            fine &= (__float_as_uint(acc[0][k]) & 0x7f800000u) != 0x7f800000u;
        }
    }
    fence_before_sync();
    fine = __syncthreads_and(fine);
    fence_after_sync();
    if (warp == 0) tmem_dealloc(taddr, 2 * NT);
    if (tid == 0) {
        a.marks[blockIdx.y * gridDim.x + b] = *failed || !fine;
        if (*failed && a.err) atomicExch(a.err, 1);
    }
    if (*failed || !fine) return;
    const int row = b * kRows + 32 * (warp & 3) + lane;
    if (warp >= kWorkers || row >= a.M) return;
    const int c0 = n0 + (warp >> 2) * W;
    float *dst = a.C + (int64_t)row * a.ldc + c0;
#pragma unroll
    for (int k = 0; k < W; k += 8) {
        if (c0 + k >= a.N) break;
        if (a.vec == 8) {
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + k), "f"(acc[0][k]),
                         "f"(acc[0][k + 1]), "f"(acc[0][k + 2]), "f"(acc[0][k + 3]), "f"(acc[0][k + 4]), "f"(acc[0][k + 5]),
                         "f"(acc[0][k + 6]), "f"(acc[0][k + 7])
                         : "memory");
        } else if (a.vec == 4) {
            *reinterpret_cast<float4 *>(dst + k) = make_float4(acc[0][k], acc[0][k + 1], acc[0][k + 2], acc[0][k + 3]);
            *reinterpret_cast<float4 *>(dst + k + 4) = make_float4(acc[0][k + 4], acc[0][k + 5], acc[0][k + 6], acc[0][k + 7]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[k + j] = acc[0][k + j];
        }
    }
}

// The marked row blocks, from the CSR arrays: a warp per row, 256 columns per pass (N a
// multiple of 8).  Usually no block is marked and the CTAs leave at once.
__global__ void __launch_bounds__(256) marked_rows_kernel(const SpmmProblem P, const int32_t *marks, int nb, int tiles,
                                                          int vec_c) {
    int marked = 0;
    for (int y = 0; y < tiles; ++y) marked |= __ldg(marks + y * nb + blockIdx.x / (kRows / 8));
    if (!marked) return;
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= P.M) return;
    const int64_t p0 = __ldg(P.rowptr + row), p1 = __ldg(P.rowptr + row + 1);
    const int col = blockIdx.y * 256 + lane * 8;
    float acc[1][8] = {};
    spmm_detail::gather_range<BF16, 32, 1, 8, true>(P, p0, p1, acc, lane, col);
    float *dst = P.C + (int64_t)row * P.ldc;
    if (vec_c) {
        spmm_detail::store_row<BF16, 32, 1>(dst, acc, lane, col, P.N, 1.0f);
    } else if (col < P.N) {
#pragma unroll
        for (int k = 0; k < 8; ++k) dst[col + k] = acc[0][k];
    }
}

template <int NT>
int launch_nt(const CUtensorMap &map, const Args &a, int nb, cudaStream_t s) {
    using SH = Shape<NT>;
    static std::once_flag once[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return fail(GBSP_ERR_UNSUPPORTED, "tc dense: device ordinal %d", dev);
    std::call_once(once[dev], [] {
        cudaFuncSetAttribute(spmm_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SH::SMEM);
    });
    spmm_kernel<NT><<<dim3((unsigned)nb, (unsigned)((a.N + NT - 1) / NT)), kThreads, SH::SMEM, s>>>(map, a);
    count_launches(1);
    return check_launch("tc dense spmm kernel");
}

}  // namespace

bool tiles_fit(int64_t M, int64_t K, int64_t nnz) {
    return M > 0 && K > 0 && nnz < (1LL << 31) - 4096 && col_tiles(K) <= kMaxTiles &&
           row_blocks(M) * (col_tiles(K) + 1) < (1LL << 31);
}

// Error of the product against 64 bits (relative 2-norm in units of 1e-8, squared) for rows of n entries, e of them
// to an accumulator: what the accumulators lose, and the rounding of the sums of n / e of them (two of half
// as many up to 128 features).  Within 4% of the errors measured at 2,048 to 24,000 columns and 2.5 to 40%
// of entries, evenly spread.
static double tile_error2(double n, double e, bool wide) {
    return 0.98 * e + 0.00725 * e * e + (wide ? 3.1 : 1.64) * n / e;
}

// Entries of a row that an accumulator takes: up to where halving them would lessen that error (by 4% or 10% of
// the rounding more than it costs).
static double entries_per_sum(double n, bool wide) {
    double lo = 0, hi = kChunk * kCols;
    for (int i = 0; i < 20; ++i) {
        const double e = 0.5 * (lo + hi);
        (0.49 * e + 0.00544 * e * e <= (wide ? 3.4 : 1.7) * n / e ? lo : hi) = e;
    }
    return lo;
}

// ... of accumulators over 512 columns or a half, a quarter, an eighth of evenly spread rows.
static double entries_evenly(double n, int64_t K, bool wide) {
    const double most = entries_per_sum(n, wide);
    double e = n * kChunk * kCols / (double)K;
    for (int k = 0; k < kLogChunk && e > most; ++k) e *= 0.5;
    return e;
}

// The entries of a block's rows past which an accumulator's columns are halved: what evenly spread rows have
// there, with room for their scatter (outputs do not change from block to block), or what suits the
// accumulator if that is more.
// 16,384 columns, 256 features: 512 columns up to 15% of entries; at 30%, 256 (error 1.44e-7 for 1.9e-7); a band of
// 600 entries a row of 4,096 columns, one sign: 64 columns.
static int sum_limit(int64_t M, int64_t K, int64_t nnz, bool wide) {
    const double n = (double)nnz / (double)M, even = 1.3 * entries_evenly(n, K, wide), most = entries_per_sum(n, wide);
    return (int)(kRows * (even > most ? even : most));
}

// Time against time, in microseconds: a tile takes 0.30 / 0.38 / 0.46 at 64 / 128 / 256 features
// whatever it holds, one CTA per SM, and a pair of launches 5 (measured on 2,048 to 24,000 rows and
// columns).
static double product_us(int64_t M, int64_t K, int64_t N, int64_t *waves) {
    const int sms = sm_count() > 0 ? sm_count() : 1;
    *waves = (row_blocks(M) * ((N + 255) / 256) + sms - 1) / sms;
    return (double)(*waves * col_tiles(K)) * (N <= 64 ? 0.30 : N <= 128 ? 0.38 : 0.46) + 5.0;
}

// Whether the sums are as exact as the CSR kernels', which split a row among 8, 4 or 2 lane groups at 64,
// 128 or 256 features: their squared error is 0.116 / 0.207 / 0.37 n at 128 / 256 / more features (within 3%
// of the measured ones).  At 128 features that is from about 660 entries a row on (660 of 2,049 columns: 8.6e-8
// both; 600 of 5,000 at 12%: 8.0e-8 against 8.3e-8), at 256 from about 360 (12,288 columns at 4%: 9.5e-8 against
// 1.0e-7; 3,000 at 11%: 8.5e-8 against 8.2e-8), but not on so few entries per tile that the rounding of the
// sums outweighs (16,384 columns at 2.5%, 256 features: 9.6e-8 against 9.2e-8).
// With values and B of one sign the CSR kernels' rounding does not add up and the accumulators' loss
// does: on the same sizes 0.4 to 0.95 of the CSR kernels' error from 129 features on, 0.7 to 1.3 at 128.
static bool sums_as_well(int64_t M, int64_t K, int64_t N, int64_t nnz) {
    if (N < 128) return false;
    const double n = (double)nnz / (double)M;
    return tile_error2(n, entries_evenly(n, K, N > 128), N > 128) <= (N <= 128 ? 0.116 : N <= 256 ? 0.207 : 0.37) * n;
}

// The plan's blocks and CSR residual take 6.8 / 9.0 / 15.9 ps per entry at 64 / 128 / 256 features
// where they do best (clustered, 5%), more on unstructured rows (11 / 13 / 20).  On 16,384^2 the
// lines cross near 6.5% / 5% / 3% of entries.
static bool faster(int64_t M, int64_t K, int64_t N, int64_t nnz) {
    if (M < 2048 || K < 2048 || N < 64 || N > 512 || (double)nnz < 0.03 * (double)M * (double)K) return false;
    int64_t waves;
    return product_us(M, K, N, &waves) < 0.9e-6 * (double)nnz * (2.5 + 0.05 * (double)N);
}

// The blocks' MMAs run one accumulator over all of a row's entries in blocks, the share s of them, and so lose
// about s^2 K / 512 times what whole tiles do: at 512 the errors are level (2,048 columns, half in
// blocks: 1.00 at 2.5% of entries, 0.79 at 10%), above that whole tiles have the smaller one (0.13 of it
// on 16,384 columns at 10%), below it only where their sums are as exact as the CSR kernels', which
// then have most of the entries (8% of 3,072 columns, a fifth in blocks: 6.2e-8 against 7.3e-8 at 64 features).
static bool no_less_exact(int64_t M, int64_t K, int64_t N, int64_t nnz, int64_t dense_nnz) {
    const double share = (double)dense_nnz / (double)nnz;
    return (double)K * share * share >= kChunk * kCols || sums_as_well(M, K, N, nnz);
}

bool spmm_pays(int64_t M, int64_t K, int64_t N, int64_t nnz, int64_t dense_nnz) {
    return faster(M, K, N, nnz) && no_less_exact(M, K, N, nnz, dense_nnz);
}

bool spmm_may_pay(int64_t M, int64_t K, int64_t nnz, int64_t dense_nnz) {
    return faster(M, K, 256, nnz) &&
           (no_less_exact(M, K, 256, nnz, dense_nnz) || no_less_exact(M, K, 512, nnz, dense_nnz));
}

// For rows of even length (the split AUTO would take is the row split).  The regrouping takes 0.5 ns
// per entry of a block of rows, the row split 13 / 24 ps per entry at 128 / 256 features: on
// 16,384^2 the lines cross near 4.5% / 2.5% of entries, on 8,192^2 near 11% / 5%.
bool spmm_pays_unplanned(int64_t M, int64_t K, int64_t N, int64_t nnz) {
    if (M < 2048 || K < 2048 || N > 512 || !sums_as_well(M, K, N, nnz)) return false;
    int64_t waves;
    const double product = product_us(M, K, N, &waves);
    const double bins = (double)waves * 0.5e-3 * (double)nnz / (double)row_blocks(M);
    return product + bins + scratch_us(4 * nnz) < 0.85e-6 * (double)nnz * (2.3 + 0.085 * (double)N);
}

int launch_bin(const int32_t *rowptr, const int32_t *colidx, const uint16_t *vals, int64_t M, int64_t K, int64_t nnz,
               Tiles t, cudaStream_t s) {
    const int nkt = (int)col_tiles(K);
    const int2 limit = make_int2(sum_limit(M, K, nnz, false), sum_limit(M, K, nnz, true));
    const auto kernel = !t.pos ? bin_kernel<true, false> : vals ? bin_kernel<true, true> : bin_kernel<false, true>;
    kernel<<<(unsigned)row_blocks(M), kBinThreads, sizeof(int32_t) * nkt, s>>>(rowptr, colidx, vals, (int)M, (int)K, nkt,
                                                                               t, limit);
    count_launches(1);
    return check_launch("tc dense regrouping");
}

int launch_spmm(const SpmmProblem &p, Tiles t, int32_t *marks, int *err, int withhold, cudaStream_t s) {
    if (p.N % 8 || p.ldb % 8 || !aligned16(p.B))
        return fail(GBSP_ERR_ALIGN, "tc dense: N and ld multiples of 8 and a 16-byte aligned B");
    EncodeTiledFn enc = encode_fn();
    if (!enc) return fail(GBSP_ERR_CUDA, "tc dense: cuTensorMapEncodeTiled is not available");
    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)p.N, (cuuint64_t)p.K};
    const cuuint64_t strides[1] = {(cuuint64_t)p.ldb * 2};
    const int nt = p.N <= 64 ? 64 : p.N <= 128 ? 128 : 256;
    const cuuint32_t box[2] = {64, kCols};
    const cuuint32_t estr[2] = {1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(p.B), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return fail(GBSP_ERR_CUDA, "tc dense: tensor map encoding failed");
    const bool c16 = aligned16(p.C) && p.ldc % 4 == 0;
    Args a{t, marks, p.C, p.ldc, p.M, p.N, (int)col_tiles(p.K), aligned32(p.C) && p.ldc % 8 == 0 ? 8 : c16 ? 4 : 1, err,
           withhold};
    const int nb = (int)row_blocks(p.M);
    int st = nt == 64 ? launch_nt<64>(map, a, nb, s) : nt == 128 ? launch_nt<128>(map, a, nb, s)
                                                                  : launch_nt<256>(map, a, nb, s);
    if (st) return st;
    marked_rows_kernel<<<dim3((unsigned)nb * (kRows / 8), (unsigned)((p.N + 255) / 256)), 256, 0, s>>>(
        p, marks, nb, (p.N + nt - 1) / nt, c16);
    count_launches(1);
    return check_launch("tc dense marked rows");
}

}  // namespace dense
}  // namespace gbsp
