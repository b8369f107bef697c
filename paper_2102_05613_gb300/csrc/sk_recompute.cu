// sk_recompute.cu -- the periodic local-field recompute H = S J^T of all
// chains of a run on the fifth-generation tensor cores (tcgen05), and the
// drift check / resynchronisation of the maintained fields against it.
//
// H[c][n] = sum_k S[c][k] J[n][k] (J symmetric), M = chains, N = K = Npad.
//   +-J couplings:     S and J as FP8 e4m3 (+-1 and 0 are exact), kind::f8f6f4,
//                      FP32 accumulation: every partial sum is an integer below
//                      2^24, so H is exact and must equal the maintained int32
//                      fields bit for bit.
//   Gaussian couplings: S as bf16 (+-1 exact), J split into `terms` bf16
//                      matrices J = J1 + J2 + J3 (three round-to-nearest terms
//                      reproduce every fp32 value exactly), kind::f16 with FP32
//                      accumulation of all terms into one accumulator.
//
// A persistent CTA per SM works through 128 x 256 output tiles with three
// roles: one thread of warp 0 streams A and B tiles with TMA (128-byte
// swizzle) through a 4-stage mbarrier ring, one thread of warp 1 issues the
// MMAs (K = 32 bytes each) into one of two 128-lane x 256-column FP32
// accumulators in tensor memory (all 512 columns) and commits each stage back
// to its "empty" barrier and each finished tile to its accumulator's "full"
// barrier, and warps 2-9 (two per 32-lane quadrant of tensor memory, one per
// half of the columns) read the finished accumulator with tcgen05.ld and
// compare it with (or replace) the maintained fields, then hand the
// accumulator back -- so one tile's epilogue overlaps the next tile's main
// loop, with eight warps' loads of the fields in flight.  Every wait is bounded; an expired wait
// sets the run's error word and stops the CTA's roles.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <numeric>
#include <cstring>
#include <mutex>
#include <set>
#include <vector>

#include "sk_device.cuh"
#include "sk_internal.h"

namespace sk {
namespace {

constexpr uint32_t BM = 128, BN = 256, NS = 4;  // 4 pipeline stages, one CTA per SM
constexpr uint32_t TILE_A = BM * 128, TILE_B = BN * 128;  // bytes, 128 B of K per row
constexpr uint32_t STAGE_BYTES = TILE_A + TILE_B;
constexpr uint32_t EW = 8;                                 // epilogue warps: 2 per tensor-memory quadrant
constexpr uint32_t SMEM_BYTES = NS * STAGE_BYTES + 1024;  // + 1 KB alignment slack
constexpr uint32_t TMEM_COLS = 512;                        // two 256-column accumulators
constexpr uint32_t WS_THREADS = 64 + 32 * EW;              // producer, MMA, epilogue warps
// MT row blocks of 128 per tile.  MT = 1: two accumulators take tiles in turn.
// MT = 2: a tile is 256 rows, each B tile in shared memory serves two MMAs, one
// per accumulator: 64 KB instead of 96 KB from L2 for the same products, where
// the main loop is bound by what an SM takes in from L2 (~64 B per clock).  Its
// epilogue does not overlap the next tile's main loop, so it is the choice
// for long sums and many rows (bf16, tall_tiles).  Stages: 192 KB either way.
template <int MT>
struct Tile {
    static constexpr uint32_t kStages = MT == 1 ? NS : 3u;
    static constexpr uint32_t kStageBytes = MT * TILE_A + TILE_B;
    static constexpr uint32_t kRows = MT * BM;
};
static_assert(Tile<2>::kStages * Tile<2>::kStageBytes == NS * STAGE_BYTES, "same shared memory");
constexpr long long kBudget = 4000000000ll;  // ~2 s of clock cycles per wait

__device__ __forceinline__ uint32_t saddr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity) {
    if (try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!try_wait(bar, parity))
        if (clock64() - t0 > kBudget) return false;
    return true;
}
__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
// Shared-memory matrix descriptor: K-major tile, 128-byte rows with the
// 128-byte swizzle, 8-row groups 1024 bytes apart (tile base 1024-aligned).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);  // start address
    d |= static_cast<uint64_t>(1) << 16;                 // leading byte offset (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;         // stride byte offset
    d |= static_cast<uint64_t>(1) << 46;                 // descriptor version
    d |= static_cast<uint64_t>(2) << 61;                 // 128-byte swizzle
    return d;
}
// Instruction descriptor: FP32 accumulator, A/B format code `fmt` (kind::f16:
// 1 = bf16; kind::f8f6f4: 0 = e4m3), both K-major, N = 256, M = 128.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t fmt) {
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((BN >> 3) << 17) | ((BM >> 4) << 24);
}

template <bool F8>
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    if constexpr (F8) {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(a), "l"(b), "r"(idesc), "r"(acc));
    } else {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(a), "l"(b), "r"(idesc), "r"(acc));
    }
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

struct Args {
    void* h;                        // maintained fields [chains][npad]: int32 (+-J) or float
    const int8_t* s;                // spins [chains][npad]
    float* out;                     // OUTPUT mode: H [chains][npad]
    double* dE;                     // per chain: sum_n s_n (h_n - H_n)
    unsigned long long* stats;      // [0] max |h - H| (double bits), [1] mismatches, [2] max |dE|
    unsigned int* cnt;              // per 32 chains: epilogue warps done with their rows (or null)
    double scale;                   // energy scale of the drift
    int* err;
    uint32_t chains, npad, kblocks, terms, mode;  // mode: 0 check, 1 resync, 2 output, 3 set fields
    uint32_t pm1;
    uint32_t fault;                 // kFaultWithholdTile: tests of the bounded waits
    uint32_t compute_only;          // tensor-pipe probe: operands loaded once, MMAs only
    // energies (KIND 2): digit slices of J (device word, 0: none), and per
    // slice and configuration the sum over n of s_n H_n
    const uint32_t* nslices;
    unsigned long long* esum;
    uint32_t esum_stride;           // configurations in all (chains: those of this launch)
    uint32_t b_row0, b_rows;        // the rows of J whose slices B holds
};

// Several operand sets in one launch: the tensor maps and arguments of each
// set in global memory (maps 64-byte aligned, written before the launch).
struct alignas(64) BatchJob {
    CUtensorMap A, B[3];
    Args args;
};
struct BatchTask {
    uint32_t job, m0, n0, pad;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Byte e (0..3) of a 32-bit word as a signed value.
__device__ __forceinline__ int sbyte32(uint32_t w, int e) {
    return static_cast<int>(static_cast<int32_t>(w << (24 - 8 * e)) >> 24);
}
__device__ __forceinline__ uint32_t word_of(const uint4& q, int e) {
    return e == 0 ? q.x : e == 1 ? q.y : e == 2 ? q.z : q.w;
}

// The epilogue of one finished accumulator for one warp: accumulator rows
// row0 .. row0 + 31 (tcgen05.ld 32x32b gives lane l the accumulator row
// row0 + l), the NCB blocks of 32 columns starting at column c0.  Each lane
// reads and writes its own row's segment of the fields and spins -- 128
// bytes of int32 / float fields as eight 16-byte loads and 32 bytes of spins
// as two -- so no transpose is needed, and the row's sum s (h - H) stays in
// the lane (an int32 for +-J, exact; a float otherwise) until one
// double-precision atomic per row.  A block's loads are issued before its
// accumulator columns are read from tensor memory (the first block's before
// the wait for the accumulator), so that their round trip covers that read.
constexpr uint32_t NCB = BN / 2 / 32;  // column blocks per epilogue warp and tile
// One column block's fields and spins of this lane's row (check and resync).
struct RowBlock {
    uint4 h[8], s[2];
};
__device__ __forceinline__ void load_row_block(RowBlock& rb, const Args& args, uint32_t row, uint32_t n, bool ok) {
    if (args.mode < 2 && ok && n < args.npad) {  // npad is a multiple of 32
        const size_t idx = static_cast<size_t>(row) * args.npad + n;  // 32-element aligned
        const uint4* hp = reinterpret_cast<const uint4*>(static_cast<const unsigned int*>(args.h) + idx);
#pragma unroll
        for (int q = 0; q < 8; ++q) rb.h[q] = __ldg(hp + q);
        const uint4* sp = reinterpret_cast<const uint4*>(args.s + idx);
        rb.s[0] = __ldg(sp);
        rb.s[1] = __ldg(sp + 1);
    }
}
// Four accumulator values as maintained fields: int32 for +-J, float32 else.
__device__ __forceinline__ uint4 field_words(const uint32_t (&v)[32], int q, uint32_t pm1) {
    uint4 w = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    if (pm1) {
        w.x = static_cast<uint32_t>(__float2int_rn(__uint_as_float(w.x)));
        w.y = static_cast<uint32_t>(__float2int_rn(__uint_as_float(w.y)));
        w.z = static_cast<uint32_t>(__float2int_rn(__uint_as_float(w.z)));
        w.w = static_cast<uint32_t>(__float2int_rn(__uint_as_float(w.w)));
    }
    return w;
}
// first: the first column block, loaded by the caller (before it waited for
// the accumulator) with load_row_block(first, args, row0 + lane, n0 + c0, ..).
__device__ __forceinline__ void epilogue_rows(uint32_t taddr, const Args& args, uint32_t row0, uint32_t n0,
                                              uint32_t c0, bool tile_ok, const RowBlock& first) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t row = row0 + lane;
    const bool row_ok = tile_ok && row < args.chains;
    const bool reads = args.mode < 2;
    int isum = 0, imax = 0;
    float fsum = 0.0f, pmax = 0.0f;
    unsigned mism = 0;
    RowBlock rb = first;
#pragma unroll
    for (uint32_t cb = 0; cb < NCB; ++cb) {
        if (cb > 0) load_row_block(rb, args, row, n0 + c0 + 32u * cb, row_ok);
        const uint32_t n = n0 + c0 + 32u * cb;
        const bool ok = row_ok && n < args.npad;
        const size_t idx = static_cast<size_t>(row) * args.npad + n;
        uint32_t v[32];
        tmem_ld32(taddr + c0 + 32u * cb, v);  // every lane: the load is warp-collective
        if (!ok) continue;
        if (args.mode >= 2) {  // output H, or the fields of a start state (h = H)
            uint4* dst = args.mode == 2 ? reinterpret_cast<uint4*>(args.out + idx)
                                        : reinterpret_cast<uint4*>(static_cast<unsigned int*>(args.h) + idx);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                dst[q] = args.mode == 3 ? field_words(v, q, args.pm1)
                                        : make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            continue;
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const float H = __uint_as_float(v[k]);
            const uint32_t hw = word_of(rb.h[k >> 2], k & 3);
            const int sv = sbyte32(word_of(rb.s[k >> 4], (k >> 2) & 3), k & 3);
            if (args.pm1) {
                const int d = static_cast<int>(hw) - __float2int_rn(H);
                mism += d != 0;
                imax = max(imax, abs(d));
                isum += sv * d;
            } else {
                const float d = __uint_as_float(hw) - H;
                pmax = fmaxf(pmax, fabsf(d));
                fsum = fmaf(static_cast<float>(sv), d, fsum);
            }
        }
        if (args.mode == 1) {  // resync: the maintained fields become H
            uint4* dst = reinterpret_cast<uint4*>(static_cast<unsigned int*>(args.h) + idx);
#pragma unroll
            for (int q = 0; q < 8; ++q) dst[q] = field_words(v, q, args.pm1);
        }
    }
    if (tile_ok && reads) {
        if (row_ok) atomicAdd(&args.dE[row], args.pm1 ? static_cast<double>(isum) : static_cast<double>(fsum));
        // the warp's maximum and mismatch count, then one atomic each (every
        // warp of every tile updates the same two words)
        if (args.pm1) {
            imax = __reduce_max_sync(0xffffffffu, imax);
        } else {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) pmax = fmaxf(pmax, __shfl_xor_sync(0xffffffffu, pmax, o));
        }
        const unsigned mw = __reduce_add_sync(0xffffffffu, mism);
        if (lane == 0) {
            const double dmax = args.pm1 ? static_cast<double>(imax) : static_cast<double>(pmax);
            atomicMax(&args.stats[0], static_cast<unsigned long long>(__double_as_longlong(dmax)));
            if (mw) atomicAdd(&args.stats[1], static_cast<unsigned long long>(mw));
        }
        if (args.cnt && row0 < args.chains) {
            // the energy drift of these 32 chains is complete once the epilogue
            // warps of all their tiles (two column halves each) have added to
            // it: the last of them takes |scale/2 dE| of each chain into the
            // maximum and clears dE and the count for the next recompute
            const uint32_t arrivals = 2u * ((args.npad + BN - 1) / BN);
            unsigned last = 0;
            __syncwarp();
            if (lane == 0) {
                __threadfence();
                last = atomicAdd(&args.cnt[row0 / 32u], 1u) == arrivals - 1u;
            }
            last = __shfl_sync(0xffffffffu, last, 0);
            if (last) {
                __threadfence();
                double e = 0.0;
                if (row < args.chains)
                    e = fabs(0.5 * args.scale * __longlong_as_double(static_cast<long long>(
                                                    atomicExch(reinterpret_cast<unsigned long long*>(&args.dE[row]), 0ull))));
                unsigned long long bmax = static_cast<unsigned long long>(__double_as_longlong(e));
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long y = __shfl_xor_sync(0xffffffffu, bmax, o);
                    bmax = y > bmax ? y : bmax;
                }
                if (lane == 0) {
                    atomicMax(&args.stats[2], bmax);  // non-negative doubles order as their bits
                    args.cnt[row0 / 32u] = 0u;
                }
            }
        }
    }
    __syncwarp();
}

// The energy epilogue for one warp: each lane adds s_n H_n of its row over the
// warp's columns in int32 (H is an integer of at most 2^20: 128 columns stay
// below 2^27) and adds the sum to the row's 64-bit word, exact in any order.
__device__ __forceinline__ void energy_rows(uint32_t taddr, const Args& args, uint32_t row0, uint32_t n0, uint32_t c0,
                                            uint32_t slice, bool tile_ok) {
    const uint32_t row = row0 + (threadIdx.x & 31);
    const bool row_ok = tile_ok && row < args.chains;
    int isum = 0;
#pragma unroll
    for (uint32_t cb = 0; cb < NCB; ++cb) {
        const uint32_t n = n0 + c0 + 32u * cb;
        const bool ok = row_ok && n < args.npad;
        uint4 sp[2];
        if (ok) {
            const uint4* p = reinterpret_cast<const uint4*>(args.s + static_cast<size_t>(row) * args.npad + n);
            sp[0] = __ldg(p);
            sp[1] = __ldg(p + 1);
        }
        uint32_t v[32];
        tmem_ld32(taddr + c0 + 32u * cb, v);  // every lane: the load is warp-collective
        if (!ok) continue;
#pragma unroll
        for (int k = 0; k < 32; ++k)
            isum += sbyte32(word_of(sp[k >> 4], (k >> 2) & 3), k & 3) * __float2int_rn(__uint_as_float(v[k]));
    }
    if (row_ok && isum)
        atomicAdd(&args.esum[static_cast<size_t>(slice) * args.esum_stride + row],
                  static_cast<unsigned long long>(static_cast<long long>(isum)));
    __syncwarp();
}

// The persistent kernel.  KIND 1 (a batch): task t is tasks[t] of operand set
// jobs[tasks[t].job] (maps in global memory, acquired before use).  KIND 0:
// the maps and arguments are the kernel's parameters and task t is output
// tile (t / tiles_n, t % tiles_n).  KIND 2 (energies): B holds the digit
// slices of the strict upper triangle of J one below the other; a task is one
// slice of one output tile, whose K range starts at the tile's own columns
// (what lies before them is zero), and the tasks with the longest range come
// first, so that the last round of the persistent CTAs is a short one.
template <bool F8, int KIND, int MT = 1>
__global__ void __launch_bounds__(WS_THREADS, 1)
    recompute_ws_kernel(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB0,
                        const __grid_constant__ CUtensorMap tB1, const __grid_constant__ CUtensorMap tB2,
                        const Args args0, const BatchJob* __restrict__ jobs, const BatchTask* __restrict__ tasks,
                        uint32_t ntasks, uint32_t tiles_n) {
    constexpr bool BATCH = KIND == 1;
    constexpr bool ENERGY = KIND == 2;
    constexpr uint32_t kNS = Tile<MT>::kStages, kSB = Tile<MT>::kStageBytes;
    static_assert(MT == 1 || (!F8 && !ENERGY), "256-row tiles: bf16 recompute");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kNS], empty[kNS], tfull[2], tempty[2], drain;
    __shared__ uint32_t tmem_holder;
    __shared__ int dead;
    // 128-byte-swizzled tiles must start on a 1024-byte boundary of shared memory
    unsigned char* smem = smem_raw + ((1024u - (saddr(smem_raw) & 1023u)) & 1023u);
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr uint32_t kElems = F8 ? 128u : 64u;  // K elements per 128-byte row
    constexpr uint32_t idesc = instr_desc(F8 ? 0u : 1u);
    volatile int* vdead = &dead;

    if (threadIdx.x == 0) {
        for (uint32_t i = 0; i < kNS; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty[i])) : "memory");
        }
        for (uint32_t i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&tfull[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(&tempty[i])), "r"(EW) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&drain)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        dead = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_holder)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;

    const uint32_t tiles_m = ENERGY ? (args0.chains + BM - 1) / BM : 0u;
    const uint32_t slices = ENERGY ? *args0.nslices : 0u;
    if constexpr (ENERGY) ntasks = slices * tiles_m * tiles_n;
    // energies: the slice of task t
    auto slice_of = [&](uint32_t t) -> uint32_t { return ENERGY ? (t / tiles_m) % slices : 0u; };
    // the task's maps, arguments and tile origin
    auto task = [&](uint32_t t, const CUtensorMap*& A, const CUtensorMap* (&B)[3], const Args*& a, uint32_t& m0,
                    uint32_t& n0) {
        if constexpr (BATCH) {
            const BatchTask tk = tasks[t];
            const BatchJob& j = jobs[tk.job];
            A = &j.A;
            B[0] = &j.B[0];
            B[1] = &j.B[1];
            B[2] = &j.B[2];
            a = &j.args;
            m0 = tk.m0;
            n0 = tk.n0;
        } else {
            A = &tA;
            B[0] = &tB0;
            B[1] = &tB1;
            B[2] = &tB2;
            a = &args0;
            if constexpr (ENERGY) {
                m0 = (t % tiles_m) * BM;
                n0 = a->b_row0 + (t / (tiles_m * slices)) * BN;
            } else {
                m0 = (t / tiles_n) * (MT * BM);
                n0 = (t % tiles_n) * BN;
            }
        }
    };

    if (warp == 0) {
        if (lane == 0) {  // producer: A (spins) and B (couplings, term by term) tiles by TMA
            uint32_t g = 0;
            uint32_t withheld = 0xFFFFFFFFu;  // a stage a test of the bounded waits leaves unfilled
            for (uint32_t t = blockIdx.x; t < ntasks && !*vdead; t += gridDim.x) {
                const CUtensorMap* A;
                const CUtensorMap* B[3];
                const Args* a;
                uint32_t m0, n0;
                task(t, A, B, a, m0, n0);
                if constexpr (BATCH) {  // maps written to global memory by a copy: acquire them for TMA
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(A) : "memory");
                    for (int q = 0; q < 3; ++q)
                        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(B[q]) : "memory");
                }
                const uint32_t kb0 = ENERGY ? n0 / kElems : 0u;  // (n0: a multiple of BN)
                const uint32_t total = ENERGY ? a->kblocks - kb0 : a->terms * a->kblocks;
                const uint32_t brow = ENERGY ? slice_of(t) * a->b_rows + n0 - a->b_row0 : n0;
                for (uint32_t i = 0; i < total; ++i, ++g) {
                    const uint32_t st = g % kNS;
                    if (a->compute_only && g >= kNS) break;  // the probe fills the ring once
                    if (g >= kNS && !wait_bounded(saddr(&empty[st]), ((g / kNS) - 1u) & 1u)) {
                        atomicExch(a->err, kDevTimeout);
                        *vdead = 1;
                    }
                    if (*vdead) break;
                    if ((a->fault & kFaultWithholdTile) && blockIdx.x == 0 && g == 0) {
                        withheld = g;
                        continue;
                    }
                    const uint32_t term = ENERGY ? 0u : i / a->kblocks, kb = ENERGY ? kb0 + i : i % a->kblocks;
                    unsigned char* sa = smem + st * kSB;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(&full[st])),
                                 "r"(kSB)
                                 : "memory");
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
                        tma_2d(saddr(sa + mt * TILE_A), A, static_cast<int>(kb * kElems),
                               static_cast<int>(m0 + mt * BM), saddr(&full[st]));
                    tma_2d(saddr(sa + MT * TILE_A), B[term], static_cast<int>(kb * kElems), static_cast<int>(brow),
                           saddr(&full[st]));
                }
            }
            // the copies of the last stages issued have landed before the
            // CTA may leave (at once after a normal run, where the MMA warp
            // consumed them; bounded after an expired wait)
            for (uint32_t q = g > kNS ? g - kNS : 0u; q < g; ++q)
                if (q != withheld) wait_bounded(saddr(&full[q % kNS]), (q / kNS) & 1u);
        }
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issuer: 4 MMAs of K = 32 bytes per stage into accumulator j % 2
            uint32_t g = 0, j = 0;
            for (uint32_t t = blockIdx.x; t < ntasks && !*vdead; t += gridDim.x, ++j) {
                const CUtensorMap* A;
                const CUtensorMap* B[3];
                const Args* a;
                uint32_t m0, n0;
                task(t, A, B, a, m0, n0);
                // MT = 1: accumulator j % 2; MT = 2: both, one tile at a time
                const uint32_t b = MT == 1 ? j & 1u : 0u, use = MT == 1 ? j >> 1 : j;
                if (use >= 1 && !wait_bounded(saddr(&tempty[b]), (use - 1u) & 1u)) {  // epilogue done with it
                    atomicExch(a->err, kDevTimeout);
                    *vdead = 1;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem + 256u * b;
                const uint32_t total = ENERGY ? a->kblocks - n0 / kElems : a->terms * a->kblocks;
                for (uint32_t i = 0; i < total; ++i, ++g) {
                    const uint32_t st = g % kNS;
                    // (the probe waits for each stage once, then reuses it)
                    if ((!a->compute_only || g < kNS) && !wait_bounded(saddr(&full[st]), (g / kNS) & 1u)) {
                        atomicExch(a->err, kDevTimeout);
                        *vdead = 1;
                    }
                    if (*vdead) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = saddr(smem + st * kSB);
                    const uint32_t sb = sa + MT * TILE_A;
#pragma unroll
                    for (uint32_t kk = 0; kk < 4; ++kk)
#pragma unroll
                        for (uint32_t mt = 0; mt < MT; ++mt)
                            mma<F8>(acc + 256u * mt, sw128_desc(sa + mt * TILE_A + 32 * kk), sw128_desc(sb + 32 * kk),
                                    idesc, (i | kk) != 0u);
                    if (!a->compute_only) mma_commit(saddr(&empty[st]));
                }
                mma_commit(saddr(&tfull[b]));  // completes when the tile's MMAs have
            }
            // every MMA issued has finished before the accumulators' tensor
            // memory is released (at once after a normal run; bounded after an
            // expired wait)
            if (j) {
                mma_commit(saddr(&drain));
                wait_bounded(saddr(&drain), 0u);
            }
        }
    } else {
        // epilogue warps 2..9: tensor-memory lane quadrant warp % 4, column
        // half (warp - 2) / 4
        const uint32_t qd = warp & 3u, half = (warp - 2u) >> 2;
        uint32_t j = 0;
        for (uint32_t t = blockIdx.x; t < ntasks; t += gridDim.x, ++j) {
            const CUtensorMap* A;
            const CUtensorMap* B[3];
            const Args* a;
            uint32_t m0, n0;
            task(t, A, B, a, m0, n0);
            const uint32_t b = MT == 1 ? j & 1u : 0u, use = MT == 1 ? j >> 1 : j;
            // the first column block's fields and spins do not depend on the
            // accumulator: their loads go out before the wait for it
            RowBlock first;
            if (!ENERGY && !a->compute_only)
                load_row_block(first, *a, m0 + qd * 32u + lane, n0 + half * (BN / 2), m0 + qd * 32u + lane < a->chains);
            // every lane waits; the outcome is made warp-uniform
            const bool ok = __all_sync(0xffffffffu, !*vdead && wait_bounded(saddr(&tfull[b]), use & 1u));
            if (!ok && lane == 0) {
                atomicExch(a->err, kDevTimeout);
                *vdead = 1;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const bool live = __all_sync(0xffffffffu, !*vdead);
            if constexpr (ENERGY)
                energy_rows(tmem + ((qd * 32u) << 16) + 256u * b, *a, m0 + qd * 32u, n0, half * (BN / 2),
                            slice_of(t), ok && live);
            else if (!a->compute_only) {
                epilogue_rows(tmem + ((qd * 32u) << 16) + 256u * b, *a, m0 + qd * 32u, n0, half * (BN / 2),
                              ok && live, first);
                if constexpr (MT == 2) {
                    const uint32_t row0 = m0 + BM + qd * 32u;
                    load_row_block(first, *a, row0 + lane, n0 + half * (BN / 2), row0 + lane < a->chains);
                    epilogue_rows(tmem + ((qd * 32u) << 16) + 256u, *a, row0, n0, half * (BN / 2), ok && live, first);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(saddr(&tempty[b]));
            if (!ok) break;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            n = v;
        else
            n = 1;
    }
    return n;
}

// Spin operands of several runs (blockIdx.y = run): +-1 -> e4m3 / bf16.
struct SegSpins {
    const int8_t* s;
    void* o;
    size_t n;
};
__global__ void spins_to_op_batch(const SegSpins* __restrict__ seg, uint32_t bf16) {
    const SegSpins g = seg[blockIdx.y];
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < g.n;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const int v = g.s[i];
        if (bf16)
            static_cast<uint16_t*>(g.o)[i] = v == 0 ? 0 : (v > 0 ? 0x3F80 : 0xBF80);
        else
            static_cast<uint8_t*>(g.o)[i] = v == 0 ? 0 : (v > 0 ? 0x38 : 0xB8);
    }
}

// max over chains of |dE| = |-scale/2 sum s (h - H)| into stats[2]; clears dE.
__global__ void finish_energy(double* dE, uint32_t chains, double scale, unsigned long long* stats) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    double e = 0.0;
    if (c < chains) {
        e = fabs(0.5 * scale * dE[c]);
        dE[c] = 0.0;
    }
    // the warp's largest drift, then one atomic per warp (non-negative doubles
    // order as their bit patterns)
    unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(e));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, b, o);
        b = y > b ? y : b;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&stats[2], b);
}

// Operand conversion: spins +-1 (padding 0) -> e4m3 bytes or bf16 words,
// 16 spins per thread and iteration (n is a multiple of 32: rows of npad).
using dev::bf16_of2;
using dev::e4m3_of4;
__global__ void spins_to_e4m3(const int8_t* __restrict__ s, uint8_t* __restrict__ o, size_t n) {
    const uint4* in = reinterpret_cast<const uint4*>(s);
    uint4* out = reinterpret_cast<uint4*>(o);
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n / 16;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const uint4 w = in[i];
        out[i] = make_uint4(e4m3_of4(w.x), e4m3_of4(w.y), e4m3_of4(w.z), e4m3_of4(w.w));
    }
}
__global__ void spins_to_bf16(const int8_t* __restrict__ s, uint16_t* __restrict__ o, size_t n) {
    const uint4* in = reinterpret_cast<const uint4*>(s);
    uint4* out = reinterpret_cast<uint4*>(o);
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n / 16;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const uint4 w = in[i];
        out[2 * i] = make_uint4(bf16_of2(w.x, 0), bf16_of2(w.x, 2), bf16_of2(w.y, 0), bf16_of2(w.y, 2));
        out[2 * i + 1] = make_uint4(bf16_of2(w.z, 0), bf16_of2(w.z, 2), bf16_of2(w.w, 0), bf16_of2(w.w, 2));
    }
}
// J in {-1, 0, +1} -> e4m3 bytes.
__global__ void pm1_to_e4m3(const int8_t* __restrict__ j, uint8_t* __restrict__ o, size_t n) {
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const int v = j[i];
        o[i] = v == 0 ? 0 : (v > 0 ? 0x38 : 0xB8);
    }
}
// fp32 J -> J1 + J2 + J3, each rounded to nearest bf16 from the remainder of
// the previous terms; the remainders are exact in fp32.
__global__ void gauss_to_bf16x3(const float* __restrict__ j, uint16_t* __restrict__ o, size_t n) {
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        float r = j[i];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const __nv_bfloat16 b = __float2bfloat16_rn(r);
            o[t * n + i] = __bfloat16_as_ushort(b);
            r -= __bfloat162float(b);
        }
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

cudaError_t encoder(PFN_cuTensorMapEncodeTiled_v12000* fn) {
    std::call_once(g_encode_once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    *fn = g_encode;
    return g_encode ? cudaSuccess : cudaErrorNotSupported;
}

// 2-D K-major map: rows x cols elements (cols innermost), box = 128 bytes of
// K x box_rows rows, 128-byte swizzle, out-of-range elements read as zero.
cudaError_t make_map(CUtensorMap* m, const void* base, bool bf16, uint64_t rows, uint64_t cols,
                     uint32_t box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc;
    cudaError_t e = encoder(&enc);
    if (e != cudaSuccess) return e;
    const uint32_t esz = bf16 ? 2 : 1;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {cols * esz};
    const cuuint32_t box[2] = {128u / esz, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                           const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

uint32_t grid1d(size_t n) {
    const size_t b = (n + 255) / 256;
    return static_cast<uint32_t>(b < 4096 ? (b ? b : 1) : 4096);
}

}  // namespace

size_t recompute_j_bytes(uint32_t kind, uint32_t npad) {
    const size_t n = static_cast<size_t>(npad) * npad;
    return kind == 0 ? n : 3 * n * 2;
}
size_t recompute_s_bytes(uint32_t kind, uint32_t chains, uint32_t npad) {
    return static_cast<size_t>(chains) * npad * (kind == 0 ? 1 : 2);
}

cudaError_t recompute_prepare_j(const void* J, uint32_t kind, uint32_t npad, void* j_op, cudaStream_t st) {
    const size_t n = static_cast<size_t>(npad) * npad;
    if (kind == 0)
        pm1_to_e4m3<<<grid1d(n), 256, 0, st>>>(static_cast<const int8_t*>(J), static_cast<uint8_t*>(j_op), n);
    else
        gauss_to_bf16x3<<<grid1d(n), 256, 0, st>>>(static_cast<const float*>(J), static_cast<uint16_t*>(j_op), n);
    return cudaGetLastError();
}

namespace {
// Whether 256-row tiles (bf16) finish first: rounds of the persistent CTAs times
// the main loop (us a 128-byte K block: 0.47 on 128-row tiles, 0.57 on 256-row
// ones) and the epilogue of a row block (8.5 us where it reads the old fields
// and spins, 6 where it only writes), which overlaps the main loop on 128-row
// tiles only.  Resync of three terms, 128 / 256 rows: N = 2048 x 8192 chains
// 191 / 135 us, 1024 x 16384 123 / 82, 2048 x 4096 101 / 68; the check of
// 512 x 65536, 108 / 129, keeps the 128.  FP8 tiles stay at 128: 2048 x 8192
// took 50 / 60 us, the best other size 42 / 40.
bool tall_tiles(uint64_t tiles128, uint64_t tiles256, uint32_t kblocks, bool reads) {
    const uint64_t sms = static_cast<uint64_t>(sm_count());
    const double e = reads ? 8.5 : 6.0;
    const double t1 = static_cast<double>((tiles128 + sms - 1) / sms) * std::max(0.47 * kblocks, e);
    const double t2 = static_cast<double>((tiles256 + sms - 1) / sms) * (0.57 * kblocks + 2.0 * e);
    return t2 < t1;
}

// The dynamic shared-memory attribute of a recompute kernel variant, set once
// per device and variant.
template <typename F>
cudaError_t smem_attribute(F kernel, int variant) {
    static std::mutex mu;
    static std::set<std::pair<int, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count({dev, variant})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) done.insert({dev, variant});
    return e;
}

// The coupling operands of several instances of one kind in one launch
// (blockIdx.y = instance): the conversions of pm1_to_e4m3 / gauss_to_bf16x3.
__global__ void prepare_j_batch(const PrepareJ* __restrict__ jobs, uint32_t pm1) {
    const PrepareJ p = jobs[blockIdx.y];
    const size_t n = static_cast<size_t>(p.npad) * p.npad;
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        if (pm1) {
            const int v = static_cast<const int8_t*>(p.J)[i];
            static_cast<uint8_t*>(p.j_op)[i] = v == 0 ? 0 : (v > 0 ? 0x38 : 0xB8);
        } else {
            float r = static_cast<const float*>(p.J)[i];
            uint16_t* o = static_cast<uint16_t*>(p.j_op);
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const __nv_bfloat16 b = __float2bfloat16_rn(r);
                o[t * n + i] = __bfloat16_as_ushort(b);
                r -= __bfloat162float(b);
            }
        }
    }
}
}  // namespace

cudaError_t recompute_prepare_j_batch(uint32_t kind, const PrepareJ* jobs, uint32_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    size_t maxn = 0;
    for (uint32_t i = 0; i < n; ++i) maxn = std::max(maxn, static_cast<size_t>(jobs[i].npad) * jobs[i].npad);
    PrepareJ* d = nullptr;
    cudaError_t e = cudaMallocAsync(&d, n * sizeof(PrepareJ), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d, jobs, n * sizeof(PrepareJ), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        prepare_j_batch<<<dim3(std::min<uint32_t>(grid1d(maxn), 512u), n), 256, 0, st>>>(d, kind == 0 ? 1u : 0u);
        e = cudaGetLastError();
    }
    if (d) cudaFreeAsync(d, st);
    return e;
}

cudaError_t launch_set_fields_batch(uint32_t kind, const RecomputeSet* sets, uint32_t n, cudaStream_t st,
                                   bool spins_converted) {
    if (n == 0) return cudaSuccess;
    const bool bf = kind != 0;
    std::vector<SegSpins> seg(n);
    std::vector<BatchJob> jobs(n);
    std::vector<BatchTask> tasks;
    size_t maxn = 0;
    uint64_t nt1 = 0, nt2 = 0, kb = 0;  // tiles of either height, K blocks of all sets
    for (uint32_t i = 0; i < n; ++i) {
        const RecomputeSet& q = sets[i];
        seg[i] = SegSpins{q.s, q.s_op, static_cast<size_t>(q.chains) * q.npad};
        maxn = std::max(maxn, seg[i].n);
        BatchJob& b = jobs[i];
        std::memset(&b, 0, sizeof b);
        cudaError_t e = make_map(&b.A, q.s_op, bf, q.chains, q.npad, BM);
        const size_t term_bytes = static_cast<size_t>(q.npad) * q.npad * (bf ? 2 : 1);
        for (uint32_t t = 0; t < 3 && e == cudaSuccess; ++t)
            e = make_map(&b.B[t], static_cast<const unsigned char*>(q.j_op) + (bf ? t : 0) * term_bytes, bf, q.npad,
                         q.npad, BN);
        if (e != cudaSuccess) return e;
        b.args.h = q.h;
        b.args.s = q.s;
        b.args.err = q.err;
        b.args.chains = q.chains;
        b.args.npad = q.npad;
        b.args.kblocks = (q.npad + (bf ? 63u : 127u)) / (bf ? 64u : 128u);
        b.args.terms = bf ? 3u : 1u;
        b.args.mode = 3;
        b.args.pm1 = bf ? 0u : 1u;
        b.args.fault = 0u;
        const uint64_t tn = (q.npad + BN - 1) / BN;
        nt1 += (q.chains + BM - 1) / BM * tn;
        nt2 += (q.chains + 2 * BM - 1) / (2 * BM) * tn;
        kb += b.args.terms * b.args.kblocks;
    }
    const bool tall = bf && tall_tiles(nt1, nt2, static_cast<uint32_t>(kb / n), false);
    // longest tiles first: CTA c takes tasks c, c + grid, ..., and the sets may
    // differ in N (mixed order would leave the last round to the long ones)
    std::vector<uint32_t> order(n);
    std::iota(order.begin(), order.end(), 0u);
    std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) { return sets[x].npad > sets[y].npad; });
    for (uint32_t i : order)
        for (uint32_t m0 = 0; m0 < sets[i].chains; m0 += tall ? 2 * BM : BM)
            for (uint32_t n0 = 0; n0 < sets[i].npad; n0 += BN) tasks.push_back(BatchTask{i, m0, n0, 0});
    SegSpins* dseg = nullptr;
    BatchJob* djobs = nullptr;
    BatchTask* dtasks = nullptr;
    cudaError_t e = cudaMallocAsync(&dseg, n * sizeof(SegSpins), st);
    if (e == cudaSuccess) e = cudaMallocAsync(&djobs, n * sizeof(BatchJob), st);
    if (e == cudaSuccess) e = cudaMallocAsync(&dtasks, tasks.size() * sizeof(BatchTask), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dseg, seg.data(), n * sizeof(SegSpins), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(djobs, jobs.data(), n * sizeof(BatchJob), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dtasks, tasks.data(), tasks.size() * sizeof(BatchTask), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !spins_converted) {
        const dim3 g(std::min<uint32_t>(grid1d(maxn), 1024u), n);
        spins_to_op_batch<<<g, 256, 0, st>>>(dseg, bf ? 1u : 0u);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        CUtensorMap none;
        std::memset(&none, 0, sizeof none);
        Args a0;
        std::memset(&a0, 0, sizeof a0);
        const uint32_t nt = static_cast<uint32_t>(tasks.size());
        const uint32_t grid = std::max<uint32_t>(1u, std::min<uint32_t>(nt, static_cast<uint32_t>(sm_count())));
        auto go = [&](auto kernel, int variant) {
            e = smem_attribute(kernel, variant);
            if (e == cudaSuccess)
                kernel<<<grid, WS_THREADS, SMEM_BYTES, st>>>(none, none, none, none, a0, djobs, dtasks, nt, 0u);
        };
        if (tall) go(recompute_ws_kernel<false, 1, 2>, 5);
        else if (bf) go(recompute_ws_kernel<false, 1>, 6);
        else go(recompute_ws_kernel<true, 1>, 7);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    cudaFreeAsync(dseg, st);
    cudaFreeAsync(djobs, st);
    cudaFreeAsync(dtasks, st);
    return e;
}

namespace {
// Operand tensor maps by (spin operand, coupling operand, type, shape): a map
// holds only addresses and shapes, so one encoded for the same buffers and
// shape is valid again; a few recent entries are kept.
cudaError_t cached_maps(const void* s_op, const void* j_op, bool bf, uint32_t chains, uint32_t npad, CUtensorMap* tA,
                        CUtensorMap* tB) {
    struct Entry {
        const void *s_op, *j_op;
        bool bf;
        uint32_t chains, npad;
        CUtensorMap A, B[3];
    };
    static std::mutex mu;
    static std::vector<Entry> cache;
    std::lock_guard<std::mutex> lk(mu);
    for (const Entry& c : cache)
        if (c.s_op == s_op && c.j_op == j_op && c.bf == bf && c.chains == chains && c.npad == npad) {
            *tA = c.A;
            for (int t = 0; t < 3; ++t) tB[t] = c.B[t];
            return cudaSuccess;
        }
    Entry c{s_op, j_op, bf, chains, npad, {}, {}};
    cudaError_t e = make_map(&c.A, s_op, bf, chains, npad, BM);
    const size_t term_bytes = static_cast<size_t>(npad) * npad * (bf ? 2 : 1);
    for (uint32_t t = 0; t < 3 && e == cudaSuccess; ++t)
        e = make_map(&c.B[t], static_cast<const unsigned char*>(j_op) + (bf ? t : 0) * term_bytes, bf, npad, npad, BN);
    if (e != cudaSuccess) return e;
    if (cache.size() >= 32) cache.erase(cache.begin());
    cache.push_back(c);
    *tA = c.A;
    for (int t = 0; t < 3; ++t) tB[t] = c.B[t];
    return cudaSuccess;
}
}  // namespace

cudaError_t launch_recompute(uint32_t kind, const int8_t* s, void* h, float* out, void* s_op,
                             const void* j_op, double* dE, unsigned long long* stats, int* err,
                             uint32_t chains, uint32_t npad, uint32_t terms, uint32_t mode, double scale,
                             cudaStream_t st, uint32_t fault, bool spins_converted, unsigned int* cnt) {
    const bool bf = kind != 0;
    if (!bf) terms = 1;
    if (terms < 1 || terms > 3) return cudaErrorInvalidValue;
    const size_t ns = static_cast<size_t>(chains) * npad;  // a multiple of 32
    cudaError_t e = cudaSuccess;
    if (!spins_converted) {
        if (bf)
            spins_to_bf16<<<grid1d(ns / 16), 256, 0, st>>>(s, static_cast<uint16_t*>(s_op), ns);
        else
            spins_to_e4m3<<<grid1d(ns / 16), 256, 0, st>>>(s, static_cast<uint8_t*>(s_op), ns);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // the operand maps of this (spins, couplings, shape): encoded once and
    // reused by later recomputes of the same buffers, so that the host work
    // between the conversion and the main kernel stays short
    CUtensorMap tA, tB[3];
    if ((e = cached_maps(s_op, j_op, bf, chains, npad, &tA, tB)) != cudaSuccess) return e;
    Args a{};
    a.h = h;
    a.s = s;
    a.out = out;
    a.dE = dE;
    a.stats = stats;
    a.cnt = mode < 2 ? cnt : nullptr;
    a.scale = scale;
    a.err = err;
    a.chains = chains;
    a.npad = npad;
    a.kblocks = (npad + (bf ? 63u : 127u)) / (bf ? 64u : 128u);
    a.terms = terms;
    a.mode = mode;
    a.pm1 = bf ? 0u : 1u;
    a.fault = fault;
    a.compute_only = 0;
    const uint32_t tiles_n = (npad + BN - 1) / BN;
    const uint32_t nt1 = ((chains + BM - 1) / BM) * tiles_n, nt2 = ((chains + 2 * BM - 1) / (2 * BM)) * tiles_n;
    if (nt1 == 0) return cudaSuccess;
    const bool tall = bf && tall_tiles(nt1, nt2, terms * a.kblocks, mode < 2);
    const uint32_t nt = tall ? nt2 : nt1;
    const uint32_t grid = std::min<uint32_t>(nt, static_cast<uint32_t>(sm_count()));
    if (tall) {
        if ((e = smem_attribute(recompute_ws_kernel<false, 0, 2>, 4)) != cudaSuccess) return e;
        recompute_ws_kernel<false, 0, 2><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB[0], tB[1], tB[2], a, nullptr,
                                                                              nullptr, nt, tiles_n);
    } else if (bf) {
        if ((e = smem_attribute(recompute_ws_kernel<false, 0>, 0)) != cudaSuccess) return e;
        recompute_ws_kernel<false, 0><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB[0], tB[1], tB[2], a, nullptr,
                                                                               nullptr, nt, tiles_n);
    } else {
        if ((e = smem_attribute(recompute_ws_kernel<true, 0>, 1)) != cudaSuccess) return e;
        recompute_ws_kernel<true, 0><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB[0], tB[0], tB[0], a, nullptr,
                                                                              nullptr, nt, tiles_n);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess || mode >= 2 || a.cnt) return e;
    finish_energy<<<(chains + 255) / 256, 256, 0, st>>>(dE, chains, scale, stats);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Energies of many configurations (sk_energy) as products on the tensor cores
// ---------------------------------------------------------------------------
// E(c) = -scale sum_n s_n H_n, H_n = sum_{k > n} J_nk s_k: a product with the
// strict upper triangle of J, taken exactly.  +-J: one FP8 slice.  Gaussian:
// every J_ij is an integer q_ij times 2^lsb, lsb the lowest bit set in any of
// them; q is written as signed base-256 digits, each exact in bf16, and a
// digit's sums stay below 2^20 (128 x 8192), exact in the FP32 accumulator.
// The digits' energy sums are integers (int32 per tile row, int64 per
// configuration) joined in 128 bits, so the sum is rounded once (twice from
// 2^64 units of the lowest bit on) and once more by the scale, where the
// double-precision sum it replaces (energy_kernel) rounds at every term: rms
// relative error against 113-bit sums 7.5e-17 and 5.2e-17 (N = 1024, 2048), that
// sum's 8.0e-17 and 1.0e-16.  Couplings
// that span more than kEnergyBits bits take energy_kernel.  Bound: FP64 adds
// run at 2 per clock and SM on this part; the 7 slices a Gaussian matrix of
// N = 2048 needs are 3e10 bf16 multiply-adds for 2048 configurations (half
// the matrix): 12.35 ms a call -> 0.14 ms, of which the fixed cost is 0.07.
namespace {
constexpr uint32_t kEnergyBits = 62;  // q fits a signed 64-bit integer and 8 digits
constexpr uint32_t kEnergySlices = 8;

// Header of the workspace: [0] slices (0: take energy_kernel), [1] lowest bit
// set in any coupling, [2] highest (biased by 256, running min / max), [3] error word.
struct EnergyHead {
    uint32_t slices;
    uint32_t lsb, msb;
    int err;
};

// The position of the lowest and highest set bits of |x|, biased by 256.
__device__ __forceinline__ void bits_of(float x, uint32_t& lo, uint32_t& hi) {
    const uint32_t b = __float_as_uint(x) & 0x7FFFFFFFu;
    if (b == 0u) return;
    const uint32_t e = b >> 23;
    const uint32_t m = (b & 0x7FFFFFu) | (e ? 0x800000u : 0u);
    const uint32_t base = (e ? e : 1u) + 256u - 150u;
    lo = min(lo, base + static_cast<uint32_t>(__ffs(static_cast<int>(m)) - 1));
    hi = max(hi, base + 31u - static_cast<uint32_t>(__clz(static_cast<int>(m))));
}
__global__ void energy_range(const float* __restrict__ J, uint64_t words4, EnergyHead* __restrict__ head) {
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    for (uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; i < words4;
         i += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(J) + i);
        bits_of(v.x, lo, hi);
        bits_of(v.y, lo, hi);
        bits_of(v.z, lo, hi);
        bits_of(v.w, lo, hi);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&head->lsb, lo);
        atomicMax(&head->msb, hi);
    }
}

// Slices of rows row0 .. row0 + gridDim.x - 1 of the strict upper triangle,
// slice t of row row0 + r at row t gridDim.x + r: the columns from the start
// of the row's own tile on (the rest is not read).  A thread writes 8 columns
// (16 bytes) of every slice.
__global__ void energy_slices(const float* __restrict__ J, uint16_t* __restrict__ out, uint32_t npad, uint32_t row0,
                              EnergyHead* __restrict__ head) {
    const uint32_t lsb = head->lsb, msb = head->msb;
    const uint32_t bits = msb >= lsb ? msb - lsb + 1u : 0u;  // none set: all couplings zero
    const uint32_t S = bits > kEnergyBits ? 0u : (bits + 2u + 7u) / 8u;
    if (blockIdx.x == 0 && threadIdx.x == 0) head->slices = S;
    const uint32_t n = row0 + blockIdx.x;
    for (uint32_t k = (n & ~(BN - 1u)) + 8u * threadIdx.x; S && k < npad; k += 8u * blockDim.x) {
        float x[8];
        *reinterpret_cast<float4*>(&x[0]) = __ldg(reinterpret_cast<const float4*>(J + static_cast<size_t>(n) * npad + k));
        *reinterpret_cast<float4*>(&x[4]) = __ldg(reinterpret_cast<const float4*>(J + static_cast<size_t>(n) * npad + k + 4));
        long long q[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t b = __float_as_uint(x[e]), f = (b >> 23) & 255u;
            const long long m = (b & 0x7FFFFFu) | (f ? 0x800000u : 0u);
            const int sh = static_cast<int>((f ? f : 1u) + 256u - 150u) - static_cast<int>(lsb);
            const long long a = m == 0 ? 0ll : sh >= 0 ? m << sh : m >> -sh;  // (the bits shifted out are zero)
            q[e] = k + e > n ? ((b >> 31) ? -a : a) : 0ll;
        }
        for (uint32_t t = 0; t < S; ++t) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t p = 0;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int d = static_cast<int>(static_cast<int8_t>(q[2 * e + h] & 0xFF));
                    q[2 * e + h] = (q[2 * e + h] - d) >> 8;
                    p |= (__float_as_uint(static_cast<float>(d)) >> 16) << (16 * h);  // |d| <= 128: exact in bf16
                }
                w[e] = p;
            }
            *reinterpret_cast<uint4*>(out + (static_cast<size_t>(t) * gridDim.x + blockIdx.x) * npad + k) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}
// The same for +-J: one slice of e4m3 bytes, 16 columns per thread.
__global__ void energy_slice_pm1(const int8_t* __restrict__ J, uint8_t* __restrict__ out, uint32_t npad,
                                 uint32_t row0, EnergyHead* __restrict__ head) {
    if (blockIdx.x == 0 && threadIdx.x == 0) head->slices = 1u;
    const uint32_t n = row0 + blockIdx.x;
    for (uint32_t k = (n & ~(BN - 1u)) + 16u * threadIdx.x; k < npad; k += 16u * blockDim.x) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(J + static_cast<size_t>(n) * npad + k));
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (uint32_t e = 0; e < 4; ++e) {
            const uint32_t k0 = k + 4u * e;  // bytes of columns k > n only
            const uint32_t keep = n < k0 ? 0xFFFFFFFFu : n >= k0 + 3u ? 0u : 0xFFFFFFFFu << (8u * (n + 1u - k0));
            w[e] = e4m3_of4(w[e] & keep);
        }
        *reinterpret_cast<uint4*>(out + static_cast<size_t>(blockIdx.x) * npad + k) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
// Configurations (rows x N, any alignment) as padded int8 rows and as the MMA
// operand; a value below 0 counts as -1, any other as +1, padding 0.
__global__ void energy_spins(const int8_t* __restrict__ spins, uint32_t N, uint32_t npad, uint32_t rows, uint32_t bf,
                             int8_t* __restrict__ s, void* __restrict__ op) {
    const uint32_t words = npad / 16u;
    for (uint32_t c = blockIdx.x; c < rows; c += gridDim.x)
        for (uint32_t wd = threadIdx.x; wd < words; wd += blockDim.x) {
            const int8_t* src = spins + static_cast<size_t>(c) * N + 16u * wd;
            uint32_t w[4];
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e) {
                w[e] = 0u;
#pragma unroll
                for (uint32_t h = 0; h < 4; ++h)
                    if (16u * wd + 4u * e + h < N) w[e] |= (__ldg(src + 4u * e + h) < 0 ? 0xFFu : 0x01u) << (8u * h);
            }
            const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
            const size_t at = static_cast<size_t>(c) * words + wd;
            reinterpret_cast<uint4*>(s)[at] = v;
            dev::spins_to_op16(op, at, v, bf != 0u);
        }
}
// The slices' sums joined: E = -scale 2^lsb sum_t 256^t esum_t, in 128 bits.
__global__ void energy_join(const unsigned long long* __restrict__ esum, const EnergyHead* __restrict__ head,
                            uint32_t rows, double scale, uint32_t pm1, double* __restrict__ out) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t S = head->slices;
    if (c >= rows || S == 0u) return;
    unsigned long long lo = 0, hi = 0;  // two's complement
    for (uint32_t t = S; t-- > 0u;) {
        hi = (hi << 8) | (lo >> 56);
        lo <<= 8;
        const unsigned long long v = esum[static_cast<size_t>(t) * rows + c];
        lo += v;
        hi += (lo < v ? 1ull : 0ull) + static_cast<unsigned long long>(static_cast<long long>(v) >> 63);
    }
    const bool neg = static_cast<long long>(hi) < 0;
    if (neg) {
        lo = ~lo + 1ull;
        hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    double v = fma(static_cast<double>(hi), 0x1p64, static_cast<double>(lo));
    if (neg) v = -v;
    if (!pm1) v = ldexp(v, S > 0u && head->msb >= head->lsb ? static_cast<int>(head->lsb) - 256 : 0);
    out[c] = -scale * v;
}

// Configurations and rows of J a launch takes: operands of at most 96 MB each,
// whole tiles of 128 and 256.
uint32_t energy_chunk(uint32_t npad, uint32_t count) {
    return std::min(count, std::max<uint32_t>(128u, ((96u << 20) / (3u * npad)) & ~127u));
}
uint32_t energy_rows_of(uint32_t kind, uint32_t npad) {
    const uint32_t row = npad * (kind == 0 ? 1u : 2u * kEnergySlices);
    return std::min(npad, std::max<uint32_t>(256u, ((96u << 20) / row) & ~255u));
}
size_t energy_up(size_t b) { return (b + 1023u) & ~static_cast<size_t>(1023u); }
}  // namespace

// Where the tensor path is the faster one (us a call, direct sum / tensor, on
// one configuration and on 4096): Gaussian N = 32 61 / 73 and 74 / 79, N = 64
// 83 / 71 and 97 / 82, N = 512 440 / 73 and 1668 / 90; +-J N = 256 61 / 67 and
// 74 / 74, N = 512 94 / 66 and 145 / 72, N = 2048 247 / 70 and 1761 / 84.  The
// tensor path has a few more launches (the fixed ~65 us), the direct sum costs
// at least a column's length of dependent adds.
bool energy_on_tensor(uint32_t kind, uint32_t N, uint32_t count) {
    const uint64_t terms = static_cast<uint64_t>(N) * N * count;
    return kind == 0 ? N >= 320u || terms >= (1ull << 29) : N >= 48u || terms >= (1ull << 24);
}

size_t energy_workspace(uint32_t kind, uint32_t npad, uint32_t count) {
    const size_t C = energy_chunk(npad, count), R = energy_rows_of(kind, npad);
    const size_t S = kind == 0 ? 1 : kEnergySlices;
    return 1024 + energy_up(R * npad * (kind == 0 ? 1 : 2 * S)) + energy_up(C * npad) +
           energy_up(C * npad * (kind == 0 ? 1 : 2)) + energy_up(count * S * 8);
}

// Energies of `count` configurations into out[count] in `ws`
// (energy_workspace bytes, 1 KB aligned).  *slices_word: where the kernels
// leave the slice count, 0 when the couplings span too many bits and the
// caller's energy_kernel launch is the one that writes out.
cudaError_t launch_energy_tensor(const void* J, uint32_t kind, uint32_t N, uint32_t npad, double scale,
                                 const int8_t* spins, uint32_t count, double* out, void* ws, const uint32_t** slices_word,
                                 const int** err_word, cudaStream_t st) {
    const bool bf = kind != 0;
    const uint32_t C = energy_chunk(npad, count), R = energy_rows_of(kind, npad), S = bf ? kEnergySlices : 1u;
    unsigned char* p = static_cast<unsigned char*>(ws);
    EnergyHead* head = reinterpret_cast<EnergyHead*>(p);
    p += 1024;
    void* jop = p;
    p += energy_up(static_cast<size_t>(R) * npad * (bf ? 2 * S : 1));
    int8_t* s = reinterpret_cast<int8_t*>(p);
    p += energy_up(static_cast<size_t>(C) * npad);
    void* sop = p;
    p += energy_up(static_cast<size_t>(C) * npad * (bf ? 2 : 1));
    unsigned long long* esum = reinterpret_cast<unsigned long long*>(p);
    *slices_word = &head->slices;
    *err_word = &head->err;
    cudaError_t e = cudaMemsetAsync(head, 0, sizeof(EnergyHead), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(&head->lsb, 0xFF, sizeof(uint32_t), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(esum, 0, static_cast<size_t>(count) * S * 8, st);
    if (e == cudaSuccess)
        e = bf ? smem_attribute(recompute_ws_kernel<false, 2>, 2) : smem_attribute(recompute_ws_kernel<true, 2>, 3);
    if (e != cudaSuccess) return e;
    if (bf) {
        const uint64_t w4 = static_cast<uint64_t>(npad) * npad / 4u;
        energy_range<<<static_cast<uint32_t>(std::min<uint64_t>((w4 + 1023u) / 1024u, 608u)), 256, 0, st>>>(
            static_cast<const float*>(J), w4, head);
    }
    for (uint32_t r0 = 0; r0 < npad; r0 += R) {
        const uint32_t rows_j = std::min(R, npad - r0);
        const uint32_t threads = std::min<uint32_t>(256u, std::max<uint32_t>(32u, (npad / (bf ? 8u : 16u) + 31u) & ~31u));
        if (bf)
            energy_slices<<<rows_j, threads, 0, st>>>(static_cast<const float*>(J), static_cast<uint16_t*>(jop), npad, r0, head);
        else
            energy_slice_pm1<<<rows_j, threads, 0, st>>>(static_cast<const int8_t*>(J), static_cast<uint8_t*>(jop), npad, r0,
                                                        head);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        CUtensorMap tB;
        if ((e = make_map(&tB, jop, bf, static_cast<uint64_t>(S) * rows_j, npad, BN)) != cudaSuccess) return e;
        for (uint32_t c0 = 0; c0 < count; c0 += C) {
            const uint32_t rows = std::min(C, count - c0);
            if (r0 == 0 || C < count) {  // (one block of configurations keeps its operand)
                const uint32_t sth = std::min<uint32_t>(128u, std::max<uint32_t>(32u, (npad / 16u + 31u) & ~31u));
                energy_spins<<<std::min<uint32_t>(rows, 2432u), sth, 0, st>>>(spins + static_cast<size_t>(c0) * N, N, npad,
                                                                             rows, bf ? 1u : 0u, s, sop);
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
            }
            CUtensorMap tA;
            if ((e = make_map(&tA, sop, bf, rows, npad, BM)) != cudaSuccess) return e;
            Args a{};
            a.s = s;
            a.err = &head->err;
            a.chains = rows;
            a.npad = npad;
            a.kblocks = (npad + (bf ? 63u : 127u)) / (bf ? 64u : 128u);
            a.terms = 1;
            a.pm1 = bf ? 0u : 1u;
            a.nslices = &head->slices;
            a.esum = esum + c0;
            a.esum_stride = count;
            a.b_row0 = r0;
            a.b_rows = rows_j;
            const uint32_t tiles_n = (rows_j + BN - 1) / BN;
            const uint32_t grid = std::min<uint32_t>(S * tiles_n * ((rows + BM - 1) / BM), static_cast<uint32_t>(sm_count()));
            if (bf)
                recompute_ws_kernel<false, 2><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB, tB, tB, a, nullptr, nullptr,
                                                                                   0u, tiles_n);
            else
                recompute_ws_kernel<true, 2><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB, tB, tB, a, nullptr, nullptr,
                                                                                  0u, tiles_n);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    energy_join<<<(count + 255u) / 256u, 256, 0, st>>>(esum, head, count, scale, bf ? 0u : 1u, out);
    return cudaGetLastError();
}

cudaError_t tensor_peak_probe(uint32_t kind, uint32_t tiles, uint32_t reps, cudaStream_t st, double* tflops) {
    const bool bf = kind != 0;
    const uint32_t kblocks = 16;  // K = 2048 (FP8) or 1024 (bf16): 16 stages of 128 bytes per row
    const uint32_t K = kblocks * (bf ? 64u : 128u);
    const uint32_t grid = static_cast<uint32_t>(sm_count());
    const uint32_t nt = grid * tiles;
    const size_t esz = bf ? 2 : 1;
    void* A = nullptr;
    void* B = nullptr;
    int* err = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float ms = 0.0f;
    // operands of each CTA's first tile (all zero: the values do not matter)
    cudaError_t e = cudaMalloc(&A, static_cast<size_t>(grid) * BM * K * esz);
    if (e == cudaSuccess) e = cudaMalloc(&B, static_cast<size_t>(BN) * K * esz);
    if (e == cudaSuccess) e = cudaMalloc(&err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(A, 0, static_cast<size_t>(grid) * BM * K * esz, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(B, 0, static_cast<size_t>(BN) * K * esz, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), st);
    CUtensorMap tA, tB;
    if (e == cudaSuccess) e = make_map(&tA, A, bf, static_cast<uint64_t>(grid) * BM, K, BM);
    if (e == cudaSuccess) e = make_map(&tB, B, bf, BN, K, BN);
    Args a{};
    a.err = err;
    a.chains = grid * BM;
    a.npad = K;
    a.kblocks = kblocks;
    a.terms = 1;
    a.mode = 2;
    a.pm1 = bf ? 0u : 1u;
    a.compute_only = 1;
    auto launch = [&]() {
        // task t: rows (t / 1) * BM, columns 0; each CTA's first task is its own block of A
        if (bf)
            recompute_ws_kernel<false, 0><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB, tB, tB, a, nullptr,
                                                                                   nullptr, nt, 1u);
        else
            recompute_ws_kernel<true, 0><<<grid, WS_THREADS, SMEM_BYTES, st>>>(tA, tB, tB, tB, a, nullptr,
                                                                                  nullptr, nt, 1u);
        return cudaGetLastError();
    };
    if (e == cudaSuccess)
        e = bf ? smem_attribute(recompute_ws_kernel<false, 0>, 0) : smem_attribute(recompute_ws_kernel<true, 0>, 1);
    if (e == cudaSuccess) e = launch();  // warm-up
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaEventRecord(e0, st);
    for (uint32_t r = 0; r < reps && e == cudaSuccess; ++r) e = launch();
    if (e == cudaSuccess) e = cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&herr, err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && herr) e = cudaErrorLaunchTimeout;  // a bounded wait expired
    if (e == cudaSuccess)
        *tflops = 2.0 * BM * BN * static_cast<double>(K) * nt * reps / (ms * 1e-3) / 1e12;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(A);
    cudaFree(B);
    cudaFree(err);
    return e;
}

}  // namespace sk
