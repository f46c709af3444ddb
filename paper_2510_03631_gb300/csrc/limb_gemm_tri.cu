// Exact mod-2^32 product of a digit matrix with Z_q vectors in three fp16 limbs, on CTA pairs:
//     OUT[i][b] = sum_j D[i][j] * X[b][j]   (mod 2^32),  D[i][j] in [0, 255].
//
// Why three limbs.  The product is bound by the tensor cores, and the limbs of the vectors set how
// often every digit is multiplied.  fp16 holds every integer up to 2048, so a limb may have 11 bits
// (balanced: -1024 .. 1023) instead of 8, and 32 bits take three limbs (11 + 11 + 10) instead of
// four: a quarter less tensor work and operand traffic.  The price is a shorter exact sum: digits centred to
// d - p / 2 (-128 .. 127) times limbs are at most 2^17 in magnitude, so fp32 sums are exact for 128 columns (2^24;
// every integer of at most that magnitude is an fp32 value), and the accumulators are drained to
// int32 every 128 columns.  Centring takes p / 2 times sum_j X[b][j] from every output of vector b; the sums
// come with the limbs.
//
// Tile.  256 rows x 64 H vectors over a pair of SMs (tcgen05 cta_group::2).  A half is 64 vectors
// = 192 limb columns; the two accumulators of 192 TMEM columns take turns: with H = 2 half 0 and
// half 1 of a chunk of 128 columns of D, so every digit tile staged in shared memory is multiplied by
// 384 limb rows (40 KB received per SM for 768 tensor cycles per 64 columns; a four-limb 256-wide tile
// receives 32 KB for 512).
//
// What bounds it.  The drains: a half's MMAs run for 768 cycles, and 192 columns are converted and added
// in that time by eight warps, whose instructions also delay the one that issues the MMAs.  F2I runs at
// 1/8 of the FP32 rate, so only the lowest limb goes through it; the other two are cut
// to the bits that count and summed in exact packed FP32 steps (high_limbs).  32768 x 32768, 256 vectors, back
// to back: four limbs 1308 us, this kernel 1190; single calls 1132 and 1024, of which 860 are left when the
// drains do nothing (a timing copy) and 95 go when their conversions are left out.  Hint of 1024
// columns 5390 -> 4550 us.  All three limbs through F2I 1670 us; sixteen epilogue warps 1160;
// a whole half's columns in registers first (setmaxnreg 208) 1090; one issue block per 64 columns
// instead of per half 1140 (single calls).
//
// Column order.  One TMA box holds 32 vectors x 3 limbs (limb-major); the MMA's columns are the leader's
// box, then the peer's: columns 96 g + 32 k + q are limb k of vector 32 g + q of the half.  Epilogue
// warpgroup g of each CTA drains the 96 columns of box g, 16 vectors at a time, and keeps 32
// running sums per half and thread: run += s_0 + (s_1 << 11) + (s_2 << 22) mod 2^32.
//
// Roles, barriers and failure handling follow limb_gemm_pair.cu: warp 0 loads the matrix tiles and arms
// each stage, warp 2 the vector boxes, warp 1 of the leader issues the MMAs, warps 4..11 drain.
//
// Schedule.  Tiles are dealt round-robin, the vector tiles of one row tile to neighbouring clusters.
// Where whole tiles leave the last wave too empty, or clusters idle, every tile is cut into the same column ranges,
// dealt range by range, whose parts add into a zeroed output (exact: addition mod 2^32 commutes).
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "limb_gemm_tri.cuh"
#include "ptx.cuh"

namespace qpadl {

namespace {

constexpr int kTM = 128;           // matrix rows per CTA (256 per pair)
constexpr int kTK = 64;            // fp16 elements per 128-byte swizzled row
constexpr int kTN = 192;           // limb columns per accumulator
constexpr int kChunkSteps = 2;     // k-steps per exact chunk: 128 columns of D
constexpr int kTThreads = 384;     // warps: 0 matrix producer, 1 MMA, 2 vector producer, 4..11 epilogue

// How the output is stored: a word per lane and vector (the lanes' rows are neighbours in column-major answers), or, for
// the hint's rows, 16 bytes a lane where they allow it (30000 x 600 digits by 512 columns: 214 us with word stores,
// 84), else 32 rows x 32 vectors turned, so that a warp writes a row's 128 bytes at a time (4864 x 1088 by 630 columns: word
// stores 46.9 us, turned 35.9; 7104 x 2471 by 1024 in all: 16-byte stores 91.5, turned 99.3).
// out[row + v * ld], or the others' out[row * ld + v].
enum { kWords, kQuads, kTurned };

template <int H>
struct TriCfg {
    static constexpr uint32_t kABytes = kTM * kTK * 2;              // 16 KB
    static constexpr uint32_t kBoxBytes = 3 * kTriGroup * kTK * 2;  // 12 KB: this CTA's vectors of one half
    static constexpr uint32_t kStageBytes = kABytes + H * kBoxBytes;
    static constexpr int kFit = (227 * 1024 - 2048) / kStageBytes;
    static constexpr int kStages = kFit < 8 ? kFit : 8;             // 8, 5 and 4 at H = 1, 2 and 3
    static constexpr int kSmemBytes = kStages * kStageBytes + 256 + 1024;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
    static_assert(kStages >= 4, "a chunk's two stages and two in flight");
};

// A cluster's pieces: unit i is column range i / tiles of tile i % tiles, chunks [c0, c1).  The vector
// tiles of a row tile are neighbours; which of them comes first turns from wave to wave, so a narrower
// last one (fewer halves) does not always fall to the same clusters.
struct TriPiece {
    uint32_t m, n, halves, c0, c1;   // row tile, vector tile, its halves with vectors
};
struct TriIter {
    uint32_t u, step, n_tiles, tiles, nchunks, ksplit, NV, H;
    __device__ __forceinline__ bool next(TriPiece &pc) {
        const uint32_t s = u / tiles;
        if (s >= ksplit) return false;
        const uint32_t t = u % tiles;
        pc.m = t / n_tiles;
        pc.n = (t % n_tiles + pc.m * n_tiles / step) % n_tiles;
        const uint32_t left = (NV - pc.n * 64u * H + 63u) / 64u;
        pc.halves = left < H ? left : H;
        pc.c0 = static_cast<uint32_t>((uint64_t)s * nchunks / ksplit);
        pc.c1 = static_cast<uint32_t>((uint64_t)(s + 1) * nchunks / ksplit);
        u += step;
        return true;
    }
};

// Two fp32 values per 64-bit register pair.
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, uint32_t &lo, uint32_t &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// A constant in both halves, kept in registers: volatile, or the compiler would make it again at every use.
__device__ __forceinline__ uint64_t both(float v) {
    uint64_t r;
    asm volatile("mov.b64 %0, {%1, %1};" : "=l"(r) : "r"(__float_as_uint(v)));
    return r;
}

// z << S on the integer pipe (a shift-and-add becomes a multiply-add on the FP32 pipe, which is the busy one).
template <int S>
__device__ __forceinline__ uint32_t shl(uint32_t z) {
    uint32_t r;
    asm("shf.l.wrap.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(0u), "r"(z), "n"(S));
    return r;
}

// 32 x 32 words over a warp turned: r[q] of lane l becomes what r[l] of lane q was.
__device__ __forceinline__ void turn32(uint32_t (&r)[32], int lane) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1)
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            if (q & s) continue;
            const bool up = (lane & s) != 0;
            const uint32_t x = __shfl_xor_sync(0xffffffffu, up ? r[q] : r[q + s], s);
            r[q] = up ? x : r[q];
            r[q + s] = up ? r[q + s] : x;
        }
}

constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: adding it leaves an integer in the low mantissa bits

struct FoldConsts {
    static constexpr float kRound1 = kMagic * 2097152.0f, kRound2 = kMagic * 1024.0f;
    uint64_t neg = both(-1.0f), round1 = both(kRound1), back1 = both(kRound1 + kMagic), round2 = both(kRound2),
             shift = both(2048.0f);
};

// 2^11 (l1 + 2^11 l2) mod 2^32 for two vectors, l1 and l2 integers held as floats (|l| <= 2^24).  F2I runs
// at an eighth of the FP32 rate, so the conversion is made of exact FP32 steps, two vectors per instruction.
// Only l1 mod 2^21 and l2 mod 2^10 matter: adding 1.5 * 2^(23 + K) rounds l to a multiple of
// 2^K, and l minus that multiple is the signed remainder, at most 2^(K - 1) in magnitude.  So
// z = 1.5 * 2^23 + r1 + 2^11 r2 is exact (|r1 + 2^11 r2| <= 2^21), its low mantissa bits are the sum, and the
// constant's bits leave the word when it is shifted by 11 (its lowest set bit is 22).
__device__ __forceinline__ void high_limbs(const FoldConsts &k, uint64_t l1, uint64_t l2, uint32_t &w0, uint32_t &w1) {
    const uint64_t t1 = add2(l1, k.round1);
    const uint64_t z1 = add2(l1, fma2(t1, k.neg, k.back1));   // 1.5 * 2^23 + r1
    const uint64_t t2 = add2(l2, k.round2);
    const uint64_t r2 = add2(l2, fma2(t2, k.neg, k.round2));
    unpack2(fma2(r2, k.shift, z1), w0, w1);
    w0 = shl<11>(w0);
    w1 = shl<11>(w1);
}

}  // namespace

template <int H, int OUT>
__global__ void __launch_bounds__(kTThreads, 1)
    limb_gemm_tri_kernel(const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map,
                         VecSums sums, uint32_t *__restrict__ out, uint64_t ld,
                         uint32_t M, uint32_t NV, uint32_t KB, uint32_t ksplit, int *__restrict__ status) {
    using Cfg = TriCfg<H>;
    constexpr int ST = Cfg::kStages;
    constexpr uint32_t VPT = 64 * H;   // vectors per tile
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + ST * Cfg::kStageBytes);   // [ST], leader's counts
    uint64_t *empty = full + ST;                                                    // [ST], own
    uint64_t *acc_full = empty + ST;                                                // [2], own
    uint64_t *acc_empty = acc_full + 2;                                             // [2], leader's counts
    uint64_t *mma_done = acc_empty + 2;                                             // [1], leader
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 16);   // eight epilogue warps of each CTA
        }
        mbar_init(mma_done, 1);
        *abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    // both CTAs' barriers exist before either touches the other's
    tc_fence_before();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t full_c = cluster_addr(full, 0);
    const uint32_t acc_empty_c = cluster_addr(acc_empty, 0);
    const uint32_t peer_abort = cluster_addr(const_cast<int *>(abort), rank ^ 1u);

    const uint32_t m_tiles = (M + 2 * kTM - 1) / (2 * kTM);
    const uint32_t n_tiles = (NV + VPT - 1) / VPT;
    const uint32_t nchunks = (KB + kChunkSteps - 1) / kChunkSteps;
    // clusters are CTAs 2c, 2c + 1
    TriIter iter{blockIdx.x >> 1, gridDim.x >> 1, n_tiles, m_tiles * n_tiles, nchunks, ksplit, NV, H};
    TriPiece pc;
    bool failed = false;
    auto fail_both = [&]() {
        failed = true;
        *abort = 1;
        st_cluster_u32(peer_abort, 1u);
    };

    // Three halves keep 96 running sums a thread: registers move from the first warpgroup to the epilogue
    // (128 * 88 + 256 * 208 = 384 * 168, what the block was launched with).
    if (warp < 4) {
        if constexpr (H == 3) asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
        if (warp == 0 || warp == 2) {
            if (lane == 0) {
                // ---------------- TMA producers (both CTAs)
                const bool mat = warp == 0;
                tma_prefetch_desc(mat ? &a_map : &b_map);
                if (!mat) griddep_wait();   // the limbs come from the kernel this one overlaps
                uint32_t it = 0, st = 0, ph = 0;
                while (!failed && iter.next(pc)) {
                    const uint32_t kb0 = pc.c0 * kChunkSteps;
                    const uint32_t kb1 = pc.c1 * kChunkSteps < KB ? pc.c1 * kChunkSteps : KB;
                    const int32_t m0 = static_cast<int32_t>(pc.m * 2 * kTM + rank * kTM);
                    const int32_t v0 = static_cast<int32_t>(pc.n * VPT + rank * kTriGroup);
                    for (uint32_t kb = kb0; kb < kb1; ++kb, ++it) {
                        if (!mbar_wait(&empty[st], ph ^ 1u, abort)) {
                            fail_both();
                            break;
                        }
                        uint8_t *sa = smem + st * Cfg::kStageBytes;
                        if (mat) {
                            if (leader)
                                mbar_arrive_expect_tx(&full[st], 2u * (Cfg::kABytes + pc.halves * Cfg::kBoxBytes));
                            tma_load_2d_pair(sa, &a_map, full_c + 8u * st, static_cast<int32_t>(kb * kTK), m0);
                        } else {
#pragma unroll
                            for (int h = 0; h < H; ++h)
                                if (h < (int)pc.halves)
                                    tma_load_3d_pair(sa + Cfg::kABytes + h * Cfg::kBoxBytes, &b_map, full_c + 8u * st,
                                                     static_cast<int32_t>(kb * kTK), v0 + 64 * h, 0);
                        }
                        if (++st == (uint32_t)ST) {
                            st = 0;
                            ph ^= 1u;
                        }
                    }
                }
                if (leader && mat) {
                    // the stages still owed bytes (both producers' and the peer's copies) must land before exit
                    const uint32_t inflight = it < (uint32_t)ST ? it : (uint32_t)ST;
                    for (uint32_t j = it - inflight; j < it; ++j)
                        if (!mbar_drain(&full[j % ST], (j / ST) & 1u)) failed = true;
                }
            }
        } else if (warp == 1) {
            if (leader) {
                // ---------------- MMA issuer (leader only): the whole warp walks the loop, one lane issues
                constexpr uint32_t idesc = umma_idesc_f16(2 * kTM, kTN);
                // One issue block per half of a chunk: its eight MMAs run for 768 cycles, and the waits, votes and
                // election between two blocks have to fit in that beside the epilogue warps' work.
                const uint64_t adesc0 = umma_desc_sw128(smem_addr(smem));
                const uint64_t bdesc0 = umma_desc_sw128(smem_addr(smem) + Cfg::kABytes);
                uint32_t item = 0, st = 0, ph = 0;
                bool issued = false;
                while (!failed && iter.next(pc)) {
                    for (uint32_t c = pc.c0; c < pc.c1; ++c) {
                        const bool two = KB - c * kChunkSteps >= 2;   // else the last 64 columns or fewer
                        const uint32_t s0 = st;
                        bool ok = mbar_wait(&full[s0], ph, abort);
                        if (++st == (uint32_t)ST) {
                            st = 0;
                            ph ^= 1u;
                        }
                        const uint32_t s1 = st;
                        if (two) {
                            ok = ok && mbar_wait(&full[s1], ph, abort);
                            if (++st == (uint32_t)ST) {
                                st = 0;
                                ph ^= 1u;
                            }
                        }
                        const uint64_t a0 = adesc0 + s0 * (Cfg::kStageBytes >> 4), a1 = adesc0 + s1 * (Cfg::kStageBytes >> 4);
                        const uint64_t b0 = bdesc0 + s0 * (Cfg::kStageBytes >> 4), b1 = bdesc0 + s1 * (Cfg::kStageBytes >> 4);
#pragma unroll
                        for (int h = 0; h < H; ++h) {
                            if (h >= (int)pc.halves) break;
                            const uint32_t buf = item & 1u;
                            ok = ok && mbar_wait(&acc_empty[buf], ((item >> 1) & 1u) ^ 1u, abort);
                            if (__any_sync(0xffffffffu, !ok)) {
                                fail_both();
                                break;
                            }
                            tc_fence_after();
                            const uint32_t d_tmem = tmem_base + buf * kTN;
                            if (elect_one()) {
#pragma unroll
                                for (int kk = 0; kk < kTK / 16; ++kk)
                                    umma_f16_pair(d_tmem, a0 + 2u * kk, b0 + h * (Cfg::kBoxBytes >> 4) + 2u * kk, idesc,
                                                  kk != 0 ? 1u : 0u);
                                if (h == (int)pc.halves - 1) umma_commit_pair(&empty[s0], 3);
                                if (two) {
#pragma unroll
                                    for (int kk = 0; kk < kTK / 16; ++kk)
                                        umma_f16_pair(d_tmem, a1 + 2u * kk, b1 + h * (Cfg::kBoxBytes >> 4) + 2u * kk, idesc,
                                                      1u);
                                    if (h == (int)pc.halves - 1) umma_commit_pair(&empty[s1], 3);
                                }
                                umma_commit_pair(&acc_full[buf], 3);
                            }
                            __syncwarp();
                            issued = true;
                            ++item;
                        }
                        if (failed) break;
                    }
                }
                // every pair MMA must finish before TMEM is released
                if (issued) {
                    if (elect_one()) umma_commit_pair(mma_done, 1);
                    __syncwarp();
                    if (!mbar_drain(mma_done, 0)) failed = true;
                }
            }
        }
    } else {
        if constexpr (H == 3) asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
        // ---------------- epilogue (both CTAs): TMEM lane quarter = warp % 4, box = (warp - 4) / 4
        const uint32_t quarter = static_cast<uint32_t>(warp & 3);
        const uint32_t box = static_cast<uint32_t>(warp - 4) >> 2;
        const uint32_t taddr = tmem_base + ((quarter * 32u) << 16) + 96u * box;
        const FoldConsts consts;
        griddep_wait();   // the sums and the zeroed output come from the kernel this one overlaps
        uint32_t item = 0;
        while (!failed && iter.next(pc)) {
            const uint32_t row = pc.m * 2 * kTM + rank * kTM + quarter * 32u + static_cast<uint32_t>(lane);
            const uint32_t v0 = pc.n * VPT + box * kTriGroup;
            uint32_t run[H][32];
            uint32_t held[H];   // lane q: what the first range of a tile adds to vector q, whose digits were centred
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t v = v0 + 64u * h + static_cast<uint32_t>(lane);
                held[h] = pc.c0 == 0 && v < NV ? sums.centred(v) : 0u;
#pragma unroll
                for (int q = 0; q < 32; ++q) run[h][q] = 0u;
            }
            for (uint32_t c = pc.c0; c < pc.c1 && !failed; ++c) {
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    if (h >= (int)pc.halves) break;
                    const uint32_t buf = item & 1u;
                    ++item;
                    const bool ok = mbar_wait(&acc_full[buf], ((item - 1) >> 1) & 1u, abort);
                    if (__any_sync(0xffffffffu, !ok)) {   // the TMEM loads below are warp-collective
                        fail_both();
                        break;
                    }
                    tc_fence_after();
                    const uint32_t acc = taddr + buf * kTN;
#pragma unroll
                    for (int j = 0; j < 32; j += 16) {
                        uint32_t l[3][16];
#pragma unroll
                        for (int k = 0; k < 3; ++k) tmem_ld16(acc + 32u * k + j, l[k]);
                        tmem_wait_ld();
                        if (j == 16) {   // everything is in registers
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive_cluster(acc_empty_c + 8u * buf);
                        }
#pragma unroll
                        for (int q = 0; q < 16; q += 2) {
                            uint32_t hi0, hi1;
                            const uint32_t lo0 = static_cast<uint32_t>(__float2int_rn(__uint_as_float(l[0][q])));
                            const uint32_t lo1 = static_cast<uint32_t>(__float2int_rn(__uint_as_float(l[0][q + 1])));
                            high_limbs(consts, pack2(l[1][q], l[1][q + 1]), pack2(l[2][q], l[2][q + 1]), hi0, hi1);
                            run[h][j + q] += lo0 + hi0;
                            run[h][j + q + 1] += lo1 + hi1;
                        }
                    }
                }
            }
            if (failed) break;
            const bool whole = pc.c0 == 0 && pc.c1 == nchunks;   // no other cluster works on this tile
#pragma unroll
            for (int h = 0; h < H; ++h)
#pragma unroll
                for (int q = 0; q < 32; ++q) run[h][q] += __shfl_sync(0xffffffffu, held[h], q);
            if constexpr (OUT == kTurned) {
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    turn32(run[h], lane);
                    const uint32_t v = v0 + 64u * h + static_cast<uint32_t>(lane), i0 = row - static_cast<uint32_t>(lane);
                    uint32_t *dst = out + (uint64_t)i0 * ld + v;
#pragma unroll
                    for (int q = 0; q < 32; ++q, dst += ld) {
                        if (v >= NV || i0 + q >= M) continue;
                        if (whole) *dst = run[h][q];
                        else atomicAdd(dst, run[h][q]);
                    }
                }
            } else if (row < M) {
#pragma unroll
                for (int h = 0; h < H; ++h) {
                    if (OUT == kQuads && v0 + 64u * h + 32u <= NV) {   // 32 neighbouring words of a row
                        uint4 *dst = reinterpret_cast<uint4 *>(out + (uint64_t)row * ld + v0 + 64u * h);
#pragma unroll
                        for (int q = 0; q < 32; q += 4)
                            dst[q / 4] = make_uint4(run[h][q], run[h][q + 1], run[h][q + 2], run[h][q + 3]);
                        continue;
                    }
                    const uint32_t v = v0 + 64u * h, n = NV > v ? NV - v : 0u;
                    uint32_t *dst = out + (OUT == kWords ? row + (uint64_t)v * ld : (uint64_t)row * ld + v);
#pragma unroll
                    for (uint32_t q = 0; q < 32; ++q, dst += OUT == kWords ? ld : 1) {
                        if (q >= n) continue;
                        if (OUT == kQuads || whole) *dst = run[h][q];
                        else atomicAdd(dst, run[h][q]);
                    }
                }
            }
        }
    }

    if (failed) {
        *abort = 1;
        *status = kDevTimeout;
        // a copy this CTA issued may still be landing (after an abort its stage is never
        // consumed): give it a bounded moment before the CTA can exit
        const uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) {
        }
    }
    // no CTA leaves (or frees TMEM) while its peer may still reach its shared memory or TMEM
    __syncwarp();
    tc_fence_before();
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// ------------------------------------------------------------------ limbs
// x = l0 + 2^11 l1 + 2^22 l2 (mod 2^32), |l0|, |l1| <= 2^10, |l2| <= 2^9.
__device__ __forceinline__ void balanced(uint32_t x, int (&l)[3]) {
    l[0] = static_cast<int>(x << 21) >> 21;
    x = (x - static_cast<uint32_t>(l[0])) >> 11;   // 21 bits
    l[1] = static_cast<int>(x << 21) >> 21;
    x = (x - static_cast<uint32_t>(l[1])) >> 11;   // 10 bits and a carry, which 2^32 drops
    l[2] = static_cast<int>(x << 22) >> 22;
}

// x = sum_k 2^{8k} l_k (mod 2^32), |l_k| <= 2^7.
__device__ __forceinline__ void balanced(uint32_t x, int (&l)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        l[k] = static_cast<int>(x << 24) >> 24;
        x = (x - static_cast<uint32_t>(l[k])) >> 8;
    }
}

__device__ __forceinline__ void store8(__half *dst, const int (&l)[8]) {
    __align__(16) __half h[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = __int2half_rn(l[i]);
    *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(h);
}

// Block (x, y) makes the limbs of columns [2048 x, 2048 x + 2048) of vector y, 8 consecutive columns per thread, and
// the sum of those words; the GEMM adds a vector's sums up.  One block per vector and whole row left SMs idle and
// made every thread walk: 130 vectors of 30000 columns 10.5 us, 7.5 this way; 256 of 32768 (three limbs) 20 and
// 16; a cluster of blocks per vector that adds up in shared memory 11.1 and 20.  z: words to zero (the output of a
// GEMM whose pieces add up).
template <int LIMBS>
__global__ void __launch_bounds__(kSumCols / 8) vec_limbs_sums_kernel(const uint32_t *__restrict__ X, uint64_t x_ld, uint64_t C,
                                                                     __half *__restrict__ L, uint64_t pitch,
                                                                     uint32_t *__restrict__ sums, uint32_t *__restrict__ Z,
                                                                     uint64_t z_words) {
    griddep_launch_dependents();   // the GEMM's start overlaps this kernel; it waits before it reads the limbs
    for (uint64_t i = ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < z_words;
         i += (uint64_t)gridDim.x * gridDim.y * blockDim.x)
        Z[i] = 0u;
    const uint32_t *src = X + (uint64_t)blockIdx.y * x_ld;
    __half *dst = L + (uint64_t)LIMBS * blockIdx.y * pitch;
    const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0;
    uint32_t sum = 0;
    const uint64_t j0 = (uint64_t)blockIdx.x * kSumCols + threadIdx.x * 8;
    if (vec && j0 + 8 <= C) {
        const uint4 a = *reinterpret_cast<const uint4 *>(src + j0);
        const uint4 b = *reinterpret_cast<const uint4 *>(src + j0 + 4);
        const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        int l[LIMBS][8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            int t[LIMBS];
            balanced(x[i], t);
#pragma unroll
            for (int k = 0; k < LIMBS; ++k) l[k][i] = t[k];
            sum += x[i];
        }
#pragma unroll
        for (int k = 0; k < LIMBS; ++k) store8(dst + k * pitch + j0, l[k]);   // pitch % 8 == 0
    } else {
        for (uint64_t j = j0; j < C && j < j0 + 8; ++j) {
            int t[LIMBS];
            balanced(src[j], t);
            for (int k = 0; k < LIMBS; ++k) dst[k * pitch + j] = __int2half_rn(t[k]);
            sum += src[j];
        }
    }
    __shared__ uint32_t part[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t w = 1; w < blockDim.x / 32; ++w) sum += part[w];
        sums[(uint64_t)blockIdx.x * gridDim.y + blockIdx.y] = sum;
    }
}

// A (uint32, C x n row-major): block (x, y) turns rows [128 x, 128 x + 128) x columns [32 y, 32 y + 32)
// through shared memory; 16 threads write one column's 128 limbs, 16 bytes each.
template <int LIMBS>
__global__ void __launch_bounds__(256) mat_col_limbs_sums_kernel(const uint32_t *__restrict__ A, uint64_t C, uint32_t n,
                                                                 __half *__restrict__ L, uint64_t pitch,
                                                                 uint32_t *__restrict__ sums, uint32_t *__restrict__ Z,
                                                                 uint64_t z_words) {
    griddep_launch_dependents();   // as in vec_limbs_sums_kernel
    for (uint64_t i = ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < z_words;
         i += (uint64_t)gridDim.x * gridDim.y * blockDim.x)
        Z[i] = 0u;
    __shared__ uint32_t tile[128][33];
    const uint64_t j0 = (uint64_t)blockIdx.x * 128;
    const uint32_t k0 = blockIdx.y * 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int row = warp + 8 * r;
        const bool in = j0 + row < C && k0 + lane < n;
        tile[row][lane] = in ? A[(j0 + row) * n + k0 + lane] : 0u;
    }
    __syncthreads();
    const int t = threadIdx.x & 15;
    const bool aligned = (reinterpret_cast<uintptr_t>(L) & 15u) == 0;
    for (uint32_t kk = threadIdx.x >> 4; kk < 32; kk += 16) {
        const uint32_t k = k0 + kk;
        int l[LIMBS][8];
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t x = tile[8 * t + i][kk];
            int u[LIMBS];
            balanced(x, u);
#pragma unroll
            for (int m = 0; m < LIMBS; ++m) l[m][i] = u[m];
            sum += x;
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);   // over the column's 16 threads
        if (k >= n) continue;
        if (t == 0) atomicAdd(sums + k, sum);
        const uint64_t j = j0 + 8 * t;
        __half *dst = L + (uint64_t)LIMBS * k * pitch + j;
#pragma unroll
        for (int u = 0; u < LIMBS; ++u) {
            if (aligned && j + 8 <= C) {
                store8(dst + u * pitch, l[u]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (j + i < C) dst[u * pitch + i] = __int2half_rn(l[u][i]);
            }
        }
    }
}

// ------------------------------------------------------------------ host side
template <int LIMBS>
static cudaError_t launch_vec_limbs_sums(const uint32_t *X, uint64_t x_ld, uint32_t NV, uint64_t C, __half *L,
                                         uint64_t pitch, const VecSums &sums, uint32_t *zero, uint64_t zero_words,
                                         cudaStream_t stream) {
    if (NV == 0 || C == 0 || NV > 65535 || pitch % 8 != 0) return cudaErrorInvalidValue;
    const uint64_t want = ((C + 7) / 8 + 31) / 32 * 32;   // threads for all columns
    vec_limbs_sums_kernel<LIMBS>
        <<<dim3(sums.parts, NV), static_cast<unsigned>(want < kSumCols / 8 ? want : kSumCols / 8), 0, stream>>>(
            X, x_ld, C, L, pitch, const_cast<uint32_t *>(sums.words), zero, zero ? zero_words : 0);
    return cudaGetLastError();
}

cudaError_t launch_vec_limbs_tri(const uint32_t *X, uint64_t x_ld, uint32_t NV, uint64_t C, __half *L, uint64_t pitch,
                                 uint32_t *zero, uint64_t zero_words, cudaStream_t stream) {
    return launch_vec_limbs_sums<3>(X, x_ld, NV, C, L, pitch, tri_sums(L, NV, pitch, limb_sum_parts(C)), zero, zero_words,
                                    stream);
}

cudaError_t launch_vec_limbs_four(const uint32_t *X, uint64_t x_ld, uint32_t NV, uint64_t C, __half *L, uint64_t pitch,
                                  uint32_t *zero, uint64_t zero_words, cudaStream_t stream) {
    return launch_vec_limbs_sums<4>(X, x_ld, NV, C, L, pitch, four_sums(L, NV, pitch, limb_sum_parts(C)), zero,
                                    zero_words, stream);
}

template <int LIMBS>
static cudaError_t launch_mat_col_limbs_sums(const uint32_t *A, uint64_t C, uint32_t n, __half *L, uint64_t pitch,
                                             const VecSums &vs, uint32_t *zero, uint64_t zero_words,
                                             cudaStream_t stream) {
    if (n == 0 || C == 0 || pitch % 8 != 0) return cudaErrorInvalidValue;
    uint32_t *sums = const_cast<uint32_t *>(vs.words);
    const cudaError_t e = cudaMemsetAsync(sums, 0, 4ull * n, stream);
    if (e != cudaSuccess) return e;
    const dim3 grid(static_cast<unsigned>((C + 127) / 128), (n + 31) / 32);
    mat_col_limbs_sums_kernel<LIMBS><<<grid, 256, 0, stream>>>(A, C, n, L, pitch, sums, zero, zero ? zero_words : 0);
    return cudaGetLastError();
}

cudaError_t launch_mat_col_limbs_tri(const uint32_t *A, uint64_t C, uint32_t n, __half *L, uint64_t pitch,
                                     uint32_t *zero, uint64_t zero_words, cudaStream_t stream) {
    return launch_mat_col_limbs_sums<3>(A, C, n, L, pitch, tri_sums(L, n, pitch, 1), zero, zero_words, stream);
}

cudaError_t launch_mat_col_limbs_four(const uint32_t *A, uint64_t C, uint32_t n, __half *L, uint64_t pitch,
                                      cudaStream_t stream) {
    return launch_mat_col_limbs_sums<4>(A, C, n, L, pitch, four_sums(L, n, pitch, 1), nullptr, 0, stream);
}

template <int H>
static cudaError_t set_tri_attrs() {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(limb_gemm_tri_kernel<H, kWords>, attr, TriCfg<H>::kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(limb_gemm_tri_kernel<H, kQuads>, attr, TriCfg<H>::kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(limb_gemm_tri_kernel<H, kTurned>, attr, TriCfg<H>::kSmemBytes);
    return e;
}

cudaError_t prepare_limb_gemm_tri_kernels() {
    cudaError_t e = set_tri_attrs<1>();
    if (e == cudaSuccess) e = set_tri_attrs<2>();
    if (e == cudaSuccess) e = set_tri_attrs<3>();
    return e;
}

template <int H>
static cudaLaunchConfig_t tri_config(unsigned clusters, cudaStream_t stream, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * clusters);
    cfg.blockDim = dim3(kTThreads);
    cfg.dynamicSmemBytes = TriCfg<H>::kSmemBytes;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // overlaps the limb kernel before it
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// CTA pairs that fit on the GPU at once, per device (a GPC with an odd number of SMs leaves one idle).
template <int H>
static int tri_resident_pairs(int num_sms) {
    static int cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return num_sms / 2;
    if (cache[dev] > 0) return cache[dev];
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = tri_config<H>(static_cast<unsigned>(num_sms / 2), nullptr, attr);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, limb_gemm_tri_kernel<H, kWords>, &cfg) != cudaSuccess || n <= 0) {
        cudaGetLastError();
        return num_sms / 2;
    }
    n = n < num_sms / 2 ? n : num_sms / 2;
    cache[dev] = n;
    return n;
}

// The time in us of tiles of `h` halves cut into `s` column ranges, limb pass and launches included: whole waves of
// ranges on `pairs` clusters, each with its chunks (a half's tensor or drain time, more for one half a tile, which
// loads a digit tile for 192 columns, and more again when the digits do not stay in L2), its filling, draining and
// storing; ranges add their parts to the output.  Fitted to 6,200 graph-replayed calls (370 shapes of 300 to 65,536
// rows, 400 to 40,000 columns and 65 to 1,024 vectors, every form of each).  The form chosen by it was 0.6% from the
// best of them on average; two or three halves in at most 8 ranges of 1024 columns had been 13% from it on the 240
// regular ones: 300 x 30000 with 66 vectors 41 us against 18, 2000 x 16000 with 320 76 / 60, 1200 x 1900 with 128 16 / 10.
static double tri_time(uint32_t M, uint32_t NV, uint64_t K, uint64_t tiles, uint64_t pairs, double chunks, int h,
                       uint32_t s) {
    const double half = h == 2 ? 0.527 : (h == 3 ? 0.592 : (2.0 * M * K > 64e6 ? 0.627 : 0.605));
    const double waves = static_cast<double>((tiles * s + pairs - 1) / pairs);
    const double adding = s > 1 ? 0.5e-6 * M * NV * s : 0.0;
    return 5.6 + 1.5e-6 * K * NV + waves * (h * (half * chunks / s + 1.7) + 0.2) + adding;
}

TriPlan limb_gemm_tri_plan(uint32_t M, uint32_t NV, uint64_t K, int num_sms) {
    const uint64_t m_tiles = ((uint64_t)M + 2 * kTM - 1) / (2 * kTM);
    const uint32_t nh = (NV - 1) / 64 + 1;
    const uint64_t chunks = (K + kTK * kChunkSteps - 1) / (kTK * kChunkSteps);
    TriPlan whole{0, 1, 0.0}, cut{0, 1, 0.0};
    for (int h = 1; h <= 3 && h <= (int)nh; ++h) {
        const int n = h == 1 ? tri_resident_pairs<1>(num_sms) : (h == 2 ? tri_resident_pairs<2>(num_sms) : tri_resident_pairs<3>(num_sms));
        const uint64_t pairs = n > 0 ? n : 1, tiles = m_tiles * ((nh + h - 1) / h);
        auto consider = [&](uint64_t s) {
            if (s > 1 && (s > pairs || s > chunks / 2)) return;   // ranges of at least two chunks
            TriPlan &best = s == 1 ? whole : cut;
            const double us = tri_time(M, NV, K, tiles, pairs, static_cast<double>(chunks), h, static_cast<uint32_t>(s));
            if (best.halves == 0 || us < best.us) best = TriPlan{h, static_cast<uint32_t>(s), us};
        };
        // up to 8 ranges, or the most that fit one, two or three waves
        for (uint64_t s = 1; s <= 8; ++s) consider(s);
        for (uint64_t w = 1; w <= 3; ++w)
            if (w * pairs / tiles > 8) consider(w * pairs / tiles);
    }
    // ranges need a zeroed output and atomics: not for less than 2%
    return cut.halves != 0 && cut.us < 0.98 * whole.us ? cut : whole;
}

template <int H>
static cudaError_t launch_tri_t(const CUtensorMap &a_map, const CUtensorMap &b_map, const VecSums &sums, uint32_t *out,
                                uint64_t ld_m, uint64_t ld_b, uint32_t M, uint32_t NV, uint32_t KB, uint32_t ranges,
                                int num_sms, int *status, cudaStream_t stream) {
    const uint64_t tiles = ((uint64_t)M + 2 * kTM - 1) / (2 * kTM) * (((uint64_t)NV + 64 * H - 1) / (64 * H));
    const uint64_t pairs = static_cast<uint64_t>(tri_resident_pairs<H>(num_sms));
    const uint64_t units = tiles * ranges;
    if (pairs == 0 || units >= (1ull << 31)) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = tri_config<H>(static_cast<unsigned>(units < pairs ? units : pairs), stream, attr);
    const bool rows = ld_m != 1, quads = ld_m % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
    if (rows && ld_b != 1) return cudaErrorInvalidValue;
    // 16-byte stores are for whole tiles: ranges add a word at a time
    const auto kernel = !rows ? limb_gemm_tri_kernel<H, kWords>
                              : (quads && ranges == 1 ? limb_gemm_tri_kernel<H, kQuads> : limb_gemm_tri_kernel<H, kTurned>);
    return cudaLaunchKernelEx(&cfg, kernel, a_map, b_map, sums, out, rows ? ld_m : ld_b, M, NV, KB, ranges, status);
}

cudaError_t launch_limb_gemm_tri(const CUtensorMap &a_map, const CUtensorMap &b_map, const VecSums &sums,
                                 uint32_t *out, uint64_t ld_m, uint64_t ld_b, uint32_t M, uint32_t NV, uint64_t K,
                                 const TriPlan &plan, int num_sms, int *status, cudaStream_t stream) {
    if (M == 0 || NV == 0 || K == 0 || plan.ranges == 0 || num_sms < 2) return cudaErrorInvalidValue;
    const uint32_t KB = static_cast<uint32_t>((K + kTK - 1) / kTK);
    switch (plan.halves) {
        case 1: return launch_tri_t<1>(a_map, b_map, sums, out, ld_m, ld_b, M, NV, KB, plan.ranges, num_sms, status, stream);
        case 2: return launch_tri_t<2>(a_map, b_map, sums, out, ld_m, ld_b, M, NV, KB, plan.ranges, num_sms, status, stream);
        case 3: return launch_tri_t<3>(a_map, b_map, sums, out, ld_m, ld_b, M, NV, KB, plan.ranges, num_sms, status, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace qpadl
