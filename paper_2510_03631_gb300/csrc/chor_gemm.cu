// GF(2) Response of a batch on the tensor cores (Chor-style PIR, Sec. 5.2, Alg. 3):
//   rho_b[c] = parity of #{ i : query bit q_b[i] and database bit DB[i][c] both set }.
//
// The counts are a matrix product of 0/1 matrices, which the 4-bit tensor-core kind takes exactly
// (tcgen05 kind::mxf4, e2m1 operands, every block scale 1, fp32 accumulators): a product is 0 or
// one constant, a count below 2^22 is exact in fp32, and its low bit is the answer.  Work per
// launch: rows x bits x queries multiply-adds at 32,768 flop per SM and clock (measured: one MMA of
// 128 x N x 64 takes N / 2 cycles), against one XOR per 32 of them on the ALUs.
//
// Operands.  M is database columns (bits), N queries, K database rows.  The database is read as
// stored; turning its bits into K-major 4-bit operands is the real work, done in two steps by
// different warps so that each byte is touched once:
//   1. Rows are transposed by nibbles: ldmatrix turns 16 x 16 bytes on the way into registers, and four
//      shift/select operations turn two such words (byte b of 4 + 4 rows) into one word for each nibble
//      of the byte: word j then holds nibble j (bits 4j..4j+3) of 8 rows.
//   2. One thread per (word, nibble j) pair, i.e. per TMEM lane, reads its 32 words (256 rows) and
//      masks out bit s of every nibble for each of the planes s it needs: x & (0x11111111 << s) is a
//      row of 8 e2m1 values 0.5, 1 or 2 (bit 3, the sign, is shifted down to 2's place).  One AND
//      makes 8 operand elements.  The four planes are four M = 128 tiles that share one load: lane
//      8w + j of plane s is bit 4j + s of word w.
// The queries' bits become e2m1 ones in a small kernel before (B x rows / 2 bytes), in the same row
// order, and TMA brings them in 128-byte-swizzled tiles.
//
// A unit is 16 database words (64 bytes per row) x 256 rows.  Up to 64 queries a CTA runs all four
// planes (accumulators 4 x 64 TMEM columns); up to 128 queries two CTAs take two planes each
// (2 x 128 columns), both reading and transposing the same words, the second from L2: the tensor
// work of 128 queries outweighs it.  Larger batches are several tiles of 128 queries (a tile of 256 queries would
// leave room for one plane, so each unit would be transposed four times), in one launch as far as the scratch
// holds their expanded bits.
//
// Measured (2^18 records of 3 KB, 805 MB): 64 queries 195 us, 128 queries 300 us; the kernels it
// replaced took 1,085 and 1,130 us there (four-Russians tables in shared memory) and 606 us at 32
// queries (masked scan).  What bounds it: at 128 queries the tensor pipe is 59% and the ALUs 63% busy,
// at 64 queries 45% and 63% (HBM floor 120 us): the chain transpose -> planes -> MMA, with about six
// units in flight.  At the 80 registers that 768 threads leave, the kernels for 32 and 64 queries spill 50 bytes.  Tried on the way: one producer for both operand streams (396 us at 128: the query
// ring held the database back); one issuing warp (an MMA costs its lane about 42 cycles and each wait
// 110); byte permutes instead of ldmatrix for step 1 (the ALUs' 64 lanes per clock); both steps in the
// same warps (373 us).
//
// Schedule.  A piece is one column tile over one band of rows; pieces are numbered band by band, so
// the CTAs that run together read neighbouring columns of the same rows (whole DRAM pages, and 256-
// byte lines shared through L2).  The number of bands is chosen so that the pieces fill the last
// wave.  A piece ends with its parities XORed into the zeroed answer (32-bit atomics: exact and
// order-independent).
//
// Warp roles (768 threads, one CTA per SM):
//   warps 0, 23   TMA producers (database boxes; query tiles)
//   warps 1, 22   MMA issue, half of the planes each (warp 1 also allocates TMEM)
//   warps 2..5    epilogue: parities of a piece's counts, collected by ballots into words
//   warps 6..13   step 1, two groups of four, each every other unit
//   warps 14..21  step 2, two groups of four (one TMEM lane per thread), each every other unit
// Every mbarrier wait is bounded; a CTA that gives up records kDevTimeout and leaves.
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "chor.cuh"
#include "ptx.cuh"

namespace qpadl {

namespace {

constexpr int kGThreads = 768;
constexpr int kIssuers = 2;   // MMA-issuing warps (1 and 22), each with half of the planes
constexpr uint32_t kUnitRows = kChorGemmUnitRows;       // 256
constexpr uint32_t kUnitWords = kChorGemmUnitWords;     // 16
constexpr uint32_t kRawBytes = kUnitRows * kUnitWords * 4;   // 16 KB
constexpr uint32_t kXBytes = kRawBytes;                 // the nibble-transposed unit
constexpr int kRawSlots = 4, kXSlots = 4, kASets = 3;
constexpr uint32_t kAccBase = 0, kScaleBase = 256, kABase = 320, kSetCols = 64, kTmem = 512;

// N queries; MT planes per CTA (4 for N <= 64, 2 for 128).
template <int N, int MT>
struct GCfg {
    static constexpr uint32_t kQBytes = N * 128;        // one unit's query tile: 256 rows as nibbles
    static constexpr int kQSlots = 6;
    static constexpr int kSets = MT == 4 ? 2 : 1;       // operand sets (64 TMEM columns) per unit
    static constexpr uint32_t kQBase = kRawSlots * kRawBytes + kXSlots * kXBytes;
    static constexpr uint32_t kBarBase = kQBase + kQSlots * kQBytes;
    static constexpr int kBars = 2 * (kRawSlots + kXSlots + kQSlots + kASets) + 3;
    static constexpr int kSmemBytes = kBarBase + kBars * 8 + 16 + 1024;
    static_assert(MT * N <= 256, "accumulators");
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
};

// D[tmem] (+)= A[tmem] * B[smem]^T, e2m1 operands in blocks of 32 with scales [sa], [sb].
__device__ __forceinline__ void umma_mxf4_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t sa, uint32_t sb,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%4], [%5], p;\n\t}" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(sa), "r"(sb), "r"(accumulate)
        : "memory");
}
// Instruction descriptor: e2m1 x e2m1 -> fp32, both K-major, ue8m0 scales.
__host__ __device__ constexpr uint32_t umma_idesc_mxf4(uint32_t M, uint32_t N) {
    return (1u << 7) | (1u << 10) | ((N >> 3) << 17) | (1u << 23) | ((M >> 7) << 27);
}

// Bit i of a byte to bit 4i.
__device__ __forceinline__ uint32_t spread4(uint32_t x) {
    x = (x | (x << 12)) & 0x000F000Fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
}

// Two 16 x 16 byte matrices (rows of 16 bytes at the lanes' addresses), transposed: lane l gets the
// four rows 4 (l % 4) .. of byte column l / 4 of the first (a0) and second (b0), and of column
// l / 4 + 8 (a1, b1).
__device__ __forceinline__ void ldmatrix_bytes(uint32_t addr, uint32_t &a0, uint32_t &a1, uint32_t &b0, uint32_t &b1) {
    asm volatile("ldmatrix.sync.aligned.m16n16.x2.trans.shared.b8 {%0, %1, %2, %3}, [%4];"
                 : "=r"(a0), "=r"(a1), "=r"(b0), "=r"(b1)
                 : "r"(addr)
                 : "memory");
}

// Order of the 16-byte chunks in lane L's 128 bytes of a transposed unit: chunk i lies at i ^ x_perm(L).
// Eight neighbouring lanes have eight values (step 2's loads), and lanes two apart have opposite
// parity (step 1's stores), so neither meets bank conflicts.
__device__ __forceinline__ uint32_t x_perm(uint32_t L) { return (L ^ ((L & 7u) >> 1) ^ (L >> 3)) & 7u; }

// A CTA's pieces: p = blockIdx.x, blockIdx.x + gridDim.x, ...; the query tiles of one column tile and band are
// neighbours, so the database is read from HBM once for all of them.
struct GPiece {
    uint32_t tile, q, u0, u1;   // column tile, query tile, units [u0, u1) along the rows
};
struct GPieceIter {
    uint32_t p;
    __device__ __forceinline__ GPieceIter() : p(blockIdx.x) {}
    __device__ __forceinline__ bool next(GPiece &pc, uint32_t tiles, uint32_t qtiles, uint32_t bands, uint32_t units) {
        if (p >= tiles * qtiles * bands) return false;
        const uint32_t t = p / qtiles, band = t / tiles;
        pc.q = p - t * qtiles;
        pc.tile = t - band * tiles;
        pc.u0 = static_cast<uint32_t>((uint64_t)band * units / bands);
        pc.u1 = static_cast<uint32_t>((uint64_t)(band + 1) * units / bands);
        p += gridDim.x;
        return true;
    }
};

}  // namespace

template <int N, int MT>
__global__ void __launch_bounds__(kGThreads, 1)
    chor_gemm_kernel(const __grid_constant__ CUtensorMap db_map, const __grid_constant__ CUtensorMap q_map, uint32_t row0,
                     uint32_t units, uint32_t tiles, uint32_t qtiles, uint32_t bands, uint32_t W, uint32_t B,
                     uint32_t *__restrict__ out, int *__restrict__ status) {
    using Cfg = GCfg<N, MT>;
    constexpr int SQ = Cfg::kQSlots, SETS = Cfg::kSets;
    if constexpr (MT == 4) qtiles = 1;   // narrow tiles take one batch each
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *raw = smem, *xt = smem + kRawSlots * kRawBytes, *qt = smem + Cfg::kQBase;
    uint64_t *rfull = reinterpret_cast<uint64_t *>(smem + Cfg::kBarBase);
    uint64_t *rfree = rfull + kRawSlots;
    uint64_t *xfull = rfree + kRawSlots;
    uint64_t *xfree = xfull + kXSlots;
    uint64_t *qfull = xfree + kXSlots;
    uint64_t *qfree = qfull + SQ;
    uint64_t *afull = qfree + SQ;
    uint64_t *afree = afull + kASets;
    uint64_t *acc_full = afree + kASets;
    uint64_t *acc_free = acc_full + 1;
    uint64_t *mma_done = acc_free + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    volatile int *abort = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t quarter = static_cast<uint32_t>(warp & 3);   // TMEM lane quarter of the warps that touch it
    if (threadIdx.x == 0) {
        for (int s = 0; s < kRawSlots; ++s) {
            mbar_init(&rfull[s], 1);
            mbar_init(&rfree[s], 4);
        }
        for (int s = 0; s < kXSlots; ++s) {
            mbar_init(&xfull[s], 4);
            mbar_init(&xfree[s], 4);
        }
        for (int s = 0; s < SQ; ++s) {
            mbar_init(&qfull[s], 1);
            mbar_init(&qfree[s], kIssuers);
        }
        for (int s = 0; s < kASets; ++s) {
            mbar_init(&afull[s], 4);
            mbar_init(&afree[s], kIssuers);
        }
        mbar_init(acc_full, kIssuers);
        mbar_init(acc_free, 4);
        mbar_init(mma_done, kIssuers);
        *abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kTmem);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp >= 2 && warp < 6) {   // every block scale is 1 (ue8m0 127): any scale layout reads the same
        uint32_t one[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) one[i] = 0x7F7F7F7Fu;
        tmem_st32(tmem + ((quarter * 32u) << 16) + kScaleBase, one);
        tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    bool failed = false;
    auto fail_here = [&]() {
        failed = true;
        *abort = 1;
    };
    GPieceIter pit;
    GPiece pc;

    if (warp == 0 || warp == 23) {
        if (lane == 0) {
            // ---------------- TMA producers: warp 0 the database, warp 23 the query tiles.  They are
            // apart because a query tile is held until its MMAs complete: one producer for both kept
            // the database at most that ring ahead of the MMAs, less than the pipeline is long.
            const bool db = warp == 0;
            const CUtensorMap *map = db ? &db_map : &q_map;
            uint64_t *full = db ? rfull : qfull, *free_ = db ? rfree : qfree;
            const uint32_t slots = db ? kRawSlots : SQ;
            uint32_t it = 0, sl = 0, ph = 0;
            tma_prefetch_desc(map);
            while (!failed && pit.next(pc, tiles, qtiles, bands, units)) {
                const int32_t x = static_cast<int32_t>((MT == 4 ? pc.tile : pc.tile >> 1) * kUnitWords);
                for (uint32_t u = pc.u0; u < pc.u1; ++u, ++it) {
                    if (!mbar_wait(&free_[sl], ph ^ 1u, abort)) {
                        fail_here();
                        break;
                    }
                    if (db) {
                        mbar_arrive_expect_tx(&full[sl], kRawBytes);
                        tma_load_2d(raw + sl * kRawBytes, map, &full[sl], x, static_cast<int32_t>(row0 + u * kUnitRows));
                    } else {
                        mbar_arrive_expect_tx(&full[sl], Cfg::kQBytes);
                        tma_load_2d(qt + sl * Cfg::kQBytes, map, &full[sl], static_cast<int32_t>(u * 128u),
                                    static_cast<int32_t>(pc.q * N));
                    }
                    if (++sl == slots) {
                        sl = 0;
                        ph ^= 1u;
                    }
                }
            }
            // copies in flight must land before the CTA exits
            for (uint32_t j = it - (it < slots ? it : slots); j < it; ++j)
                if (!mbar_drain(&full[j % slots], (j / slots) & 1u)) failed = true;
        }
    } else if (warp == 1 || warp == 22) {
        // ---------------- MMA issuers: the whole warp walks the loop, one lane issues.  Two warps issue,
        // each for its own planes' accumulators: one alone took about 1,000 cycles per unit (64
        // queries) where the tensor cores take 512.
        constexpr uint32_t idesc = umma_idesc_mxf4(128, N);
        constexpr int KSTEPS = 4 / SETS;                 // 64-row steps per set and plane
        constexpr int PW = MT / kIssuers;                // planes per issuer
        const uint32_t s0 = warp == 1 ? 0u : PW;
        uint32_t it = 0, is = 0, np = 0;                 // units, sets, pieces
        while (!failed && pit.next(pc, tiles, qtiles, bands, units)) {
            bool ok = mbar_wait(acc_free, (np & 1u) ^ 1u, abort);
            for (uint32_t u = pc.u0; u < pc.u1; ++u, ++it) {
                const uint32_t q = it % SQ;
                const uint64_t bdesc = umma_desc_sw128(smem_addr(qt + q * Cfg::kQBytes));
#pragma unroll
                for (int h = 0; h < SETS; ++h, ++is) {
                    const uint32_t a = is % kASets;
                    const bool a_there = mbar_test(&afull[a], (is / kASets) & 1u);
                    const bool q_there = h != 0 || mbar_test(&qfull[q], (it / SQ) & 1u);
                    if (!a_there) ok = ok && mbar_wait(&afull[a], (is / kASets) & 1u, abort);
                    if (!q_there) ok = ok && mbar_wait(&qfull[q], (it / SQ) & 1u, abort);
                    if (__any_sync(0xffffffffu, !ok)) {   // warp-uniform before the elected issue
                        fail_here();
                        break;
                    }
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t a_tmem = tmem + kABase + a * kSetCols + s0 * (kSetCols / MT);
                        const uint32_t d_tmem = tmem + kAccBase + s0 * N;
#pragma unroll
                        for (int k = 0; k < KSTEPS; ++k)
#pragma unroll
                            for (int s = 0; s < PW; ++s)
                                umma_mxf4_ts(d_tmem + s * N, a_tmem + s * (kSetCols / MT) + 8u * k,
                                             bdesc + 2u * (h * KSTEPS + k), idesc, tmem + kScaleBase,
                                             tmem + kScaleBase + 16u, (u != pc.u0 || h != 0 || k != 0) ? 1u : 0u);
                        umma_commit(&afree[a]);
                        if (h == SETS - 1) umma_commit(&qfree[q]);
                        if (h == SETS - 1 && u == pc.u1 - 1) umma_commit(acc_full);
                    }
                    __syncwarp();
                }
                if (failed) break;
            }
            ++np;
        }
        if (is) {   // every MMA must finish before TMEM is released
            if (elect_one()) umma_commit(mma_done);
            __syncwarp();
            if (!mbar_drain(mma_done, 0)) failed = true;
        }
    } else if (warp < 6) {
        // ---------------- epilogue
        const uint32_t lane_addr = (quarter * 32u) << 16;
        uint32_t np = 0;
        while (!failed && pit.next(pc, tiles, qtiles, bands, units)) {
            const bool ok = mbar_wait(acc_full, np & 1u, abort);
            if (__any_sync(0xffffffffu, !ok)) {
                fail_here();
                break;
            }
            tc_fence_after();
            const uint32_t z = MT == 4 ? 0u : 2u * (pc.tile & 1u);   // first plane of this CTA
            const uint32_t w0 = (MT == 4 ? pc.tile : pc.tile >> 1) * kUnitWords + 4u * quarter;
#pragma unroll 1
            for (uint32_t n0 = 0; n0 < (uint32_t)N; n0 += 32) {
                uint32_t bits[MT];   // lane n: bit l = parity of lane l's count for query n0 + n
#pragma unroll
                for (int s = 0; s < MT; ++s) {
                    uint32_t v[32];
                    tmem_ld32(tmem + lane_addr + kAccBase + s * N + n0, v);
                    tmem_wait_ld();
                    // operand values 0.5, 1, 2, 2 of planes 0..3 scale the counts; the low bit of the
                    // count under the exponent of 2^23 is its parity
                    const uint32_t plane = z + s;
                    const float inv = plane == 0 ? 2.0f : (plane == 1 ? 1.0f : 0.5f);
#pragma unroll
                    for (int n = 0; n < 32; ++n) {
                        const uint32_t odd = __float_as_uint(__fmaf_rn(__uint_as_float(v[n]), inv, 8388608.0f)) & 1u;
                        const uint32_t b = __ballot_sync(0xffffffffu, odd);
                        if (lane == n) bits[s] = b;
                    }
                }
                if (n0 + 32 == (uint32_t)N) {   // the counts are in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acc_free);
                }
                const uint32_t b = pc.q * N + n0 + static_cast<uint32_t>(lane);
                if (b < B) {
#pragma unroll
                    for (uint32_t wl = 0; wl < 4; ++wl) {
                        uint32_t word = 0;
#pragma unroll
                        for (int s = 0; s < MT; ++s) word |= spread4((bits[s] >> (8u * wl)) & 255u) << (z + s);
                        if (w0 + wl < W && word != 0) atomicXor(out + (uint64_t)b * W + w0 + wl, word);
                    }
                }
            }
            ++np;
        }
    } else if (warp < 14) {
        // ---------------- step 1: nibble transposition.  A warp takes one quad (16 bytes) of all rows.
        // ldmatrix turns 16 x 16 bytes: thread (c = lane / 4, gi = lane % 4) gets byte column c (and c + 8)
        // of four rows of group gi.  Two matrices hold the two halves of four groups of 8 rows, odd
        // groups in the other order, so that the eight row addresses of a phase lie in distinct banks
        // (64-byte swizzled rows).
        const uint32_t group = static_cast<uint32_t>(warp - 6) >> 2;
        const uint32_t v = static_cast<uint32_t>(warp - 6) & 3u;   // words 4v .. 4v + 3
        const uint32_t ul = static_cast<uint32_t>(lane);
        const uint32_t lrow = 8u * ((ul >> 2) & 3u) + (ul & 3u) + 4u * (((ul >> 2) & 1u) ^ (ul >> 4));
        const uint32_t laddr = lrow * 64u + ((v ^ ((lrow >> 1) & 3u)) << 4);
        const uint32_t c = ul >> 2, gi = ul & 3u;
        uint32_t it = 0;
        while (!failed && pit.next(pc, tiles, qtiles, bands, units)) {
            for (uint32_t u = pc.u0; u < pc.u1; ++u, ++it) {
                if ((it & 1u) != group) continue;
                const uint32_t r = it % kRawSlots, x = it % kXSlots;
                bool ok = mbar_wait(&rfull[r], (it / kRawSlots) & 1u, abort);
                ok = ok && mbar_wait(&xfree[x], ((it / kXSlots) & 1u) ^ 1u, abort);
                if (__any_sync(0xffffffffu, !ok)) {
                    fail_here();
                    break;
                }
                const uint32_t src = smem_addr(raw + r * kRawBytes) + laddr;
                uint32_t o[4][8];   // [byte column c, low and high nibble; c + 8, low and high][rows 32 rb ..]
#pragma unroll
                for (uint32_t rb = 0; rb < 8; ++rb) {
                    uint32_t y0, y1, w0, w1;
                    ldmatrix_bytes(src + rb * 2048u, y0, y1, w0, w1);
                    o[0][rb] = (y0 & 0x0F0F0F0Fu) | ((w0 << 4) & 0xF0F0F0F0u);
                    o[1][rb] = ((y0 >> 4) & 0x0F0F0F0Fu) | (w0 & 0xF0F0F0F0u);
                    o[2][rb] = (y1 & 0x0F0F0F0Fu) | ((w1 << 4) & 0xF0F0F0F0u);
                    o[3][rb] = ((y1 >> 4) & 0x0F0F0F0Fu) | (w1 & 0xF0F0F0F0u);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&rfree[r]);
                uint8_t *dst = xt + x * kXBytes;
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) {
                    // TMEM lane 8 w + j, its words 8 gi .. 8 gi + 7
                    const uint32_t w = 4u * v + (c >> 2) + 2u * (k >> 1), j = 2u * (c & 3u) + (k & 1u), L = 8u * w + j;
#pragma unroll
                    for (uint32_t h = 0; h < 2; ++h)
                        *reinterpret_cast<uint4 *>(dst + L * 128u + (((2u * gi + h) ^ x_perm(L)) << 4)) =
                            make_uint4(o[k][4 * h], o[k][4 * h + 1], o[k][4 * h + 2], o[k][4 * h + 3]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&xfull[x]);
            }
        }
    } else {
        // ---------------- step 2: planes into TMEM
        const uint32_t group = static_cast<uint32_t>(warp - 14) >> 2;
        const uint32_t L = quarter * 32u + static_cast<uint32_t>(lane);
        const uint32_t perm = x_perm(L);
        const uint32_t lane_addr = (quarter * 32u) << 16;
        uint32_t it = 0;
        while (!failed && pit.next(pc, tiles, qtiles, bands, units)) {
            const bool upper = MT == 2 && (pc.tile & 1u);   // planes 2 and 3
            for (uint32_t u = pc.u0; u < pc.u1; ++u, ++it) {
                if ((it & 1u) != group) continue;
                const uint32_t x = it % kXSlots;
                bool ok = mbar_wait(&xfull[x], (it / kXSlots) & 1u, abort);
                const uint8_t *src = xt + x * kXBytes + L * 128u;
#pragma unroll
                for (int h = 0; h < SETS; ++h) {
                    const uint32_t is = it * SETS + h, a = is % kASets;
                    ok = ok && mbar_wait(&afree[a], ((is / kASets) & 1u) ^ 1u, abort);
                    if (__any_sync(0xffffffffu, !ok)) {
                        fail_here();
                        break;
                    }
                    tc_fence_after();
                    constexpr int WORDS = 32 / SETS;
                    uint32_t m[WORDS];
#pragma unroll
                    for (int c = 0; c < WORDS / 4; ++c) {
                        const uint4 t =
                            *reinterpret_cast<const uint4 *>(src + (((h * (WORDS / 4) + c) ^ perm) & 7u) * 16u);
                        m[4 * c] = t.x, m[4 * c + 1] = t.y, m[4 * c + 2] = t.z, m[4 * c + 3] = t.w;
                    }
                    const uint32_t a_tmem = tmem + lane_addr + kABase + a * kSetCols;
                    if constexpr (MT == 4) {
                        uint32_t o[32];
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            o[i] = m[i] & 0x11111111u;
                            o[16 + i] = m[i] & 0x22222222u;
                        }
                        tmem_st32(a_tmem, o);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            o[i] = m[i] & 0x44444444u;
                            o[16 + i] = (m[i] >> 1) & 0x44444444u;
                        }
                        tmem_st32(a_tmem + 32u, o);
                    } else {
                        const uint32_t mask = upper ? 0x44444444u : 0x11111111u;
                        uint32_t o[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = m[i] & mask;
                        tmem_st32(a_tmem, o);
                        if (upper) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = (m[i] >> 1) & 0x44444444u;
                        } else {
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = m[i] & 0x22222222u;
                        }
                        tmem_st32(a_tmem + 32u, o);
                    }
                    if (h == SETS - 1) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&xfree[x]);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&afull[a]);
                }
                if (failed) break;
            }
        }
    }

    if (failed) {
        *abort = 1;
        *status = kDevTimeout;
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmem);
    }
}

// Query bits of the rows [row0, row0 + 256 units) as e2m1 ones, in the order that step 1 leaves: word
// 8 i + k of unit u of query b holds the 8 rows of group 4 k + i (rows 256 u + 32 k + 8 i ..), nibble
// 2 t of row t and nibble 2 t + 1 of row 4 + t (odd i: the other way round).  Bits past the last row
// meet zero database rows.
__global__ void __launch_bounds__(256) chor_nibbles_kernel(const uint32_t *__restrict__ Q, uint64_t qw, uint64_t word0,
                                                           uint32_t units, uint32_t *__restrict__ QF) {
    const uint32_t t = blockIdx.x * 256u + threadIdx.x;   // one query word: 4 groups of 8 rows
    if (t >= units * 8u) return;
    const uint32_t b = blockIdx.y;
    const uint64_t k = word0 + t;
    const uint32_t x = k < qw ? Q[(uint64_t)b * qw + k] : 0u;
    uint32_t *dst = QF + ((uint64_t)b * units + (t >> 3)) * 32u + (t & 7u);
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t y = (x >> (8u * i)) & 255u;
        uint32_t first = y & 15u, second = y >> 4;
        if (i & 1u) {
            first = y >> 4;
            second = y & 15u;
        }
        const uint32_t lo = (first * 0x00204081u) & 0x01010101u, hi = (second * 0x00204081u) & 0x01010101u;
        dst[8u * i] = (lo << 1) | (hi << 5);
    }
}

// ------------------------------------------------------------------ host side
cudaError_t prepare_chor_gemm_kernels() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(chor_gemm_kernel<32, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  GCfg<32, 4>::kSmemBytes)) != cudaSuccess)
        return e;
    if ((e = cudaFuncSetAttribute(chor_gemm_kernel<64, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  GCfg<64, 4>::kSmemBytes)) != cudaSuccess)
        return e;
    return cudaFuncSetAttribute(chor_gemm_kernel<128, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                GCfg<128, 2>::kSmemBytes);
}

uint32_t chor_gemm_n(uint32_t B) { return B <= 32 ? 32u : (B <= 64 ? 64u : 128u); }

cudaError_t launch_chor_nibbles(const uint32_t *Q, uint64_t qw, uint32_t B, uint64_t row0, uint32_t units, uint32_t *QF,
                                cudaStream_t stream) {
    chor_nibbles_kernel<<<dim3((units * 8u + 255u) / 256u, B), 256, 0, stream>>>(Q, qw, row0 / 32, units, QF);
    return cudaGetLastError();
}

// Bands of rows: pieces = tiles x bands, dealt to the SMs in turn.  A piece of n units costs about
// n + 6 unit times (its epilogue, 2,000-3,000 cycles, runs beside no MMA of the next piece), so the
// bands minimise waves x (units per band + 6).
static uint32_t chor_bands(uint32_t tiles, uint32_t units, uint32_t sms) {
    uint32_t best = 1;
    uint64_t cost = ~0ull;
    for (uint32_t nb = 1; nb <= units && nb <= 64; ++nb) {
        const uint64_t waves = ((uint64_t)tiles * nb + sms - 1) / sms;
        const uint64_t c = waves * ((units + nb - 1) / nb + 6);
        if (c < cost) {
            cost = c;
            best = nb;
        }
    }
    return best;
}

template <int N, int MT>
static cudaError_t launch_gemm_t(const CUtensorMap &db_map, const CUtensorMap &q_map, uint32_t row0, uint32_t units,
                                 uint32_t W, uint32_t B, uint32_t *out, int num_sms, int *status, cudaStream_t stream) {
    const uint32_t tiles = (W + kUnitWords - 1) / kUnitWords * (4 / MT), qtiles = (B + N - 1) / N;
    const uint32_t bands = chor_bands(tiles * qtiles, units, static_cast<uint32_t>(num_sms));
    const uint64_t pieces = (uint64_t)tiles * qtiles * bands;
    if (pieces >= (1ull << 31)) return cudaErrorInvalidValue;
    const unsigned grid = static_cast<unsigned>(pieces < (uint64_t)num_sms ? pieces : (uint64_t)num_sms);
    chor_gemm_kernel<N, MT><<<grid, kGThreads, GCfg<N, MT>::kSmemBytes, stream>>>(db_map, q_map, row0, units, tiles, qtiles,
                                                                                 bands, W, B, out, status);
    return cudaGetLastError();
}

cudaError_t launch_chor_gemm(const CUtensorMap &db_map, const CUtensorMap &q_map, uint64_t row0, uint32_t units,
                             uint32_t W, uint32_t B, uint32_t *out, int num_sms, int *status, cudaStream_t stream) {
    const uint32_t r0 = static_cast<uint32_t>(row0);
    switch (chor_gemm_n(B)) {
        case 32: return launch_gemm_t<32, 4>(db_map, q_map, r0, units, W, B, out, num_sms, status, stream);
        case 64: return launch_gemm_t<64, 4>(db_map, q_map, r0, units, W, B, out, num_sms, status, stream);
        default: return launch_gemm_t<128, 2>(db_map, q_map, r0, units, W, B, out, num_sms, status, stream);
    }
}

}  // namespace qpadl
