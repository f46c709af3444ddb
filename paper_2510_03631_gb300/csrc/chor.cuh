// Launch interface of the Chor-style GF(2) Response kernels (chor.cu).
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

namespace qpadl {

constexpr uint32_t kChorMaxBatch = 256;   // queries per launch; larger batches run in chunks

cudaError_t prepare_chor_kernels();

// Tile width (words), band height (rows), TMA box width (words) and QT words
// per row that a launch for B queries in scan form `form` (0..3: bit 1 = 8 words
// per thread, bit 0 = predicated XOR) uses; false if B is 0 or > kChorMaxBatch.
bool chor_launch_shape(uint32_t B, int form, uint32_t *tw, uint32_t *rb, uint32_t *box_words, uint32_t *qtw);

// Q (B x qw words) -> QT (r x qtw words): bit j of QT[i][g] = bit i of query 32 g + j.
cudaError_t launch_chor_transpose(const uint32_t *Q, uint64_t qw, uint32_t B, uint64_t r, uint32_t qtw, uint32_t *QT,
                                  int num_sms, cudaStream_t stream);

// out (B x W words, zeroed by the caller) ^= the GF(2) responses; db_map covers
// the database {W, r} words with box {box_words, rb}, qt_map QT {qtw, r} with box {qtw, rb}.
cudaError_t launch_chor_answer(const CUtensorMap &db_map, const CUtensorMap &qt_map, uint64_t r, uint32_t W,
                               uint32_t B, uint32_t qtw, uint32_t *out, int num_sms, int *status,
                               cudaStream_t stream, int form);

// Four-Russians path (few rows of long records): box shape of its database map.
constexpr uint32_t kChorM4TileWords = 64;
constexpr uint32_t kChorM4BandRows = 64;

// Q (B x qw words) -> QS (qw x 256 words): word k of query b at QS[k * 256 + b];
// the buffer must hold roundup(qw, 2) x 256 words (a band reads two query words).
cudaError_t launch_chor_words(const uint32_t *Q, uint64_t qw, uint32_t B, uint64_t r, uint32_t *QS, int num_sms,
                              cudaStream_t stream);

// out (B x W words, zeroed by the caller) ^= the responses of B <= 256 queries;
// db_map covers the database {W, r} words with box {64, 64}.
cudaError_t launch_chor_m4rm(const CUtensorMap &db_map, const uint32_t *QS, uint64_t r, uint32_t W, uint32_t B,
                             uint32_t *out, int num_sms, int *status, cudaStream_t stream);

// Tensor-core path (chor_gemm.cu): units of 256 rows x 16 words, tiles of up to 128 queries.
constexpr uint32_t kChorGemmUnitRows = 256;
constexpr uint32_t kChorGemmUnitWords = 16;
constexpr uint32_t kChorGemmTile = 128;
// Rows per launch: bounds the expanded queries and, far below 2^22, the counts.
constexpr uint64_t kChorGemmRows = 1ull << 18;
// Queries per launch over `units` units (128 bytes of expanded bits per query and unit): up to eight tiles in 256 KiB, which
// cudaMalloc mostly gives out of memory it holds (else a setup takes 100 us instead of 20), but at least two, or one
// where two are more than 16 MiB.
constexpr uint32_t chor_gemm_group(uint32_t units) {
    const uint32_t tiles = (256u << 10) / (128u * kChorGemmTile * units);
    return kChorGemmTile * (tiles > 8 ? 8 : (tiles >= 2 ? tiles : (units <= 512 ? 2 : 1)));
}
constexpr uint64_t chor_gemm_scratch(uint32_t units) { return 128ull * chor_gemm_group(units) * units; }
// Up to this many units x column tiles, what a batch leaves for its last tile shares the launch of the others even when
// it is narrow: a launch of its own costs about 9 us, 128 instead of 64 columns of MMAs 2.2 ns per unit and tile.
constexpr uint64_t kChorGemmSmall = 4096;

cudaError_t prepare_chor_gemm_kernels();
// Query rows of a tile (32, 64 or 128) for B queries: the box height of q_map.
uint32_t chor_gemm_n(uint32_t B);

// Q (B x qw words) -> QF: the bits of rows [row0, row0 + 256 units) as e2m1 ones, B rows of
// 128 * units bytes; row0 a multiple of 32.
cudaError_t launch_chor_nibbles(const uint32_t *Q, uint64_t qw, uint32_t B, uint64_t row0, uint32_t units, uint32_t *QF,
                                cudaStream_t stream);

// out (B x W words, zeroed by the caller) ^= the responses of B queries over the rows
// [row0, row0 + 256 units); db_map covers the database {W, r} words with box {16, 256} and 64-byte swizzle, q_map QF
// {128 units, B} bytes with box {128, chor_gemm_n(B)} and 128-byte swizzle.
cudaError_t launch_chor_gemm(const CUtensorMap &db_map, const CUtensorMap &q_map, uint64_t row0, uint32_t units,
                             uint32_t W, uint32_t B, uint32_t *out, int num_sms, int *status, cudaStream_t stream);

}  // namespace qpadl
