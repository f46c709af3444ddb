// Database compression of the spectrum records (Sec. 5.3, "Database
// Compression Techniques"): the DB entries are sorted and each is stored as
// its difference from the entry before it, so close entries take fewer bits
// and every PIR Response scans fewer bytes.
//
// Layout (the reading this library takes): the entries are 32-bit unsigned
// integers x_0 <= x_1 <= ... <= x_{n-1}; block j (one PIR record, i.e. one
// column of the database) holds entries jE .. jE + E - 1, positions past
// n - 1 repeating x_{n-1}.  A block is stored as its first entry in full (4
// little-endian bytes) followed by its E - 1 differences x_{jE+i} -
// x_{jE+i-1} (mod 2^32), each in w little-endian bytes, w the fewest bytes
// that hold every such difference.  The database is then R' = 4 + w (E - 1)
// rows of digits by C = ceil(n / E) columns, row-major, and the usual LWE
// Response, Recover and hint run on it unchanged.  A client that recovers
// block j decodes it on its own by prefix sums.
//
//   delta_width_kernel   largest within-block difference: four entries per 16-byte
//                        load over the entries in order, a CTA max, one atomic max
//   delta_encode_kernel  a CTA per 128 blocks x 128 positions: four entries of four
//                        blocks per thread, packed into row words in registers and
//                        turned through shared memory into 128-byte row segments;
//                        blocks of up to 80 entries are staged whole instead
//   delta_decode_kernel  one CTA per recovered block: eight entries per thread,
//                        a CTA-wide scan of their sums, 16-byte stores
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "qpadl_pir.h"

namespace {

__device__ __forceinline__ uint32_t entry_at(const uint32_t *__restrict__ x, uint64_t n, uint64_t k) {
    return x[k < n ? k : n - 1];
}

// Largest within-block difference.  Thread t of the grid takes the four entries 4 t .. 4 t + 3, then
// strides; its place in the block advances by a constant, so no iteration divides.  Four independent
// 16-byte loads per thread are in flight; the entry before a thread's four comes from its neighbour
// lane.  HBM-bound: each entry is read once.  2^26 entries: 50 us, a warp striding over one block at a
// time 86; eight loads per thread are no faster.
constexpr int kWidthThreads = 256;
__global__ void __launch_bounds__(kWidthThreads) delta_width_kernel(const uint32_t *__restrict__ x, uint64_t n,
                                                                    uint64_t E, int vec,
                                                                    uint32_t *__restrict__ dmax) {
    const int lane = threadIdx.x & 31;
    const uint64_t stride = 4ull * gridDim.x * kWidthThreads;
    const uint64_t base = 4ull * ((uint64_t)blockIdx.x * kWidthThreads + threadIdx.x);
    const uint64_t step = stride % E;
    uint64_t place = base % E;   // of entry k in its block
    uint32_t m = 0;
    constexpr int U = 4;
    for (uint64_t k0 = base; k0 - 4ull * lane < n; k0 += U * stride) {   // warp-uniform
        uint32_t v[U][4], before[U];
        if (vec && k0 + 4ull * (32 - lane) + (U - 1) * stride <= n) {   // the warp's loads all in range
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint4 w = *reinterpret_cast<const uint4 *>(x + k0 + u * stride);
                v[u][0] = w.x, v[u][1] = w.y, v[u][2] = w.z, v[u][3] = w.w;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) before[u] = lane == 0 && k0 + u > 0 ? x[k0 + u * stride - 1] : 0u;
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t k = k0 + u * stride;
#pragma unroll
                for (int q = 0; q < 4; ++q) v[u][q] = entry_at(x, n, k + q);
                before[u] = lane == 0 && k > 0 ? entry_at(x, n, k - 1) : 0u;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t prev = __shfl_up_sync(0xffffffffu, v[u][3], 1);
            if (lane == 0) prev = before[u];
            uint64_t p = place;
#pragma unroll
            for (int q = 0; q < 4; ++q) {   // entries past n - 1 repeat it: difference 0
                const uint32_t d = p == 0 ? 0u : v[u][q] - prev;
                m = d > m ? d : m;
                prev = v[u][q];
                if (++p == E) p = 0;
            }
            place += step;
            if (place >= E) place -= E;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint32_t other = __shfl_xor_sync(0xffffffffu, m, o);
        m = other > m ? other : m;
    }
    __shared__ uint32_t wm[kWidthThreads / 32];
    if (lane == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kWidthThreads / 32; ++w) m = wm[w] > m ? wm[w] : m;
        if (m) atomicMax(dmax, m);
    }
}

// A CTA writes the rows of 128 consecutive blocks (columns) that hold positions kEncPos y ..
// kEncPos y + 127 (position 0: the four rows of the first entry).  Lane l of a warp takes positions
// 4 l .. 4 l + 3 of four neighbouring columns: four 16-byte loads, 512 contiguous bytes a warp and
// column.  Byte b of the four columns' differences makes one row word; the words are turned through
// shared memory (word index xor lane: no bank conflicts either way) so that a warp writes one row's
// 128 bytes at a time.  HBM-bound: each entry is read once, each digit written once.  2^26 entries in
// blocks of 8192, one byte: 56 us (6.0 TB/s), 117 with the entries staged in shared memory by single
// words; with a range check before each load instead of once per CTA, which makes every load wait for the
// one before it, 150.
constexpr int kEncCols = 128;     // columns per CTA: each database row segment is 128 bytes
constexpr int kEncPos = 128;      // positions per block per CTA
constexpr uint32_t kMaxEncodeEntries = 4194241;   // longest block the encoder takes
constexpr int kEncThreads = 256;
constexpr int kEncQuads = kEncCols / 4 / (kEncThreads / 32);   // column quads per warp

__global__ void __launch_bounds__(kEncThreads) delta_encode_kernel(const uint32_t *__restrict__ x, uint64_t n,
                                                                   uint64_t E, uint32_t w, uint64_t C, int vec,
                                                                   uint8_t *__restrict__ db) {
    __shared__ uint32_t tile[kEncPos * (kEncCols / 4)];   // word of quad c, position p at 32 p + (c ^ (p / 4))
    const uint64_t j0 = (uint64_t)blockIdx.x * kEncCols;
    const uint64_t p0 = (uint64_t)blockIdx.y * kEncPos;
    const uint32_t ncols = static_cast<uint32_t>(C - j0 < (uint64_t)kEncCols ? C - j0 : (uint64_t)kEncCols);
    const uint32_t npos = static_cast<uint32_t>(E - p0 < (uint64_t)kEncPos ? E - p0 : (uint64_t)kEncPos);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t d[kEncQuads][4][4];   // entries, then differences [quad][column][position]
    uint32_t prev[kEncQuads][4];   // lane 0: the entry before its four (none before position 0)
    const bool inside = vec && ncols == (uint32_t)kEncCols && npos == (uint32_t)kEncPos &&
                        (j0 + kEncCols - 1) * E + p0 + kEncPos <= n;
    if (inside) {   // all of a thread's loads go out before the first is used
        const uint32_t *src = x + (j0 + 4u * warp) * E + p0 + 4u * lane;
#pragma unroll
        for (int u = 0; u < kEncQuads; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 q = *reinterpret_cast<const uint4 *>(src + (32u * u + c) * E);
                d[u][c][0] = q.x, d[u][c][1] = q.y, d[u][c][2] = q.z, d[u][c][3] = q.w;
            }
#pragma unroll
        for (int u = 0; u < kEncQuads; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) prev[u][c] = lane == 0 && p0 > 0 ? *(src + (32u * u + c) * E - 1) : 0u;
    } else {
#pragma unroll
        for (int u = 0; u < kEncQuads; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t col = 4u * (warp + 8 * u) + c;
                const uint64_t k = (j0 + col) * E + p0 + 4u * lane;
#pragma unroll
                for (int q = 0; q < 4; ++q) d[u][c][q] = col < ncols ? entry_at(x, n, k + q) : 0u;
                prev[u][c] = col < ncols && lane == 0 && p0 > 0 ? entry_at(x, n, k - 1) : 0u;
            }
    }
#pragma unroll
    for (int u = 0; u < kEncQuads; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t up = __shfl_up_sync(0xffffffffu, d[u][c][3], 1);
            d[u][c][3] -= d[u][c][2];
            d[u][c][2] -= d[u][c][1];
            d[u][c][1] -= d[u][c][0];
            d[u][c][0] -= lane > 0 ? up : prev[u][c];   // position 0: the entry itself
        }
    const bool words = (C % 4 == 0) && ((reinterpret_cast<uintptr_t>(db) & 3u) == 0);
    const uint32_t quad_cols = ncols - (4u * lane < ncols ? 4u * lane : ncols);   // columns of this lane's row word
    for (uint32_t b = 0; b < 4; ++b) {
        if (b >= w && p0 != 0) break;   // bytes past w: only the first entries' rows
        const uint32_t lo = b | ((b + 4) << 4);   // byte b of each of two words
#pragma unroll
        for (int u = 0; u < kEncQuads; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t a = __byte_perm(d[u][0][q], d[u][1][q], lo), c = __byte_perm(d[u][2][q], d[u][3][q], lo);
                tile[(4 * lane + q) * 32 + ((warp + 8 * u) ^ lane)] = __byte_perm(a, c, 0x5410);
            }
        __syncthreads();
        const uint32_t last = b < w ? npos : 1u;
        for (uint32_t p = warp; p < last; p += kEncThreads / 32) {
            const uint32_t v = tile[p * 32 + (lane ^ (p >> 2))];
            const uint64_t pos = p0 + p;
            const uint64_t row = pos == 0 ? b : 4 + (pos - 1) * w + b;
            uint8_t *dst = db + row * C + j0 + 4u * lane;
            if (words) {
                if (quad_cols) *reinterpret_cast<uint32_t *>(dst) = v;   // C % 4 == 0: whole words
            } else {
#pragma unroll
                for (uint32_t c = 0; c < 4; ++c)
                    if (c < quad_cols) dst[c] = static_cast<uint8_t>(v >> (8 * c));
            }
        }
        __syncthreads();
    }
}

// The same for blocks of up to 80 entries, of which the tile above would be mostly positions past the block's
// end: a CTA stages its 128 blocks whole (one contiguous run of 128 E entries) and writes their rows.  Bound by
// the row stores.  2^24 entries, one byte, blocks of 2 / 5 / 16 / 33 / 64 / 80 entries: 84 / 47 / 31 / 41 / 27 /
// 26 us, in 128 x 128 tiles 969 / 399 / 132 / 73 / 41 / 35; 81 entries 37 in tiles, 90 entries 41 staged, 35 in tiles.
constexpr uint32_t kShortEntries = 80;
template <uint32_t COLS>   // blocks per CTA: 128, or 32 where that would leave SMs without a CTA
__global__ void __launch_bounds__(kEncThreads) delta_encode_short_kernel(const uint32_t *__restrict__ x, uint64_t n,
                                                                         uint32_t E, uint32_t w, uint64_t C,
                                                                         uint8_t *__restrict__ db) {
    extern __shared__ uint32_t ent[];   // [COLS][ld]; an odd stride puts neighbouring columns in distinct banks
    const uint32_t ld = E | 1u;
    const uint64_t j0 = (uint64_t)blockIdx.x * COLS;
    const uint32_t ncols = static_cast<uint32_t>(C - j0 < (uint64_t)COLS ? C - j0 : (uint64_t)COLS);
    const uint64_t k0 = j0 * E;
    if (k0 + (uint64_t)ncols * E <= n) {   // one check: the loads do not wait for one another
#pragma unroll 4
        for (uint32_t f = threadIdx.x; f < ncols * E; f += kEncThreads) {
            const uint32_t c = f / E;
            ent[c * ld + f - c * E] = x[k0 + f];
        }
    } else {
        for (uint32_t f = threadIdx.x; f < ncols * E; f += kEncThreads) {
            const uint32_t c = f / E;
            ent[c * ld + f - c * E] = entry_at(x, n, k0 + f);
        }
    }
    __syncthreads();
    // row r < 4: byte r of the first entries; row 4 + (i - 1) w + b: byte b of the differences at position i
    const uint32_t rows = (E - 1) * w;
    uint8_t *diffs = db + 4 * C + j0;
    db += j0;
    if (C % 4 == 0 && (reinterpret_cast<uintptr_t>(db) & 3u) == 0) {   // four columns in one store
        constexpr uint32_t kQuads = COLS / 4;
        for (uint32_t t = threadIdx.x; t < rows * kQuads; t += kEncThreads) {
            const uint32_t r = t / kQuads, c = 4 * (t % kQuads);
            if (c >= ncols) continue;   // C % 4 == 0: whole quads
            const uint32_t i = r / w, sh = 8u * (r - i * w);
            uint32_t v = 0;
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) v |= (((ent[(c + k) * ld + i + 1] - ent[(c + k) * ld + i]) >> sh) & 255u) << (8u * k);
            *reinterpret_cast<uint32_t *>(diffs + r * C + c) = v;
        }
    } else {
        for (uint32_t t = threadIdx.x; t < rows * COLS; t += kEncThreads) {
            const uint32_t r = t / COLS, c = t % COLS, i = r / w;
            if (c < ncols) diffs[r * C + c] = static_cast<uint8_t>((ent[c * ld + i + 1] - ent[c * ld + i]) >> (8u * (r - i * w)));
        }
    }
    for (uint32_t t = threadIdx.x; t < 4 * COLS; t += kEncThreads) {   // the first entry of each block in full
        const uint32_t r = t / COLS, c = t % COLS;
        if (c < ncols) db[r * C + c] = static_cast<uint8_t>(ent[c * ld] >> (8u * r));
    }
}

// The same for few blocks (columns): their rows are so short that the database is written as one run of bytes, four to
// a thread, each from two neighbouring entries.  The tile above would be mostly columns past the last one: one block of
// 2^20 entries, one byte, 138 us in tiles, 8 so.
// A byte costs it the same whatever the rest, so wider digits leave it earlier: 2^24 entries, 25 blocks, one and four bytes
// 94 and 220 us in tiles, 45 and 175 so; 41 blocks 60 and 136.
constexpr uint64_t few_blocks(uint32_t w) { return w == 1 ? 40 : (w == 2 ? 32 : 28); }
__global__ void __launch_bounds__(kEncThreads) delta_encode_few_kernel(const uint32_t *__restrict__ x, uint64_t n, uint32_t E,
                                                                       uint32_t w, uint32_t C, uint8_t *__restrict__ db) {
    const uint32_t total = (4 + w * (E - 1)) * C;   // at most 28 x 4 x 2^22 bytes
    const uint32_t at = 4 * (blockIdx.x * kEncThreads + threadIdx.x);
    if (at >= total) return;
    uint32_t row = at / C, c = at - row * C, v = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
        const uint64_t first = (uint64_t)c * E;
        uint32_t d;
        if (row < 4) {
            d = entry_at(x, n, first) >> (8 * row);
        } else {
            const uint32_t i = (row - 4) / w, b = row - 4 - i * w;   // difference i + 1
            d = (entry_at(x, n, first + i + 1) - entry_at(x, n, first + i)) >> (8 * b);
        }
        v |= (d & 255u) << (8 * k);
        if (++c == C) {
            c = 0;
            ++row;
        }
    }
    if (at + 4 <= total && (reinterpret_cast<uintptr_t>(db) & 3u) == 0) {
        *reinterpret_cast<uint32_t *>(db + at) = v;
    } else {
        for (uint32_t k = 0; k < 4 && at + k < total; ++k) db[at + k] = static_cast<uint8_t>(v >> (8 * k));
    }
}

// Block b: digits b * Rp .. (4-byte first entry, then E - 1 differences of W bytes) -> out b * E ..
// Thread t takes positions 8 t .. 8 t + 7 of a run of 8 blockDim.x (its digits are independent loads of
// adjacent bytes), a two-level shuffle scan gives the sum before them, and the runs of a longer
// block follow one another with the last sum carried.  64 blocks of 8192: 4.2 us, 12.1 with each thread
// adding up a run of 32 bytes of its own.  A CTA has as many warps as its block of entries needs, at most 32:
// 4096 blocks of 2048 / 4096 entries 12 / 25 us, 32 / 39 with 32 warps for each; 2^18 blocks of 16 135, 1644.
constexpr int kDecodeThreads = 1024;   // at most
constexpr int kDecodeRun = 8;

template <int W, bool FULL>   // FULL: 32 warps
__global__ void __launch_bounds__(kDecodeThreads) delta_decode_kernel(const uint8_t *__restrict__ digits, uint64_t E,
                                                                      uint64_t Rp, int vec,
                                                                      uint32_t *__restrict__ out) {
    __shared__ uint32_t part[2][kDecodeThreads / 32];
    const uint8_t *dg = digits + (uint64_t)blockIdx.x * Rp;
    uint32_t *o = out + (uint64_t)blockIdx.x * E;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t threads = FULL ? kDecodeThreads : blockDim.x;
    uint32_t carry = 0;
    int turn = 0;
    for (uint64_t e0 = 0; e0 < E; e0 += threads * kDecodeRun, turn ^= 1) {
        const uint64_t t0 = e0 + (uint64_t)threadIdx.x * kDecodeRun;
        uint32_t v[kDecodeRun];
#pragma unroll
        for (int i = 0; i < kDecodeRun; ++i) {
            const uint64_t t = t0 + i;
            v[i] = 0u;
            if (t < E) {
                if (t == 0) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) v[i] |= static_cast<uint32_t>(dg[k]) << (8 * k);
                } else {
                    const uint8_t *p = dg + 4 + (t - 1) * W;
#pragma unroll
                    for (int k = 0; k < W; ++k) v[i] |= static_cast<uint32_t>(p[k]) << (8 * k);
                }
            }
        }
#pragma unroll
        for (int i = 1; i < kDecodeRun; ++i) v[i] += v[i - 1];
        uint32_t sum = v[kDecodeRun - 1];   // inclusive over the warp, then over the CTA
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t a = __shfl_up_sync(0xffffffffu, sum, off);
            if (lane >= off) sum += a;
        }
        if (lane == 31) part[turn][warp] = sum;
        __syncthreads();   // the other buffer's readers are done before this one is written again
        uint32_t ps = FULL || lane < static_cast<int>(threads >> 5) ? part[turn][lane] : 0u;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t a = __shfl_up_sync(0xffffffffu, ps, off);
            if (lane >= off) ps += a;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, ps, 31);
        const uint32_t warps_before = __shfl_sync(0xffffffffu, ps, (warp + 31) & 31);   // unused in warp 0
        const uint32_t before = carry + (warp ? warps_before : 0u) + sum - v[kDecodeRun - 1];
        carry += total;
        if (vec && t0 + kDecodeRun <= E) {
#pragma unroll
            for (int i = 0; i < kDecodeRun; i += 4)
                *reinterpret_cast<uint4 *>(o + t0 + i) =
                    make_uint4(before + v[i], before + v[i + 1], before + v[i + 2], before + v[i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < kDecodeRun; ++i)
                if (t0 + i < E) o[t0 + i] = before + v[i];
        }
    }
}

// The width reduction's result word: one per device, used under g_width_mu for
// the whole (synchronous) call, so the call allocates nothing.
__device__ uint32_t g_width_word;
std::mutex g_width_mu;

int num_sms_current() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    return sms;
}

bool delta_shape_ok(uint64_t n, uint64_t E, uint32_t w) {
    if (n == 0 || E == 0 || w < 1 || w > 4) return false;
    const uint64_t C = (n + E - 1) / E;
    const uint64_t Rp = 4 + (uint64_t)w * (E - 1);
    return C < (1ull << 31) && Rp < (1ull << 31);
}

}  // namespace

extern "C" {

int qpadl_pir_delta_width(const uint32_t *entries_dev, uint64_t n, uint32_t E, uint32_t *w_out,
                          qpadl_stream_t stream) {
    if (!entries_dev || !w_out || !delta_shape_ok(n, E, 4)) return QPADL_EINVAL;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int sms = num_sms_current();
    if (sms <= 0) return QPADL_ECUDA;
    const int vec = (reinterpret_cast<uintptr_t>(entries_dev) & 15u) == 0;
    const uint64_t want = (n + 16 * kWidthThreads - 1) / (16 * kWidthThreads);   // 16 entries per thread and pass
    const unsigned grid = static_cast<unsigned>(want < (uint64_t)sms * 4 ? want : (uint64_t)sms * 4);
    std::lock_guard<std::mutex> guard(g_width_mu);
    uint32_t *dmax = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void **>(&dmax), g_width_word) != cudaSuccess) return QPADL_ECUDA;
    uint32_t h = 0;
    bool ok = cudaMemsetAsync(dmax, 0, sizeof(uint32_t), s) == cudaSuccess;
    if (ok) {
        delta_width_kernel<<<grid, kWidthThreads, 0, s>>>(entries_dev, n, E, vec, dmax);
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = ok && cudaMemcpyAsync(&h, dmax, sizeof(uint32_t), cudaMemcpyDeviceToHost, s) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(s) == cudaSuccess;
    if (!ok) return QPADL_ECUDA;
    uint32_t w = 1;
    while (w < 4 && h >= (1u << (8u * w))) ++w;
    *w_out = w;
    return QPADL_OK;
}

int qpadl_pir_delta_encode(const uint32_t *entries_dev, uint64_t n, uint32_t E, uint32_t w, uint8_t *db_dev,
                           qpadl_stream_t stream) {
    if (!entries_dev || !db_dev || !delta_shape_ok(n, E, w)) return QPADL_EINVAL;
    const uint64_t C = (n + E - 1) / E;
    if (E > kMaxEncodeEntries) return QPADL_EINVAL;
    const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (E <= kShortEntries) {
        const int sms = num_sms_current();
        if (sms <= 0) return QPADL_ECUDA;
        const uint32_t cols = C > (uint64_t)sms * kEncCols ? kEncCols : 32u;
        const auto kernel = cols == 32u ? delta_encode_short_kernel<32> : delta_encode_short_kernel<kEncCols>;
        kernel<<<static_cast<unsigned>((C + cols - 1) / cols), kEncThreads, cols * (E | 1u) * 4, s>>>(entries_dev, n, E, w, C,
                                                                                                   db_dev);
        return cudaGetLastError() == cudaSuccess ? QPADL_OK : QPADL_ECUDA;
    }
    if (C <= few_blocks(w)) {
        const uint64_t threads = ((4 + (uint64_t)w * (E - 1)) * C + 3) / 4;
        delta_encode_few_kernel<<<static_cast<unsigned>((threads + kEncThreads - 1) / kEncThreads), kEncThreads, 0, s>>>(
            entries_dev, n, E, w, static_cast<uint32_t>(C), db_dev);
        return cudaGetLastError() == cudaSuccess ? QPADL_OK : QPADL_ECUDA;
    }
    const int vec = (E % 4 == 0) && (reinterpret_cast<uintptr_t>(entries_dev) & 15u) == 0;
    const dim3 grid(static_cast<unsigned>((C + kEncCols - 1) / kEncCols),
                    static_cast<unsigned>((E + kEncPos - 1) / kEncPos));
    delta_encode_kernel<<<grid, kEncThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(entries_dev, n, E, w, C, vec,
                                                                                          db_dev);
    return cudaGetLastError() == cudaSuccess ? QPADL_OK : QPADL_ECUDA;
}

int qpadl_pir_delta_decode(const uint8_t *digits_dev, uint32_t B, uint32_t E, uint32_t w, uint32_t *entries_dev,
                           qpadl_stream_t stream) {
    if (!digits_dev || !entries_dev || B == 0 || !delta_shape_ok(E, E, w)) return QPADL_EINVAL;
    const uint64_t Rp = 4 + (uint64_t)w * (E - 1);
    const int vec = (E % 4 == 0) && (reinterpret_cast<uintptr_t>(entries_dev) & 15u) == 0;
    const uint64_t want = ((uint64_t)E + 32 * kDecodeRun - 1) / (32 * kDecodeRun) * 32;   // whole warps for one run
    const unsigned threads = static_cast<unsigned>(want < kDecodeThreads ? want : kDecodeThreads);
    auto launch = [&](auto full, auto part) {
        const auto kernel = threads == kDecodeThreads ? full : part;
        kernel<<<B, threads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(digits_dev, E, Rp, vec, entries_dev);
    };
    switch (w) {
        case 1: launch(delta_decode_kernel<1, true>, delta_decode_kernel<1, false>); break;
        case 2: launch(delta_decode_kernel<2, true>, delta_decode_kernel<2, false>); break;
        case 3: launch(delta_decode_kernel<3, true>, delta_decode_kernel<3, false>); break;
        default: launch(delta_decode_kernel<4, true>, delta_decode_kernel<4, false>); break;
    }
    return cudaGetLastError() == cudaSuccess ? QPADL_OK : QPADL_ECUDA;
}

}  // extern "C"
