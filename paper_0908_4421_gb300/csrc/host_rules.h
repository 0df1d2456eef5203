// Decisions of the host side that need no GPU: plain C++, so that a test can compile them alone.
#pragma once

#include <cstdint>

namespace imrt {

// Where a caller's array lives.
enum class Memory { kHost, kDevice, kManaged };

// Whether kernels on device `dev` may read and write an array in place: managed memory and the device's own.
// Another GPU's memory is reached only by copies (peer access may be off, and a kernel's access would then
// fault), host memory likewise.
constexpr bool kernels_may_use(Memory where, int owner, int dev) {
    return where == Memory::kManaged || (where == Memory::kDevice && owner == dev);
}

// The beamlet-major build counts each chunk of voxel rows' entries per beamlet in a table of one 32-bit word a
// chunk and beamlet, a temporary of plan creation (serve.py's admission estimate bounds it by the same figures).
constexpr int kTChunkRows = 512;      // rows of a chunk to start with
constexpr int kTChunkRowsMin = 32;
constexpr int64_t kTCountBytes = 256ll << 20;      // most the table may take: chunks double beyond it
constexpr int64_t kTCountFineBytes = 32ll << 20;   // most it may grow to for the sake of smaller chunks

constexpr int64_t count_table_bytes(int32_t m, int32_t n, int rows) {
    return ((int64_t)m + rows - 1) / rows * n * 4;
}

// Rows of a chunk: small enough to keep the GPU's SMs evenly busy (the rows of one chunk are one CTA's work,
// and long rows lie together): halved while there are fewer than eight chunks an SM and the table stays small
// (it is written, scanned and read, and a wide plan has few entries a row to pay for it). Measured on a GB300, count
// + scan + scatter: 24k voxels x 620 beamlets 124 us at 512 rows, 23 us at 32; 305k x 3,140 (61M entries) 2.08 ms at
// 512 rows, 2.03 ms at 128. plan_create, halving without and with the bound on the table: 100k x 20,000 1.85 and
// 1.47 ms (119 and 32 MiB; 1.82 ms at 512 rows by itself), 305k x 28,000 3.53 and 2.73 ms (255 and 64 MiB).
inline int transpose_chunk_rows(int32_t m, int32_t n, int sm_count) {
    int rows = kTChunkRows;
    while (rows > kTChunkRowsMin && ((int64_t)m + rows - 1) / rows < 8 * (int64_t)sm_count &&
           count_table_bytes(m, n, rows / 2) <= kTCountFineBytes)
        rows /= 2;
    while (count_table_bytes(m, n, rows) > kTCountBytes && rows < m) rows *= 2;
    return rows;
}

}  // namespace imrt
