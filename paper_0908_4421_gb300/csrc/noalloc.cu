// Allocation-free evaluation of the dose and the objective from a caller's device CSR.
//
// Some callers cannot allocate device memory at the moment they need an evaluation:
// controllers in a treatment-delivery loop whose device memory is reserved once at
// start-up and may not grow afterwards, host frameworks that give this library a fixed
// device budget and own every allocation themselves, and processes in which another
// component already holds nearly all of the device's memory. For them,
// imrt_eval_csr_noalloc keeps its scratch (per-tile objective partials, structure voxel
// counts, a completion counter, an input-error flag and the final objective) in one
// file-scope __device__ array instead of asking the runtime for memory. The caller passes
// the inputs and the output buffers.
//
// The array is created when the library is loaded and every GPU that loads the library
// holds it (about 129 KiB) until the process exits. All calls on a device share it and
// it keeps the last call's contents: each call clears the parts that must start at zero,
// and calls whose work overlaps on the GPU (different streams, or different host
// threads) race on it and must be serialised by the caller. Each call waits for its
// stream and copies the objective into host memory before it returns.
//
// The computation is the forward evaluation of the optimiser (the dose z = D x and the
// objective of the one-sided quadratic penalties with per-structure thresholds, each
// term scaled by w / |V_s|) done directly on the CSR rows: one warp per voxel row, a
// fixed shuffle tree per row, FP64 objective partials per tile of rows summed in tile order
// by the last block to finish, so the result does not depend on scheduling. The kernel
// reads only inside the caller's arrays: a row whose offsets leave [0, nnz] or decrease,
// and an entry whose beamlet index is outside [0, n), are skipped and flagged, and the
// call then returns IMRT_EINVAL.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>

#include "../../include/imrt.h"
#include "imrt_internal.cuh"
#include "ptx.cuh"

namespace {

constexpr int kNaThreads = 256;                        // 8 warps per block
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaBlocksPerSm = 4;                 // resident blocks
constexpr int kNaUnit = 32;                            // voxel rows of a unit: one per lane of the epilogue
constexpr int kNaRows = kNaUnit / kNaWarps;            // of them per warp
constexpr int kNaMaxTiles = 16384;                     // objective partials
constexpr int kNaMaxTileRows = 1024;                   // => at most 16,777,216 voxels
constexpr int64_t kNaMaxVoxels = (int64_t)kNaMaxTileRows * kNaMaxTiles;
constexpr int kNaMaxStruct = 8;
constexpr int kNaMaxDevices = 64;
constexpr int kNaCountBlocks = 32;

// What the host reads back, in one copy.
struct NaResult {
    double G;                       // the objective of the last call
    int32_t bad;                    // input errors: 1 row offsets, 2 beamlet index
    int32_t pad;
};

struct NaScratch {
    double partial[kNaMaxTiles];    // per-tile objective partials
    NaResult res;                   // `bad` cleared by every call
    __align__(16) int32_t counts[kNaCountBlocks][kNaMaxStruct];  // structure voxel counts per counting block
    int32_t next;                   // tiles taken in the current launch (cleared by every call)
    int32_t ticket;                 // blocks finished in the current launch (cleared by every call)
    int32_t pad[6];
};

static __device__ __align__(256) NaScratch g_na_scratch;

struct NaTerms {
    int32_t S;
    float Tu[kNaMaxStruct], To[kNaMaxStruct];  // NaN: no such term
    float wu[kNaMaxStruct], wo[kNaMaxStruct];
};

// Structure voxel counts, one set per block (every block writes its own, so nothing has to be
// cleared first), and the words of the scratch that k_na_eval needs at zero. A thread counts
// eight structures of up to 255 mask bytes in the bytes of two words (bit t of a mask byte is
// spread to byte t), so the loop has no atomics. 32 blocks, so that one lane a block reads them back in one
// round trip; the evaluation waits for them, which the largest sizes notice (1M voxels with 4 entries each: a
// call 572 -> 253 us with both kernels rewritten, 16.7M: 7.17 -> 3.88 ms, of which the counts 0.18 ms).
__global__ void __launch_bounds__(kNaThreads) k_na_counts(const uint8_t* __restrict__ mask, int32_t m, NaScratch* s) {
    __shared__ int32_t local[kNaMaxStruct];
    imrt::pdl_launch_dependents();  // k_na_eval reads what this writes after its own wait
    if (threadIdx.x < kNaMaxStruct) local[threadIdx.x] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        s->res.bad = 0;
        s->next = 0;
        s->ticket = 0;
    }
    __syncthreads();
    int32_t n[kNaMaxStruct];
#pragma unroll
    for (int t = 0; t < kNaMaxStruct; ++t) n[t] = 0;
    const int64_t step = (int64_t)gridDim.x * kNaThreads;
    int64_t j = (int64_t)blockIdx.x * kNaThreads + threadIdx.x;
    while (j < m) {
        uint32_t lo = 0, hi = 0;  // structures 0..3 and 4..7, a byte each
        constexpr int kU = 8;
        for (int k = 0; k < 248 && j < m; k += kU) {
            uint32_t b[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) b[u] = j + u * step < m ? mask[j + u * step] : 0u;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                lo += ((b[u] & 15u) * 0x00204081u) & 0x01010101u;
                hi += ((b[u] >> 4) * 0x00204081u) & 0x01010101u;
            }
            j += kU * step;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            n[t] += (int)((lo >> (8 * t)) & 0xffu);
            n[4 + t] += (int)((hi >> (8 * t)) & 0xffu);
        }
    }
#pragma unroll
    for (int t = 0; t < kNaMaxStruct; ++t) {
        const int w = __reduce_add_sync(0xffffffffu, n[t]);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&local[t], w);
    }
    __syncthreads();
    if (threadIdx.x < kNaMaxStruct) s->counts[blockIdx.x][threadIdx.x] = local[threadIdx.x];
}

// The terms with their coefficients c = w / |V_s| (Eq. (1)).
struct NaCoefs {
    float Tu[kNaMaxStruct], To[kNaMaxStruct];
    double cu[kNaMaxStruct], co[kNaMaxStruct];
    uint32_t has_u, has_o;  // bit t: structure t has an under / over term
};

// Warp 0 of a block; the caller has a block barrier before the first use.
__device__ __forceinline__ void na_coefs(NaCoefs& C, const NaTerms& terms, const int32_t (*counts)[kNaMaxStruct],
                                         int count_blocks) {
    if (threadIdx.x >= 32) return;
    const int t = threadIdx.x;
    // lane b holds counting block b's counts (one round trip), summed over the warp
    static_assert(kNaCountBlocks <= 32 && kNaMaxStruct == 8, "one lane a block, two 16-byte loads");
    int4 lo = make_int4(0, 0, 0, 0), hi = lo;
    if (t < count_blocks) {
        lo = __ldcg(reinterpret_cast<const int4*>(counts[t]));
        hi = __ldcg(reinterpret_cast<const int4*>(counts[t]) + 1);
    }
    const int part[kNaMaxStruct] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < kNaMaxStruct; ++k) {
        const int c = __reduce_add_sync(0xffffffffu, part[k]);
        if (t == k) cnt = c;
    }
    // lane k: the under-dose term of structure k, lane 8 + k its over-dose term (one FP64 division each)
    const int k = t & 7;
    const bool under = t < 8;
    cnt = __shfl_sync(0xffffffffu, cnt, k);
    const float T = under ? terms.Tu[k] : terms.To[k], w = under ? terms.wu[k] : terms.wo[k];
    const bool has = t < 16 && k < terms.S && !isnan(T) && w != 0.0f && cnt > 0;
    if (t < 16) {
        (under ? C.Tu : C.To)[k] = T;
        (under ? C.cu : C.co)[k] = has ? (double)w / (double)cnt : 0.0;
    }
    const uint32_t b = __ballot_sync(0xffffffffu, has);
    if (t == 0) {
        C.has_u = b & 0xffu;
        C.has_o = b >> 8 & 0xffu;
    }
}

// F_j at dose z. FP64 arithmetic runs at a small fraction of the FP32 rate here (compares and
// conversions too), so only a violated term of one of the voxel's own structures uses it.
__device__ __forceinline__ double na_penalty(float z, uint32_t bits, const NaCoefs& C) {
    double F = 0.0;
    bits &= C.has_u | C.has_o;
    while (bits) {
        const int t = __ffs((int)bits) - 1;
        bits &= bits - 1;
        if ((C.has_u >> t) & 1u) {
            const float e = C.Tu[t] - z;
            if (e > 0.0f) F += C.cu[t] * ((double)e * (double)e);
        }
        if ((C.has_o >> t) & 1u) {
            const float e = z - C.To[t];
            if (e > 0.0f) F += C.co[t] * ((double)e * (double)e);
        }
    }
    return isfinite(z) ? F : __longlong_as_double(0x7ff8000000000000LL);
}

__device__ __forceinline__ double na_warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// z = D x and the objective partials. Meant to be bound by HBM (8 bytes an entry, no reuse); what limits
// it is the latency of a row's rounds, so it keeps many rows and bytes in flight and the work even over
// rows of very uneven length (0 to n entries, long rows next to each other, and as many short ones):
//  * persistent blocks take tiles of consecutive rows from a counter, two tiles ahead; a unit of 32
//    rows is shared by the block's 8 warps, row k to warp k mod 8, so neighbouring long rows spread over
//    the block and the tiles over the chip. The row bounds of the next unit are loaded while the
//    current one streams;
//  * a lane keeps two rounds of 6 columns and 6 values: the next round of its row is in flight while the
//    gathers of x of the current one are (coalesced 4-byte loads: rows start on any entry, and
//    consecutive entries of a row gather neighbouring x);
//  * the penalties of a unit are evaluated one row per lane by one warp, from the row sums in shared
//    memory (FP64 arithmetic is scarce: one lane doing a warp's rows in turn was a serial chain).
// Measured on a GB300, a call: 61M entries in 305k rows 1703 -> 151 us (3.3 TB/s), 0.57M in 44k rows
// 253 -> 42 us, against blocks of 1024 consecutive rows whose warps took 128 rows in series. Tried and
// slower at 61M entries: single rounds of 8 to 16 loads (165-204 us), two rounds of 4, 5 or 8 (158-171 us),
// a cp.async ring per warp over equal shares of the entries (163-202 us: a row's own cost, not its entries,
// sets the balance), 16-byte loads (169-175 us), L2 prefetch of the next unit (209 us).
__global__ void __launch_bounds__(kNaThreads, kNaBlocksPerSm)
    k_na_eval(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, const float* __restrict__ val,
              int32_t m, int32_t n, int64_t nnz, const uint8_t* __restrict__ mask, const NaTerms terms,
              const float* __restrict__ x, float* __restrict__ z, int32_t tile_rows, int32_t n_tiles,
              int32_t count_blocks, NaScratch* s) {
    __shared__ NaCoefs C;
    __shared__ double wsum[kNaWarps];
    __shared__ float zt[2][kNaUnit];
    __shared__ int s_tile[2];
    __shared__ int is_last;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    // The block's units in order: the 32-row units of its tiles. A tile's first is its index.
    int tile = blockIdx.x;
    int rb = tile * tile_rows, r1 = min(m, rb + tile_rows);  // tile_rows * n_tiles < m + 1024: no overflow
    // the bounds of this warp's rows rb + wib + 8 k: lane k holds row k's
    int64_t la = 0, lb = 0;
    if (lane < kNaRows && rb + wib + kNaWarps * lane < r1) {
        la = row_ptr[rb + wib + kNaWarps * lane];
        lb = row_ptr[rb + wib + kNaWarps * lane + 1];
    }
    int bad = 0;
    if (blockIdx.x == 0 && tid == 0 && (row_ptr[0] != 0 || row_ptr[m] != nnz)) bad |= 1;
    imrt::pdl_wait();  // the counts and the cleared words
    na_coefs(C, terms, s->counts, count_blocks);  // (first used after the first unit's barrier)
    int next_tile = (int)(blockIdx.x + gridDim.x), tb = 0, buf = 0;  // later tiles come from the counter
    uint32_t most = 0;  // the largest beamlet index read
    double F = 0.0;     // warp 0: this lane's rows of the tile
    const uint32_t n1 = (uint32_t)n - 1u;
    // x at a column index; one outside [0, n) is noted (and its entry left out of the sum). No branch, so
    // a round's gathers are all in flight together.
    auto x_at = [&](int32_t c) {
        most = max(most, (uint32_t)c);
        return __ldg(x + min((uint32_t)c, n1));
    };
    while (tile < n_tiles) {
        const bool ends = rb + kNaUnit >= r1;  // the tile's last unit
        if (ends && tid == 0) s_tile[tb ^ 1] = 2 * (int)gridDim.x + atomicAdd(&s->next, 1);
        // the next unit, and the bounds of its rows
        const int n_tile = ends ? next_tile : tile;
        int n_rb = rb + kNaUnit, n_r1 = r1;
        if (ends) {
            n_rb = n_tile < n_tiles ? n_tile * tile_rows : 0;
            n_r1 = n_tile < n_tiles ? min(m, n_rb + tile_rows) : 0;
        }
        int64_t na = 0, nb = 0;
        if (lane < kNaRows && n_rb + wib + kNaWarps * lane < n_r1) {
            na = row_ptr[n_rb + wib + kNaWarps * lane];
            nb = row_ptr[n_rb + wib + kNaWarps * lane + 1];
        }
        if (la < 0 || lb < la || lb > nnz) {  // malformed offsets: read nothing of this row
            bad |= 1;
            la = lb = 0;
        }
        float acc[kNaRows];
        constexpr int kU = 6;  // columns and values in flight per lane and stage
        struct Round {
            int32_t c[kU];
            float v[kU];
        };
        // entries i, i + 32, ... of a row of `len` entries starting at c0 / v0
        auto load = [&](Round& q, const int32_t* c0, const float* v0, int i, int len) {
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool in = i + 32 * u < len;
                q.c[u] = in ? __ldcs(c0 + i + 32 * u) : 0;
                q.v[u] = in ? __ldcs(v0 + i + 32 * u) : 0.0f;
            }
        };
        auto use = [&](const Round& q, int i, int len, float& sum) {
            float xv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) xv[u] = x_at(q.c[u]);
#pragma unroll
            for (int u = 0; u < kU; ++u) sum = i + 32 * u < len && (uint32_t)q.c[u] <= n1 ? fmaf(q.v[u], xv[u], sum) : sum;
        };
#pragma unroll
        for (int k = 0; k < kNaRows; ++k) {
            acc[k] = 0.0f;
            int64_t a = __shfl_sync(0xffffffffu, la, k);
            const int64_t b = __shfl_sync(0xffffffffu, lb, k);
            while (a < b) {  // (once, but for rows longer than an int)
                const int len = (int)min(b - a, (int64_t)1 << 30);
                const int32_t* c0 = col + a;
                const float* v0 = val + a;
                a += len;
                Round p, q;
                int i = lane;
                load(p, c0, v0, i, len);
                while (true) {
                    const int j = i + 32 * kU;
                    if (j - lane >= len) {
                        use(p, i, len, acc[k]);
                        break;
                    }
                    load(q, c0, v0, j, len);
                    use(p, i, len, acc[k]);
                    i = j + 32 * kU;
                    if (i - lane >= len) {
                        use(q, j, len, acc[k]);
                        break;
                    }
                    load(p, c0, v0, i, len);
                    use(q, j, len, acc[k]);
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < kNaRows; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        }
#pragma unroll
        for (int k = 0; k < kNaRows; ++k)
            if (lane == k) zt[buf][wib + kNaWarps * k] = acc[k];
        __syncthreads();  // the unit's row sums (the other buffer is free after the barrier before)
        const int j = rb + lane;
        if (wib == 0 && j < r1) {
            const float d = zt[buf][lane];
            if (z) z[j] = d;
            const uint32_t bits = mask[j];
            F += na_penalty(d, bits, C);
        }
        buf ^= 1;
        if (ends) {
            if (wib == 0) {
                F = na_warp_sum(F);
                if (lane == 0) s->partial[tile] = F;
                F = 0.0;
            }
            tb ^= 1;
            next_tile = s_tile[tb];  // written before the barrier above
        }
        tile = n_tile;
        rb = n_rb;
        r1 = n_r1;
        la = na;
        lb = nb;
    }
    if (most > n1) bad |= 2;
    bad = __reduce_or_sync(0xffffffffu, (unsigned)bad);
    if (lane == 0 && bad) atomicOr(&s->res.bad, bad);
    __threadfence();
    __syncthreads();
    if (tid == 0) is_last = atomicAdd(&s->ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // the last block adds the partials in tile order (fixed per-thread strides, fixed tree)
    double t = 0.0;
    constexpr int kP = 8;
    for (int i = tid; i < n_tiles; i += kP * kNaThreads) {
        double p[kP];
#pragma unroll
        for (int u = 0; u < kP; ++u) p[u] = i + u * kNaThreads < n_tiles ? __ldcg(&s->partial[i + u * kNaThreads]) : 0.0;
#pragma unroll
        for (int u = 0; u < kP; ++u) t += p[u];
    }
    t = na_warp_sum(t);
    if (lane == 0) wsum[wib] = t;
    __syncthreads();
    if (tid == 0) {
        double g = 0.0;
        for (int k = 0; k < kNaWarps; ++k) g += wsum[k];
        s->res.G = g;
    }
}

void na_set_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    imrt::set_last_error_message(buf);  // reported by imrt_last_error()
}

std::mutex na_mutex;
NaScratch* na_ptr[kNaMaxDevices] = {};

// Device address of the scratch array on the current device; looked up once per device.
imrt_status na_scratch(NaScratch** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        na_set_error("cudaGetDevice failed: %s", cudaGetErrorString(e));
        return IMRT_ECUDA;
    }
    if (dev < 0 || dev >= kNaMaxDevices) {
        na_set_error("device %d is beyond the %d devices this entry point tracks", dev, kNaMaxDevices);
        return IMRT_EUNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(na_mutex);
    if (!na_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess || !p) {
            na_set_error("cudaGetSymbolAddress of the scratch array failed: %s", cudaGetErrorString(e));
            return IMRT_ECUDA;
        }
        na_ptr[dev] = static_cast<NaScratch*>(p);
    }
    *out = na_ptr[dev];
    return IMRT_OK;
}

// Device (or managed) memory that the current device can read as its own: device memory of
// another GPU is refused, since the kernels would read it as peer memory or fault.
bool on_device(const void* p, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeDevice) return a.device == dev;
    return a.type == cudaMemoryTypeManaged;
}

// Memory that only a copy can write from the host (device memory of any GPU).
bool needs_copy(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice;
}

}  // namespace

extern "C" imrt_status imrt_eval_csr_noalloc(const imrt_csr* D, const uint8_t* structures, int32_t n_structures,
                                             const float* thresholds, const float* weights, const float* x,
                                             float* z_out, double* G_out, void* stream) {
    imrt::set_last_error_message("");
    if (!D || !structures || !thresholds || !weights || !x || !G_out) {
        na_set_error("NULL argument");
        return IMRT_EINVAL;
    }
    if (D->m < 1 || D->n < 1 || D->nnz < 0 || n_structures < 1 || n_structures > kNaMaxStruct) {
        na_set_error("need m >= 1, n >= 1, nnz >= 0 and 1..8 structures");
        return IMRT_EINVAL;
    }
    if ((int64_t)D->m > kNaMaxVoxels) {
        na_set_error("m = %d voxels exceeds the allocation-free limit of %lld voxels", D->m,
                     (long long)kNaMaxVoxels);
        return IMRT_EUNSUPPORTED;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        na_set_error("no CUDA device");
        return IMRT_ECUDA;
    }
    if (!D->on_device || !on_device(D->row_ptr, dev) ||
        (D->nnz > 0 && (!on_device(D->col_idx, dev) || !on_device(D->val, dev))) || !on_device(structures, dev) ||
        !on_device(x, dev) || (z_out && !on_device(z_out, dev))) {
        na_set_error("D, structures, x and z_out must be device pointers of the current device (%d)", dev);
        return IMRT_EINVAL;
    }
    for (int i = 0; i < 2 * n_structures; ++i)
        if (!(weights[i] >= 0.0f) || !isfinite(weights[i]) || isinf(thresholds[i])) {
            na_set_error("weights must be finite and >= 0; thresholds finite or NaN");
            return IMRT_EINVAL;
        }
    NaTerms terms;
    memset(&terms, 0, sizeof(terms));
    terms.S = n_structures;
    for (int t = 0; t < n_structures; ++t) {
        terms.Tu[t] = thresholds[2 * t];
        terms.To[t] = thresholds[2 * t + 1];
        terms.wu[t] = weights[2 * t];
        terms.wo[t] = weights[2 * t + 1];
    }
    NaScratch* s = nullptr;
    imrt_status st = na_scratch(&s);
    if (st != IMRT_OK) return st;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // tiles of 32 rows up to 524,288 voxels, then as many rows as keep the partials in the scratch
    const int tile_rows = (int)((D->m + (int64_t)kNaUnit * kNaMaxTiles - 1) / ((int64_t)kNaUnit * kNaMaxTiles)) * kNaUnit;
    const int n_tiles = (D->m + tile_rows - 1) / tile_rows;
    const int blocks = n_tiles < sms * kNaBlocksPerSm ? n_tiles : sms * kNaBlocksPerSm;
    const int want = (D->m + 8 * kNaThreads - 1) / (8 * kNaThreads);
    const int count_blocks = want < kNaCountBlocks ? want : kNaCountBlocks;
    const bool copy_G = needs_copy(G_out);  // an objective wanted in device memory takes a copy of its own
    NaResult out{};
    if (e == cudaSuccess) {
        k_na_counts<<<count_blocks, kNaThreads, 0, cs>>>(structures, D->m, s);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {  // may launch while the counts are taken; waits for them before it reads
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(kNaThreads);
        cfg.stream = cs;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, k_na_eval, D->row_ptr, D->col_idx, D->val, D->m, D->n, D->nnz, structures,
                               terms, x, z_out, tile_rows, n_tiles, count_blocks, s);
    }
    // the objective and the error flag in one copy
    if (e == cudaSuccess) e = cudaMemcpyAsync(&out, &s->res, sizeof(out), cudaMemcpyDeviceToHost, cs);
    if (e == cudaSuccess && copy_G) e = cudaMemcpyAsync(G_out, &s->res.G, sizeof(double), cudaMemcpyDefault, cs);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
    if (e != cudaSuccess) {
        na_set_error("CUDA error: %s", cudaGetErrorString(e));
        return IMRT_ECUDA;
    }
    const int32_t bad = out.bad;
    if (!copy_G) *G_out = out.G;
    if (bad) {
        na_set_error("invalid CSR: %s%s%s", (bad & 1) ? "row offsets outside [0, nnz] or decreasing" : "",
                     (bad & 3) == 3 ? "; " : "", (bad & 2) ? "beamlet index outside [0, n)" : "");
        return IMRT_EINVAL;
    }
    return IMRT_OK;
}
