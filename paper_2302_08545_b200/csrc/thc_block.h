// What the host side needs to launch the kernels of thc_block.cu.
#pragma once
#include "thc_pipeline.cuh"

namespace thc {

// How a block size is held: 0 up to 2^13, one tile of 2^13; 1: 2^14, one tile of 2^14; 2: 2^15, a
// cluster of two tiles of 2^14; 3 and 4: 2^16 and 2^17, a cluster of eight tiles of 2^13 or 2^14.  A tile of 2^13 has 128
// threads and four CTAs per SM, one of 2^14 256 threads and two.
__host__ __device__ constexpr int block_kind(uint32_t k) { return k <= 13u ? 0 : k == 14u ? 1 : k == 15u ? 2 : k == 16u ? 3 : 4; }
__host__ __device__ constexpr int block_tile_log2(int kind) { return kind == 0 || kind == 3 ? 13 : 14; }
__host__ __device__ constexpr uint32_t block_cluster_log2(int kind) { return kind == 2 ? 1u : kind >= 3 ? 3u : 0u; }

// Scales and compress in one launch (kinds 0 and 1): block sizes from 2^8 on, up to this many workers (a cluster of one
// CTA per worker, of the size that every GPU can hold).
constexpr uint32_t kScalesMinLog2 = 8, kScalesMaxWorkers = 8;

struct BlockParams {
    uint64_t d;
    uint64_t d_pad;
    const float *scales;
    DeviceBlock *dev;
    uint32_t tasks;            // (tile or block) x worker; worker minor
    uint32_t n_local;
    uint32_t k;
    uint32_t granularity;
    uint32_t divisor;
    uint32_t round;
    uint32_t worker_base;
    float    c_block;
    uint32_t exact_range;      // scales = nblocks minima then nblocks maxima (else M per block)
    uint32_t nblocks;
    uint32_t const_slots;      // blocks a tile can overlap
    uint32_t *range_keys;      // range mode: see add_range
    float   *range_out;        // ... finished by the last CTA (or null: by range_final_kernel)
    uint32_t *head;            // counter of claimed tasks, or null: fixed stride (see launch_block)
    uint32_t *exited;          // CTAs that have ended (both are zero between launches)
    float   *scales_out;       // scales + compress: = scales, written by the kernel; tasks are tiles of all workers
    double   t_p, sqrt_block;
    uint32_t agg_n;            // aggregate + decompress: workers whose table values are summed
    uint32_t agg_chunk;        // ... and how many of them before a byte could overflow
    uint32_t agg_acc_bits;     // ... and the width of the sums written on request (outp.p[1])
};

// The kernel for a mode, index width and block size (signature: TmaMaps, BlockParams, PtrArrayP,
// MutPtrArrayP outputs, MutPtrArrayP rotated, PhiloxKeys); with claims, the one for launches that are given P.head.
const void *block_kernel(PipeMode mode, uint32_t bits, bool identity, uint32_t k, bool claims = false);

}  // namespace thc
