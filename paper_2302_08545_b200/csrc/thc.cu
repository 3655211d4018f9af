// libthc: kernels and C ABI.  See include/thc.h for the contract of every entry point.
//
// Structure of the transform.  RHT blocks of up to 2^15 coordinates, and few blocks of 2^16 or 2^17, are held
// in shared memory by one CTA or a cluster (thc_block.cu; block_kernel_serves has the rule); the others go
// through the persistent two-pass pipeline of thc_pipeline.cuh.
#include "../../include/thc.h"
#include "thc_device.cuh"

#include <atomic>
#include <math.h>
#include <mutex>
#include <new>
#include <stdio.h>
#include <string.h>

namespace thc {

struct PtrArray { const void *p[THC_MAX_WORKERS]; };
struct MutPtrArray { void *p[THC_MAX_WORKERS]; };

constexpr int kQrBlockCache = 1024;

// Quantise + pack coordinates that are already rotated (the epilogue of compress alone).
template <int BITS, bool IDENTITY>
__global__ void __launch_bounds__(kThreads)
quantize_rotated_kernel(PtrArray rotated, MutPtrArray packed, uint64_t d_pad, uint32_t k,
                        uint32_t granularity, uint32_t round, uint32_t worker_base, uint32_t exact_range,
                        const float *scales, const DeviceBlock *dev, PhiloxKeys keys)
{
    // dynamic shared memory: the quantiser table, one copy per lane group, then the block
    // constants of the first kQrBlockCache RHT blocks (the fp64 division is done once per block)
    extern __shared__ __align__(16) unsigned char qr_smem[];
    unsigned char *lut = qr_smem;
    float2 *bc = reinterpret_cast<float2 *>(qr_smem + (size_t)(granularity + 1) * kLutEntryBytes);
    if (!IDENTITY) lut_fill(lut, dev, granularity, threadIdx.x, kThreads);
    depend_on_previous();
    const uint64_t nblocks = d_pad >> k;
    const uint32_t cached = nblocks < (uint64_t)kQrBlockCache ? (uint32_t)nblocks : (uint32_t)kQrBlockCache;
    for (uint32_t b = threadIdx.x; b < cached; b += kThreads)
        bc[b] = compress_constants(block_range(scales, b, nblocks, exact_range));
    __syncthreads();
    const uint32_t wl = blockIdx.y;
    const float *rot = static_cast<const float *>(rotated.p[wl]);
    unsigned char *pk = static_cast<unsigned char *>(packed.p[wl]);
    const float gf = (float)granularity;
    const uint32_t my_lut = lut_lane_addr(lut, threadIdx.x);
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < d_pad / 8;
         u += (uint64_t)gridDim.x * kThreads) {
        const uint64_t j = u * 8;
        const float4 a = ld_global_once(reinterpret_cast<const float4 *>(rot + j));
        const float4 b = ld_global_once(reinterpret_cast<const float4 *>(rot + j + 4));
        const float r[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        const uint64_t blk = j >> k;
        const float2 kc = blk < cached ? bc[blk] : compress_constants(block_range(scales, blk, nblocks, exact_range));
        const float kappa = kc.x, offset = kc.y;
        const uint4 rnd = round_call(j, worker_base + wl, round, keys);
        const uint64_t z = quantize8<BITS, IDENTITY>(r, kappa, offset, gf, rnd, my_lut);
        store_unit<BITS>(pk, j, z);
    }
}

// 32 bytes of sums to a 16-byte aligned address; in one store where it is 32-byte aligned, so that no
// sector of 32 bytes reaches the L2 in two halves.
__device__ __forceinline__ void store_sums32(uint4 *p, bool aligned32, const uint32_t (&v)[8])
{
    if (aligned32) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" :: "l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                     "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
    } else {
        p[0] = make_uint4(v[0], v[1], v[2], v[3]);
        p[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}

// Fast path of the PS sum for 4-bit indices, 8-bit sums and table values below 128 (the
// paper's prototype: 4-bit indices, 8-bit table values and sums, Section 3).  The 16 table
// bytes sit in four registers; `prmt` looks four indices up at once.  A selector nibble with
// bit 3 set makes prmt return the sign of the selected byte, i.e. 0 for values < 128, so the
// low half of the table answers indices 0-7 and, with bit 3 flipped, the high half answers
// 8-15; the two results are disjoint and are added into packed byte accumulators (no byte
// can overflow because workers * g <= 255).
__global__ void __launch_bounds__(kThreads)
aggregate_b4w8_kernel(PtrArray in, uint32_t n, uint64_t units32, const DeviceBlock *dev,
                      uint4 *__restrict__ sum)
{
    uint32_t t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        t[q] = dev->table[4 * q] | (dev->table[4 * q + 1] << 8) | (dev->table[4 * q + 2] << 16) |
               (dev->table[4 * q + 3] << 24);
    depend_on_previous();
    const bool aligned32 = (reinterpret_cast<uintptr_t>(sum) & 31u) == 0;
    // A thread sums 32 coordinates: 16 bytes of indices per worker, the loads of up to eight
    // workers in flight together, 32 bytes of sums out.
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < units32;
         u += (uint64_t)gridDim.x * kThreads) {
        uint32_t acc[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};     // 32 sums of 8 bits
#pragma unroll 1
        for (uint32_t i0 = 0; i0 < n; i0 += 8) {
            uint4 w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)         // index 0 everywhere adds T[0] = 0
                w[j] = i0 + j < n ? ld_global_once(reinterpret_cast<const uint4 *>(in.p[i0 + j]) + u) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t words[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const uint32_t a = words[h], b = a ^ 0x88888888u;
                    acc[2 * h] += prmt(t[0], t[1], a) + prmt(t[2], t[3], b);
                    acc[2 * h + 1] += prmt(t[0], t[1], a >> 16) + prmt(t[2], t[3], b >> 16);
                }
            }
        }
        store_sums32(sum + 2 * u, aligned32, acc);
    }
}

// The same with 16-bit sums (more workers than fit a byte: workers * g > 255).  Table values are
// summed in byte lanes for CHUNK workers at a time (CHUNK * g <= 255), then widened into
// 16-bit lanes (even and odd coordinates apart) and put back in order at the end.
template <int CHUNK>
__global__ void __launch_bounds__(kThreads)
aggregate_b4w16_kernel(PtrArray in, uint32_t n, uint64_t units32, const DeviceBlock *dev,
                       uint4 *__restrict__ sum)
{
    uint32_t t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
        t[q] = dev->table[4 * q] | (dev->table[4 * q + 1] << 8) | (dev->table[4 * q + 2] << 16) |
               (dev->table[4 * q + 3] << 24);
    depend_on_previous();
    const bool aligned32 = (reinterpret_cast<uintptr_t>(sum) & 31u) == 0;
    // A thread sums 32 coordinates: 16 bytes of indices per worker, 64 bytes of sums out.
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < units32;
         u += (uint64_t)gridDim.x * kThreads) {
        uint32_t even[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u}, odd[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll 1
        for (uint32_t i0 = 0; i0 < n; i0 += CHUNK) {
            uint4 w[CHUNK];
#pragma unroll
            for (int j = 0; j < CHUNK; ++j)      // index 0 everywhere adds T[0] = 0
                w[j] = i0 + j < n ? ld_global_once(reinterpret_cast<const uint4 *>(in.p[i0 + j]) + u) : make_uint4(0u, 0u, 0u, 0u);
            uint32_t acc[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
            for (int j = 0; j < CHUNK; ++j) {
                const uint32_t words[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const uint32_t a = words[h], b = a ^ 0x88888888u;
                    acc[2 * h] += prmt(t[0], t[1], a) + prmt(t[2], t[3], b);
                    acc[2 * h + 1] += prmt(t[0], t[1], a >> 16) + prmt(t[2], t[3], b >> 16);
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                even[q] += acc[q] & 0x00FF00FFu;
                odd[q] += (acc[q] >> 8) & 0x00FF00FFu;
            }
        }
#pragma unroll
        for (int q4 = 0; q4 < 2; ++q4) {
            uint32_t o[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                o[2 * q] = prmt(even[4 * q4 + q], odd[4 * q4 + q], 0x5410u);          // coordinates 4q, 4q+1
                o[2 * q + 1] = prmt(even[4 * q4 + q], odd[4 * q4 + q], 0x7632u);      // coordinates 4q+2, 4q+3
            }
            store_sums32(sum + 4 * u + 2 * q4, aligned32, o);
        }
    }
}

// 1- and 2-bit indices with 8-bit sums: T[z] = g z for one bit, the identity table for two, so
// the sum of table values is g times the sum of the indices.  Index fields are spread into
// byte lanes by shift and mask (lane j of the k-th spread holds coordinate (8/BITS) j + k), added
// across workers, and transposed into coordinate order at the end.  A thread handles 32
// coordinates.
template <int BITS>
__global__ void __launch_bounds__(kThreads)
aggregate_small_w8_kernel(PtrArray in, uint32_t n, uint64_t units32, uint32_t g_mult,
                          uint4 *__restrict__ sum)
{
    depend_on_previous();
    constexpr int kWords = BITS;                       // 32 coordinates = BITS words
    constexpr int kSpread = 8 / BITS;                  // spreads per word
    constexpr uint32_t kMask = BITS == 1 ? 0x01010101u : 0x03030303u;
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < units32;
         u += (uint64_t)gridDim.x * kThreads) {
        uint32_t acc[kWords][kSpread];
#pragma unroll
        for (int q = 0; q < kWords; ++q)
#pragma unroll
            for (int k = 0; k < kSpread; ++k) acc[q][k] = 0u;
#pragma unroll 4
        for (uint32_t i = 0; i < n; ++i) {
            uint32_t words[kWords];
            if constexpr (BITS == 1) {
                words[0] = ld_global(reinterpret_cast<const uint32_t *>(in.p[i]) + u);
            } else {
                const uint2 w = ld_global(reinterpret_cast<const uint2 *>(in.p[i]) + u);
                words[0] = w.x; words[1] = w.y;
            }
#pragma unroll
            for (int q = 0; q < kWords; ++q)
#pragma unroll
                for (int k = 0; k < kSpread; ++k) acc[q][k] += (words[q] >> (k * BITS)) & kMask;
        }
        // byte j of acc[q][k] is coordinate (32/BITS) q + kSpread j + k: gather four consecutive
        // coordinates into each output word
        uint32_t o[8];
#pragma unroll
        for (int q = 0; q < kWords; ++q) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
                for (int h = 0; h < kSpread / 4; ++h) {
                    const uint32_t *a = &acc[q][4 * h];
                    const uint32_t sel = (uint32_t)j | ((uint32_t)(4 + j) << 4);
                    const uint32_t p01 = prmt(a[0], a[1], sel);            // bytes: a0[j], a1[j]
                    const uint32_t p23 = prmt(a[2], a[3], sel);            // bytes: a2[j], a3[j]
                    const uint32_t word = prmt(p01, p23, 0x5410u);         // a0[j], a1[j], a2[j], a3[j]
                    o[(q * (32 / BITS) + kSpread * j + 4 * h) / 4] = word * g_mult;
                }
            }
        }
        store_sums32(sum + 2 * u, (reinterpret_cast<uintptr_t>(sum) & 31u) == 0, o);
    }
}

// 3-bit indices, any table: eight bytes in two registers, looked up four at a time.  The 24 bits of eight
// indices are spread into nibbles (three shift-and-mask steps); table values are summed in byte
// lanes for `chunk` workers at a time (chunk * g <= 255) and, for 16-bit sums, widened into 16-bit lanes
// in between.  A thread sums 64 coordinates: three 8-byte loads per worker, of four workers in flight.
// (The shared-memory table of aggregate_kernel takes a look-up per index: 12.6 us on 10 workers x 2^22.)
template <int W>
__global__ void __launch_bounds__(128)
aggregate_b3_kernel(PtrArray in, uint32_t n, uint64_t units64, uint32_t chunk, const DeviceBlock *dev, uint4 *__restrict__ sum)
{
    const uint32_t t0 = dev->table[0] | (dev->table[1] << 8) | (dev->table[2] << 16) | (dev->table[3] << 24);
    const uint32_t t1 = dev->table[4] | (dev->table[5] << 8) | (dev->table[6] << 16) | (dev->table[7] << 24);
    depend_on_previous();
    const bool aligned32 = (reinterpret_cast<uintptr_t>(sum) & 31u) == 0;
    for (uint64_t u = (uint64_t)blockIdx.x * 128 + threadIdx.x; u < units64; u += (uint64_t)gridDim.x * 128) {
        uint32_t wide[W == 16 ? 32 : 1];
#pragma unroll
        for (int q = 0; q < (W == 16 ? 32 : 1); ++q) wide[q] = 0u;
        uint32_t acc[16];                              // 64 sums of 8 bits
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[q] = 0u;
#pragma unroll 1
        for (uint32_t i0 = 0; i0 < n; i0 += chunk) {
            const uint32_t i1 = min(n, i0 + chunk);
#pragma unroll 4
            for (uint32_t i = i0; i < i1; ++i) {
                uint32_t w[7];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const uint2 v = ld_global(reinterpret_cast<const uint2 *>(in.p[i]) + 3 * u + q);
                    w[2 * q] = v.x; w[2 * q + 1] = v.y;
                }
                w[6] = 0u;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t x = __funnelshift_r(w[24 * e / 32], w[24 * e / 32 + 1], 24 * e % 32);
                    const uint32_t y = (x & 0x00000FFFu) | ((x << 4) & 0x0FFF0000u);
                    const uint32_t z = (y & 0x003F003Fu) | ((y << 2) & 0x3F003F00u);
                    const uint32_t s = (z & 0x07070707u) | ((z << 1) & 0x70707070u);
                    acc[2 * e] += prmt(t0, t1, s);
                    acc[2 * e + 1] += prmt(t0, t1, s >> 16);
                }
            }
            if (W == 16) {
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    wide[(2 * q) % (W == 16 ? 32 : 1)] += acc[q] & 0x00FF00FFu;
                    wide[(2 * q + 1) % (W == 16 ? 32 : 1)] += (acc[q] >> 8) & 0x00FF00FFu;
                    acc[q] = 0u;
                }
            }
        }
        if (W == 8) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t o[8] = {acc[8 * q], acc[8 * q + 1], acc[8 * q + 2], acc[8 * q + 3],
                                       acc[8 * q + 4], acc[8 * q + 5], acc[8 * q + 6], acc[8 * q + 7]};
                store_sums32(sum + 4 * u + 2 * q, aligned32, o);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t o[8];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t even = wide[(8 * q + 2 * c) % (W == 16 ? 32 : 1)], odd = wide[(8 * q + 2 * c + 1) % (W == 16 ? 32 : 1)];
                    o[2 * c] = prmt(even, odd, 0x5410u);
                    o[2 * c + 1] = prmt(even, odd, 0x7632u);
                }
                store_sums32(sum + 8 * u + 2 * q, aligned32, o);
            }
        }
    }
}

// 8-bit indices with the identity table (g = 255) and 16-bit sums: bytes are widened into
// 16-bit lanes (even and odd coordinates apart).  A thread handles 16 coordinates.
__global__ void __launch_bounds__(kThreads)
aggregate_b8w16_kernel(PtrArray in, uint32_t n, uint64_t units16, uint4 *__restrict__ sum)
{
    depend_on_previous();
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < units16;
         u += (uint64_t)gridDim.x * kThreads) {
        uint32_t even[4] = {0u, 0u, 0u, 0u}, odd[4] = {0u, 0u, 0u, 0u};
#pragma unroll 4
        for (uint32_t i = 0; i < n; ++i) {
            const uint4 w = ld_global(reinterpret_cast<const uint4 *>(in.p[i]) + u);
            const uint32_t words[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                even[q] += words[q] & 0x00FF00FFu;
                odd[q] += (words[q] >> 8) & 0x00FF00FFu;
            }
        }
        uint32_t o[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o[2 * q] = prmt(even[q], odd[q], 0x5410u);
            o[2 * q + 1] = prmt(even[q], odd[q], 0x7632u);
        }
        store_sums32(sum + 2 * u, (reinterpret_cast<uintptr_t>(sum) & 31u) == 0, o);
    }
}

// ------------------------------------------------------------------------ error feedback
// x <- x + e of all workers in one launch: four 16-byte loads of each in flight per thread, a scalar tail.
// (One launch per worker: 4 x 7,000,003 coordinates 62 us, now 50 us = 6.7 TB/s.)
constexpr int kAccUnits = 4;
__global__ void __launch_bounds__(kThreads)
accumulate_kernel(MutPtrArray xs, PtrArray es, uint64_t d)
{
    depend_on_previous();
    float *x = static_cast<float *>(xs.p[blockIdx.y]);
    const float *e = static_cast<const float *>(es.p[blockIdx.y]);
    const uint64_t n4 = d / 4;
    const uint64_t c0 = (uint64_t)blockIdx.x * (kThreads * kAccUnits) + threadIdx.x;
    float4 a[kAccUnits], b[kAccUnits];
#pragma unroll
    for (int i = 0; i < kAccUnits; ++i) {
        const uint64_t c = c0 + (uint64_t)i * kThreads;
        if (c < n4) { a[i] = reinterpret_cast<float4 *>(x)[c]; b[i] = ld_global_once(reinterpret_cast<const float4 *>(e) + c); }
    }
#pragma unroll
    for (int i = 0; i < kAccUnits; ++i) {
        const uint64_t c = c0 + (uint64_t)i * kThreads;
        if (c < n4)
            reinterpret_cast<float4 *>(x)[c] = make_float4(a[i].x + b[i].x, a[i].y + b[i].y, a[i].z + b[i].z, a[i].w + b[i].w);
    }
    if (blockIdx.x == 0 && threadIdx.x < (d & 3)) {
        const uint64_t j = n4 * 4 + threadIdx.x;
        x[j] = x[j] + e[j];
    }
}

// ------------------------------------------------------------------------------ prepare
// Sums of squares in fp64.  HBM-bound: 16 bytes per load, all of a thread's loads for a worker in
// flight together (4 x 2^26 fp32 coordinates: 5.8 -> 6.3 TB/s), and one launch where the second one
// of a small call cost as much as the first.

// 16 bytes of a gradient: 4 fp32 or 8 bf16 coordinates from j on, zero behind d.
template <bool BF16>
__device__ __forceinline__ uint4 load_unit(const void *x, uint64_t j, uint64_t d)
{
    constexpr int kPer = BF16 ? 8 : 4;
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (j + kPer <= d) {
        const char *p = static_cast<const char *>(x) + j * (16 / kPer);
        asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "l"(p));
    } else if (j < d) {
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        for (int e = 0; e < kPer; ++e) {
            if (j + e >= d) break;
            if (BF16) w[e >> 1] |= (uint32_t)ld_global(static_cast<const uint16_t *>(x) + j + e) << ((e & 1) * 16);
            else w[e & 3] = ld_global(static_cast<const uint32_t *>(x) + j + e);
        }
        q = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return q;
}

template <bool BF16>
__device__ __forceinline__ double add_squares(double s, uint4 q)
{
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (BF16) {
            const double lo = (double)__uint_as_float(w[e] << 16), hi = (double)__uint_as_float(w[e] & 0xFFFF0000u);
            s = fma(lo, lo, s);
            s = fma(hi, hi, s);
        } else {
            const double v = (double)__uint_as_float(w[e]);
            s = fma(v, v, s);
        }
    }
    return s;
}

// M = t_p ell / sqrt(B) to scales[blk], and the status bits.
__device__ __forceinline__ void store_scale(double ell, double t_p, uint32_t k, uint64_t blk, float *scales, DeviceBlock *dev)
{
    float M = (float)(t_p * ell / sqrt((double)((uint64_t)1 << k)));
    uint32_t flags = 0;
    if (!isfinite(M)) { M = 0.0f; flags |= THC_STATUS_NONFINITE; }
    if (M == 0.0f) flags |= THC_STATUS_ZERO_BLOCK;
    scales[blk] = M;
    if (flags) atomicOr(&dev->status, flags);
}

__device__ __forceinline__ double max_norm(double a, double b) { return (b > a || b != b) ? b : a; }   // a NaN norm sticks

// Blocks of up to 2^12: a CTA takes 2^12 coordinates of all workers and writes the scales of their blocks.
// A warp takes 512 consecutive coordinates, in slabs of 32 loads; blocks of 2^9 and more are whole
// warps (one reduction per worker and warp), smaller ones two slabs, one slab or 2^g lanes of it.
constexpr int kSmallPrepLog2 = 12;
template <bool BF16>
__global__ void __launch_bounds__(kThreads)
prepare_small_kernel(PtrArray in, uint32_t n, uint64_t d, uint64_t d_pad, uint32_t k, double t_p, float *__restrict__ scales,
                     DeviceBlock *dev)
{
    depend_on_previous();
    constexpr uint32_t kPerLog2 = BF16 ? 3u : 2u;
    constexpr int kSlabs = 1 << (9 - 5 - kPerLog2);
    __shared__ double s_warp[THC_MAX_WORKERS][kThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t g = min(k - kPerLog2, 5u);
    const bool pairs = k == 6u + kPerLog2;             // a block is two slabs
    const uint64_t j0 = ((uint64_t)blockIdx.x << kSmallPrepLog2) + 512u * warp + ((uint64_t)lane << kPerLog2);
    double ell[kSlabs];
#pragma unroll
    for (int i = 0; i < kSlabs; ++i) ell[i] = 0.0;
#pragma unroll 4
    for (uint32_t w = 0; w < n; ++w) {
        uint4 q[kSlabs];
#pragma unroll
        for (int i = 0; i < kSlabs; ++i) q[i] = load_unit<BF16>(in.p[w], j0 + ((uint64_t)i << (5 + kPerLog2)), d);
        if (k >= 9u) {
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < kSlabs; ++i) s = add_squares<BF16>(s, q[i]);
            for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
            if (lane == 0) s_warp[w][warp] = s;
        } else {
#pragma unroll
            for (int i = 0; i < kSlabs; ++i) {
                double s = add_squares<BF16>(0.0, q[i]);
                if (pairs) {
                    if (i & 1) continue;
                    s = add_squares<BF16>(s, q[i + 1 < kSlabs ? i + 1 : i]);
                }
                for (uint32_t b = 0; b < g; ++b) s += __shfl_xor_sync(0xFFFFFFFFu, s, 1 << b);
                ell[i] = max_norm(ell[i], sqrt(s));
            }
        }
    }
    if (k < 9u) {
        if ((lane & ((1 << g) - 1)) != 0) return;
#pragma unroll
        for (int i = 0; i < kSlabs; ++i) {
            const uint64_t j = j0 + ((uint64_t)i << (5 + kPerLog2));
            if (j < d_pad && !(pairs && (i & 1))) store_scale(ell[i], t_p, k, j >> k, scales, dev);
        }
        return;
    }
    // a warp per block, the lanes share the workers
    __syncthreads();
    const int warps = 1 << (k - 9u);
    if (warp >= (1 << (kSmallPrepLog2 - k))) return;
    double m = 0.0;
    for (uint32_t w = (uint32_t)lane; w < n; w += 32u) {
        double s = 0.0;
        for (int v = 0; v < warps; ++v) s += s_warp[w][warp * warps + v];
        m = max_norm(m, sqrt(s));
    }
    for (int off = 16; off > 0; off >>= 1) m = max_norm(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
    const uint64_t blk = ((uint64_t)blockIdx.x << (kSmallPrepLog2 - k)) + (uint32_t)warp;
    if (lane == 0 && (blk << k) < d_pad) store_scale(m, t_p, k, blk, scales, dev);
}

// Larger blocks: partial sums of one (chunk of 2^chunk_log2 coordinates, worker) per CTA; with
// `counters` the CTA that finishes the last chunk of an RHT block (over all workers) computes its scale
// from the stored sums in a fixed order (atomicInc wraps, so the counters are zero again).
template <bool BF16>
__global__ void __launch_bounds__(kThreads)
prepare_partial_kernel(PtrArray in, uint64_t d, uint32_t chunk_log2, uint64_t chunks_per_worker,
                       double *__restrict__ partial, uint32_t *counters, uint32_t chunks_per_block, double t_p, uint32_t k,
                       float *__restrict__ scales, DeviceBlock *dev)
{
    depend_on_previous();
    constexpr uint32_t kPerLog2 = BF16 ? 3u : 2u;
    const uint64_t chunk = blockIdx.x;
    const uint32_t wl = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t j0 = (chunk << chunk_log2) + ((uint64_t)tid << kPerLog2);
    const uint32_t units = 1u << (chunk_log2 - 8u - kPerLog2);           // per thread: a multiple of four
    double s = 0.0;
#pragma unroll 1
    for (uint32_t i = 0; i < units; i += 4) {
        uint4 q[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) q[e] = load_unit<BF16>(in.p[wl], j0 + ((uint64_t)(i + e) << (8 + kPerLog2)), d);
#pragma unroll
        for (int e = 0; e < 4; ++e) s = add_squares<BF16>(s, q[e]);
    }
    __shared__ double red[kThreads / 32];
    __shared__ uint32_t last;
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, off);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    const uint64_t blk = chunk / chunks_per_block;
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) t += red[w];
        __stcg(partial + (uint64_t)wl * chunks_per_worker + chunk, t);
        last = 0u;
        if (counters != nullptr) {
            const uint32_t total = gridDim.y * chunks_per_block;
            __threadfence();
            last = atomicInc(counters + blk, total - 1u) == total - 1u;
        }
    }
    __syncthreads();
    if (!last) return;
    // a warp per worker in turn
    __threadfence();
    double ell = 0.0;
    for (uint32_t w = (uint32_t)warp; w < gridDim.y; w += kThreads / 32) {
        const double *p = partial + (uint64_t)w * chunks_per_worker + blk * chunks_per_block;
        double t = 0.0;
        for (uint32_t c = (uint32_t)lane; c < chunks_per_block; c += 32u) t += __ldcg(p + c);
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, off);
        ell = max_norm(ell, sqrt(t));
    }
    if (lane == 0) red[warp] = ell;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kThreads / 32; ++w) ell = max_norm(ell, red[w]);
        store_scale(ell, t_p, k, blk, scales, dev);
    }
}

// M per block from the partial sums (Section 5.3: M = t_p * max_i ||x_i|| / sqrt(B)).  One warp
// per RHT block, eight workers at a time with four lanes per worker: a lane adds every fourth
// partial sum of its worker (loads independent of each other), the four lanes are combined,
// one square root per worker, then the maximum over workers.  The order is fixed, so the
// result does not depend on timing.  For more blocks than there are counters.
__global__ void __launch_bounds__(128)
prepare_final_kernel(const double *partial, uint32_t n, uint64_t nblocks,
                     uint64_t chunks_per_block, uint64_t chunks_per_worker, double t_p, uint32_t k,
                     float *__restrict__ scales, DeviceBlock *dev)
{
    depend_on_previous();
    const uint64_t blk = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (blk >= nblocks) return;
    double ell = 0.0;
    for (uint32_t i0 = 0; i0 < n; i0 += 8u) {
        const uint32_t i = i0 + ((uint32_t)lane >> 2);
        const bool live = i < n;
        const double *p = partial + (uint64_t)(live ? i : 0u) * chunks_per_worker + blk * chunks_per_block;
        double s = 0.0;
        for (uint64_t c = (uint64_t)(lane & 3); c < chunks_per_block; c += 4) s += p[c];
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
        double norm = live ? sqrt(s) : 0.0;
        for (int off = 4; off < 32; off <<= 1) {
            norm = max_norm(norm, __shfl_xor_sync(0xFFFFFFFFu, norm, off));
        }
        ell = max_norm(ell, norm);
    }
    if (lane != 0) return;
    store_scale(ell, t_p, k, blk, scales, dev);
}

// Exact range (Algorithm 1's preliminary stage on the rotated coordinates) of more blocks than the context
// has keys for: keys in the workspace, cleared before and turned into the ranges after the transform.
__global__ void range_final_kernel(uint32_t *keys, uint64_t nblocks, float *scales, DeviceBlock *dev)
{
    depend_on_previous();
    const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nblocks) finish_range(keys, nblocks, r, scales, dev);
}

// ---------------------------------------------------------------------------- aggregate
// Y[j] = sum_i T[z_i[j]] (Algorithm 2, PS line).  One thread per 32 coordinates.
template <int BITS, int W>
__global__ void __launch_bounds__(kThreads)
aggregate_kernel(PtrArray in, uint32_t n, uint64_t units, uint64_t d_pad, const DeviceBlock *dev,
                 unsigned char *__restrict__ sum)
{
    __shared__ uint32_t T[256];
    for (int z = threadIdx.x; z < (1 << BITS); z += kThreads) T[z] = dev->table[z];
    depend_on_previous();
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // coordinates past the last whole group of 32 (blocks of 8 or 16 coordinates only)
        for (uint64_t j = units * 32; j < d_pad; ++j) {
            uint32_t acc = 0;
            for (uint32_t i = 0; i < n; ++i) {
                const unsigned char *pb = static_cast<const unsigned char *>(in.p[i]);
                const uint64_t bit = j * BITS;
                uint32_t two = pb[bit >> 3];
                if (((bit & 7) + BITS) > 8) two |= (uint32_t)pb[(bit >> 3) + 1] << 8;
                acc += T[(two >> (bit & 7)) & ((1u << BITS) - 1u)];
            }
            if constexpr (W == 8) sum[j] = (unsigned char)acc;
            else if constexpr (W == 16) reinterpret_cast<uint16_t *>(sum)[j] = (uint16_t)acc;
            else reinterpret_cast<uint32_t *>(sum)[j] = acc;
        }
    }
    constexpr int kInWords = BITS;                 // 32 indices * BITS bits = BITS words
    for (uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x; u < units;
         u += (uint64_t)gridDim.x * kThreads) {
        uint32_t acc[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) acc[e] = 0;
        for (uint32_t i = 0; i < n; ++i) {
            const uint32_t *src = reinterpret_cast<const uint32_t *>(
                static_cast<const unsigned char *>(in.p[i]) + u * (4 * BITS));
            uint32_t w[kInWords];
            if constexpr (BITS == 8) {
                const uint4 a = ld_global(reinterpret_cast<const uint4 *>(src));
                const uint4 b = ld_global(reinterpret_cast<const uint4 *>(src) + 1);
                w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
                w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
            } else if constexpr (BITS == 4) {
                const uint4 a = ld_global(reinterpret_cast<const uint4 *>(src));
                w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
            } else if constexpr (BITS == 3) {
                w[0] = ld_global(src); w[1] = ld_global(src + 1); w[2] = ld_global(src + 2);
            } else if constexpr (BITS == 2) {
                const uint2 a = ld_global(reinterpret_cast<const uint2 *>(src));
                w[0] = a.x; w[1] = a.y;
            } else {
                w[0] = ld_global(src);
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const int bit = e * BITS;
                // a 3-bit index may straddle two words: funnel shift over the pair
                const uint32_t lo = w[bit >> 5], hi = w[((bit >> 5) + 1) < kInWords ? (bit >> 5) + 1 : (bit >> 5)];
                const uint32_t z = __funnelshift_r(lo, hi, bit & 31) & ((1u << BITS) - 1u);
                acc[e] += T[z];
            }
        }
        unsigned char *dst = sum + u * (32 * W / 8);
        if constexpr (W == 8) {
            uint32_t o[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                o[q] = (acc[4 * q] & 0xFFu) | ((acc[4 * q + 1] & 0xFFu) << 8) |
                       ((acc[4 * q + 2] & 0xFFu) << 16) | (acc[4 * q + 3] << 24);
            reinterpret_cast<uint4 *>(dst)[0] = make_uint4(o[0], o[1], o[2], o[3]);
            reinterpret_cast<uint4 *>(dst)[1] = make_uint4(o[4], o[5], o[6], o[7]);
        } else if constexpr (W == 16) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t o[4];
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    o[t] = (acc[8 * q + 2 * t] & 0xFFFFu) | (acc[8 * q + 2 * t + 1] << 16);
                reinterpret_cast<uint4 *>(dst)[q] = make_uint4(o[0], o[1], o[2], o[3]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                reinterpret_cast<uint4 *>(dst)[q] =
                    make_uint4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
        }
    }
}

}  // namespace thc

#include "thc_pipeline.cuh"
#include "thc_block.h"

// =========================================================================== host side
using namespace thc;

struct thc_ctx {
    thc_config cfg;
    uint32_t acc_bits;
    bool identity;
    int device;                 // -1: no CUDA device, host-only context
    DeviceBlock *dev;
    PhiloxKeys keys;
    bool pipeline_next;         // the queue of the next pipeline launch is set (thc_debug_skip_tasks); until then
                                // blocks above 2^14 take the pipeline
    int sm_count;
    int lone_clusters;          // see block_kernel_serves; blocks of 2^17 only
    // Encoded tensor maps of recent launches, keyed by what they describe: a training loop calls
    // with the same buffers every step, and encoding up to n + 1 maps per call costs more host
    // time than a small launch takes on the device.
    struct MapEntry { const void *base; uint64_t cols, rows, pitch; uint32_t box_rows, box_cols, half, groups; CUtensorMap map; };
    static constexpr int kMapCache = 2 * (THC_MAX_WORKERS + 2);
    mutable MapEntry map_cache[kMapCache];
    mutable int map_cache_used, map_cache_next;
    mutable std::mutex map_mutex;
    // Per mode, what resident_units answered for this context's block kernel (0: not asked yet); then for clusters
    // of one CTA per worker.
    mutable std::atomic<uint32_t> resident[kPipeModes + kScalesMaxWorkers + 1];
};

static thread_local cudaError_t g_last_cuda = cudaSuccess;
static thread_local char g_err_text[256];

static int cuda_fail(cudaError_t e)
{
    g_last_cuda = e;
    return THC_ECUDA;
}

#define THC_CUDA(...)                                         \
    do {                                                      \
        cudaError_t e__ = (__VA_ARGS__);                      \
        if (e__ != cudaSuccess) return cuda_fail(e__);        \
    } while (0)

// A launch that may start while the one before it on the stream is still running (depend_on_previous):
// 1 to 1.5 us less between two launches of a round.
template <class... P, class... A>
static cudaError_t launch_after(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// No launch takes more dynamic shared memory: a pipeline CTA, a tile of 2^14 or one of 2^13 with the constants
// of 1024 blocks, each with a table of 256 entries, take up to 101 KB.  (More than half an SM's 228 KB, so that
// count_lone_clusters can ask for one CTA per SM.)
constexpr size_t kMaxDynamicSmem = 120u << 10;
static_assert(1024 + 2 * kPElems * 4 + kPSignWords * 4 + 256 * kLutEntryBytes + kBlockConstMax * 8 <= kMaxDynamicSmem, "pipeline");
static_assert(1024 + (4 << 14) + (1 << 14) / 4 + 16 + 256 * kLutEntryBytes <= kMaxDynamicSmem, "tile of 2^14");
static_assert(1024 + (4 << 13) + (1 << 13) / 4 + 1024 * 16 + 256 * kLutEntryBytes <= kMaxDynamicSmem, "tile of 2^13");

// Lets a kernel use more than the default 48 KB.  The limit is the same for every launch of every kernel, so
// that no thread can lower it between another's call and its launch; what is done is remembered per kernel
// and device, and done again (to the same effect) should the table be full.
static int ensure_dynamic_smem(const void *kern)
{
    constexpr uint32_t kSlots = 2048;                  // of some 300 kernels
    static std::mutex guard;
    static const void *seen_kern[kSlots];
    static int seen_dev[kSlots];
    static uint32_t used = 0;
    int dev = 0;
    THC_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(guard);
    uint32_t slot = (uint32_t)((reinterpret_cast<uintptr_t>(kern) >> 4) * 0x9E3779B9u + (uint32_t)dev) % kSlots;
    while (seen_kern[slot] != nullptr) {               // never full: a quarter stays free
        if (seen_kern[slot] == kern && seen_dev[slot] == dev) return THC_OK;
        slot = (slot + 1u) % kSlots;
    }
    THC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynamicSmem));
    if (used < kSlots / 4 * 3) { seen_kern[slot] = kern; seen_dev[slot] = dev; ++used; }
    return THC_OK;
}

// Clusters of eight CTAs that find an SM for each CTA (15 on a B200 of 148 SMs: a cluster stays within one GPC).
static cudaError_t count_lone_clusters(int sm_count, int *n)
{
    const void *kern = block_kernel(kDecompress8, 4, true, 17u);
    if (ensure_dynamic_smem(kern) != THC_OK) return g_last_cuda;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1u << block_cluster_log2(block_kind(17u));
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t shape;
    memset(&shape, 0, sizeof shape);
    shape.gridDim = dim3((unsigned)sm_count * attr.val.clusterDim.x);
    shape.blockDim = dim3((1u << block_tile_log2(block_kind(17u))) / 64u);
    shape.dynamicSmemBytes = kMaxDynamicSmem;
    shape.attrs = &attr;
    shape.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(n, kern, &shape);
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

const char *thc_version(void) { return "thc-b200 0.1 (sm_100a)"; }

const char *thc_strerror(int code)
{
    switch (code) {
    case THC_OK: return "ok";
    case THC_EINVAL: return "invalid configuration or argument";
    case THC_EUNSUPPORTED: return "unsupported configuration";
    case THC_EWORKSPACE: return "workspace too small (see thc_sizes)";
    case THC_ECUDA:
        if (g_last_cuda == cudaSuccess) return "CUDA error: context has no device";
        snprintf(g_err_text, sizeof g_err_text, "CUDA error: %s", cudaGetErrorString(g_last_cuda));
        return g_err_text;
    default: return "unknown error code";
    }
}

static int validate_config(const thc_config *c, uint32_t *acc_bits, bool *identity)
{
    if (c == nullptr) return THC_EINVAL;
    if (!(c->bits == 1 || c->bits == 2 || c->bits == 3 || c->bits == 4 || c->bits == 8)) return THC_EINVAL;
    const uint32_t levels = 1u << c->bits;
    if (c->granularity < levels - 1) return THC_EINVAL;
    if (c->granularity > 255) return THC_EUNSUPPORTED;
    if (c->table[0] != 0 || c->table[levels - 1] != c->granularity) return THC_EINVAL;
    for (uint32_t z = 0; z + 1 < levels; ++z)
        if (c->table[z + 1] <= c->table[z]) return THC_EINVAL;
    if (!(c->t_p > 0.0) || !isfinite(c->t_p)) return THC_EINVAL;
    if (c->log2_block < 3 || c->log2_block > 22) return THC_EINVAL;
    if (c->in_dtype != THC_F32 && c->in_dtype != THC_BF16) return THC_EINVAL;
    if (c->workers == 0 || c->workers > THC_MAX_WORKERS) return THC_EINVAL;
    if (c->range_mode != THC_RANGE_NORM && c->range_mode != THC_RANGE_MINMAX) return THC_EINVAL;
    if (c->range_mode == THC_RANGE_MINMAX && c->in_dtype != THC_F32) return THC_EUNSUPPORTED;
    const uint64_t max_sum = (uint64_t)c->workers * c->granularity;
    uint32_t w = c->acc_bits;
    if (w == 0) w = max_sum <= 0xFFu ? 8 : max_sum <= 0xFFFFu ? 16 : 32;
    if (!(w == 8 || w == 16 || w == 32)) return THC_EINVAL;
    if (w < 32 && max_sum > ((1ull << w) - 1)) return THC_EINVAL;
    *acc_bits = w;
    bool id = c->granularity == levels - 1;
    for (uint32_t z = 0; id && z < levels; ++z) id = c->table[z] == z;
    *identity = id;
    return THC_OK;
}

int thc_create(const thc_config *cfg, thc_ctx **out)
{
    if (out == nullptr) return THC_EINVAL;
    *out = nullptr;
    uint32_t acc_bits = 0;
    bool identity = false;
    const int rc = validate_config(cfg, &acc_bits, &identity);
    if (rc != THC_OK) return rc;
    thc_ctx *ctx = new (std::nothrow) thc_ctx;
    if (ctx == nullptr) return THC_EINVAL;
    ctx->cfg = *cfg;
    ctx->acc_bits = acc_bits;
    ctx->identity = identity;
    ctx->device = -1;
    ctx->dev = nullptr;
    ctx->sm_count = 148;
    ctx->lone_clusters = 15;
    ctx->map_cache_used = 0;
    ctx->map_cache_next = 0;
    for (auto &r : ctx->resident) r.store(0u, std::memory_order_relaxed);
    uint32_t k0 = (uint32_t)cfg->seed, k1 = (uint32_t)(cfg->seed >> 32);
    for (int r = 0; r < 10; ++r) {
        ctx->keys.k[2 * r] = k0;
        ctx->keys.k[2 * r + 1] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    const uint32_t g = cfg->granularity;
    ctx->pipeline_next = false;

    // host copy of the device block
    DeviceBlock *h = new (std::nothrow) DeviceBlock;
    if (h == nullptr) { delete ctx; return THC_EINVAL; }
    memset(h, 0, sizeof *h);
    const uint32_t levels = 1u << cfg->bits;
    for (uint32_t z = 0; z < levels; ++z) h->table[z] = cfg->table[z];
    for (uint32_t f = 0; f <= g; ++f) {
        const uint32_t ff = f < g ? f : g - 1;            // u = 1 falls in the last interval
        uint32_t z0 = 0;
        while (z0 + 1 <= levels - 2 && cfg->table[z0 + 1] <= ff) ++z0;
        const float ntf = -(float)cfg->table[z0];
        const float r16 = 65536.0f / (float)(cfg->table[z0 + 1] - cfg->table[z0]);
        uint32_t b0, b1;
        memcpy(&b0, &ntf, 4);
        memcpy(&b1, &r16, 4);
        h->lut[f] = make_uint4(b0, b1, z0, 0u);
    }

    int count = 0;
    if (cudaGetDeviceCount(&count) == cudaSuccess && count > 0) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void **>(&ctx->dev), sizeof(DeviceBlock));
        if (e == cudaSuccess) e = cudaMemcpy(ctx->dev, h, sizeof(DeviceBlock), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess && cfg->log2_block == 17) e = count_lone_clusters(ctx->sm_count, &ctx->lone_clusters);
        if (e != cudaSuccess) {
            if (ctx->dev) cudaFree(ctx->dev);
            delete h;
            delete ctx;
            return cuda_fail(e);
        }
        ctx->device = dev;
    } else {
        (void)cudaGetLastError();   // no device: host-only context
    }
    delete h;
    *out = ctx;
    return THC_OK;
}

int thc_destroy(thc_ctx *ctx)
{
    if (ctx == nullptr) return THC_OK;
    if (ctx->dev != nullptr) cudaFree(ctx->dev);
    delete ctx;
    return THC_OK;
}

static uint64_t round_up(uint64_t v, uint64_t a) { return (v + a - 1) / a * a; }

// Which blocks are held in shared memory (thc_block.cu), by size and coordinates over all workers; the others
// take the two-pass pipeline, whose chain of queue, ring and counters is all latency on a few blocks.
// Blocks up to 2^15 always.  2^16 and 2^17 as long as the clusters run side by side.  us, cluster / pipeline:
//   2^16   blocks          8           32           64           65           72           96
//          compress    8.5 / 13.2  13.6 / 18.0  20.2 / 22.1  21.1 / 22.2  24.8 / 23.2  29.0 / 24.6
//          decompress  7.3 / 11.6  12.4 / 16.3  18.7 / 20.6  19.4 / 20.7  21.1 / 21.8  29.0 / 23.1
//   (71 clusters are resident, four CTAs to an SM; from 72 on there is a second wave.  The one-call tail is the
//   exception, level at 64 and 0.6 to 1.9 us slower in clusters from 48 to 56; 2^24 coordinates 74 / 53.)
//   2^17   blocks          8           14           15           16           18           32
//          compress   12.3 / 14.9  13.3 / 18.2  13.3 / 18.2  18.6 / 18.3  19.5 / 18.5  25.4 / 22.5
//          decompress 11.3 / 14.1  12.2 / 17.4  12.2 / 17.4  17.4 / 17.3  17.9 / 17.2  22.6 / 20.8
//   (up to 15 clusters have an SM for each CTA; from 16 on two CTAs share one.  Scales + compress of 15 blocks:
//   18.7 in two calls, 21.2 as one launch of the pipeline.)
static bool block_kernel_serves(const thc_ctx *ctx, uint64_t coords)
{
    const uint32_t k = ctx->cfg.log2_block;
    return k <= 15u || (k == 16u && coords <= (1ull << 22)) || (k == 17u && coords <= (uint64_t)ctx->lone_clusters << 17);
}

// Scales and compress in one launch for blocks held in shared memory by one CTA: the gradients are read once, and the
// clusters of one CTA per worker need no memory to exchange their sums in and no wait but the hardware's.  Up to
// eight workers, the cluster size that every GPU can place; below 2^8 a thread's 64 coordinates span several blocks.
// us, two calls / one launch, 4 bits, workers x coordinates:
//                    2 x 3000    8 x 300,000  1 x 3 M      3 x 3 M      8 x 3 M      1 x 20 M     3 x 20 M     8 x 20 M
//   fp32  2^11       8.9 / 8.1   13.6 / 10.8  13.7 / 10.4  26.2 / 22.8  62.1 / 53.0  53.4 / 40.4  134 / 115    340 / 295
//         2^13       9.8 / 8.2   12.4 / 11.1  13.9 / 10.2  26.0 / 23.2  60.0 / 53.3  51.3 / 42.3  133 / 118    338 / 304
//         2^14      11.1 / 9.7   15.5 / 12.7  15.7 / 11.8  26.2 / 23.5  61.3 / 62.7  52.0 / 43.5  137 / 129    348 / 344
//   bf16  2^11       9.2 / 8.3   13.3 / 11.4  13.3 / 10.6  25.5 / 23.4  59.3 / 54.0  55.3 / 43.4  136 / 123    334 / 314
//         2^13      10.5 / 8.6   12.2 / 11.5  13.8 / 10.6  25.7 / 23.8  55.8 / 55.8  47.7 / 45.1  122 / 126    307 / 319
//         2^14      11.1 / 9.8   15.1 / 13.0  15.2 / 11.9  25.1 / 24.3  53.9 / 64.2  46.8 / 44.9  121 / 134    307 / 364
//   (bf16 has half the bytes to save; with tiles of 2^14 there are two CTAs to an SM, and fewer to cover the wait for the slowest
//   worker.)  Inputs of one wave of tiles always gain: the launch and its latency.
static bool block_scales_serve(const thc_ctx *ctx, uint64_t coords, uint32_t n)
{
    const uint32_t k = ctx->cfg.log2_block;
    if (k < kScalesMinLog2 || k > (uint32_t)kChunkLog2 || n > kScalesMaxWorkers || ctx->cfg.range_mode != THC_RANGE_NORM) return false;
    return k <= 12u || coords <= (1ull << 22) || (ctx->cfg.in_dtype == THC_F32 && (k == 13u || n <= 6u));
}

// Schedule of the persistent pipeline for `wb_count` worker-blocks of 2^k coordinates:
// how far pass B trails pass A (lag, in worker-blocks) and how many ring slots that needs.
struct PipePlan { uint32_t grid, lag, ring; };

static PipePlan plan_pipeline(const thc_ctx *ctx, uint64_t wb_count)
{
    const uint32_t k = ctx->cfg.log2_block;
    const uint64_t T = 1ull << (k - kPLog2);
    const uint64_t resident = (uint64_t)ctx->sm_count * 3;
    PipePlan p;
    const uint64_t tasks = wb_count * T * 2;
    p.grid = (uint32_t)(tasks < resident ? tasks : resident);
    // tasks in flight: per CTA one running, one handed over, and at times one being claimed
    const uint64_t inflight = resident * 5 / 2;
    uint64_t lag = (inflight + 2 * T - 1) / (2 * T) + 1;
    uint64_t ring = lag + (inflight + 2 * T - 1) / (2 * T) + 1;
    if (lag > wb_count) lag = wb_count;
    if (ring > wb_count) ring = wb_count;
    if (ring > (uint64_t)kMaxRing) {           // tiny blocks on a huge grid: shrink the window
        ring = kMaxRing;
        if (lag > ring - 2) lag = ring - 2;
    }
    p.lag = (uint32_t)lag;
    p.ring = (uint32_t)ring;
    return p;
}

// The same for the fused-scales kernel: pass B of a block can start only when all n workers'
// tiles of the block are done, so it trails by n - 1 more worker-blocks and the ring grows by
// as many slots.  Used only where that ring still fits comfortably in L2 and the per-block
// counters (160 residues) cannot alias; otherwise the caller runs prepare and compress apart.
static bool plan_pipeline_fused(const thc_ctx *ctx, uint64_t nblocks, uint32_t n, PipePlan *out)
{
    const uint32_t k = ctx->cfg.log2_block;
    // (2^16: 4 % at most)
    if (k < 17u || k > 20u || ctx->cfg.in_dtype != THC_F32 || block_kernel_serves(ctx, (nblocks * n) << k)) return false;
    if (ctx->cfg.range_mode != THC_RANGE_NORM) return false;
    const uint64_t wb_count = nblocks * n;
    PipePlan p = plan_pipeline(ctx, wb_count);
    const uint64_t window = p.ring - p.lag;
    const uint64_t lag = (uint64_t)p.lag + n - 1;
    const uint64_t ring = lag + window;
    if (ring > wb_count || ring > (uint64_t)kMaxRing) return false;
    if (((ring << k) * 4) > ((uint64_t)96 << 20)) return false;
    if ((ring + n - 1) / n + 2 > (uint64_t)kFusedBlocks) return false;
    p.lag = (uint32_t)lag;
    p.ring = (uint32_t)ring;
    *out = p;
    return true;
}

// Workspace a pipeline launch over `wb_count` worker-blocks really touches when it computes no
// scales: the ring and, behind it, one word pair per block for the exact-range keys.
static uint64_t pipeline_workspace_need(const thc_ctx *ctx, uint64_t nblocks, uint64_t wb_count)
{
    const PipePlan pl = plan_pipeline(ctx, wb_count);
    return ((uint64_t)pl.ring << ctx->cfg.log2_block) * 4 + nblocks * 8;
}

int thc_sizes(const thc_ctx *ctx, uint64_t d, uint32_t n_local, thc_sizes_t *s)
{
    if (ctx == nullptr || s == nullptr || d == 0 || n_local == 0 || n_local > THC_MAX_WORKERS)
        return THC_EINVAL;
    const uint32_t k = ctx->cfg.log2_block;
    const uint64_t B = 1ull << k;
    if (d > (1ull << 40)) return THC_EINVAL;
    memset(s, 0, sizeof *s);
    s->d_pad = round_up(d, B);
    s->nblocks = s->d_pad / B;
    s->packed_bytes = s->d_pad * ctx->cfg.bits / 8;
    s->sum_bytes = s->d_pad * ctx->acc_bits / 8;
    s->rotated_bytes = s->d_pad * 4;
    s->acc_bits = ctx->acc_bits;
    s->scales_count = ctx->cfg.range_mode == THC_RANGE_MINMAX ? 2 * s->nblocks : s->nblocks;
    const uint32_t chunk_log2 = k < (uint32_t)kChunkLog2 ? k : (uint32_t)kChunkLog2;
    const uint64_t prepare_ws = (uint64_t)n_local * (s->d_pad >> chunk_log2) * 8;
    uint64_t two_pass_ws = 0;
    if (k > (uint32_t)kChunkLog2) {
        const PipePlan pl = plan_pipeline(ctx, s->nblocks * n_local);
        two_pass_ws = (uint64_t)pl.ring * B * 4 + s->nblocks * 8;       // + range keys
        PipePlan pf;
        if (plan_pipeline_fused(ctx, s->nblocks, n_local, &pf)) {
            const uint64_t fused_ws = (uint64_t)pf.ring * B * 4 + s->nblocks * n_local * (B >> kPLog2) * 8 +
                                      s->nblocks * 8;       // ring, tile sums, per-block quantiser constants
            if (fused_ws > two_pass_ws) two_pass_ws = fused_ws;
            s->fused_scales = 1;
        }
    }
    if (block_scales_serve(ctx, s->d_pad * n_local, n_local)) s->fused_scales = 1;
    // scratch of prepare / the pipeline's ring, then the sums (thc_aggregate_decompress where it runs the two calls)
    s->workspace_bytes = round_up((prepare_ws > two_pass_ws ? prepare_ws : two_pass_ws) + 256, 256) +
                         round_up(s->sum_bytes, 256);
    return THC_OK;
}

static int check_launch_ctx(const thc_ctx *ctx)
{
    if (ctx == nullptr) return THC_EINVAL;
    if (ctx->device < 0 || ctx->dev == nullptr) { g_last_cuda = cudaSuccess; return THC_ECUDA; }
    // the context's device block, tables and counters live on the device it was created on
    int cur = -1;
    THC_CUDA(cudaGetDevice(&cur));
    if (cur != ctx->device) return THC_EINVAL;
    return THC_OK;
}

static int check_ptr_array(const void *const *arr, uint32_t n)
{
    if (arr == nullptr) return THC_EINVAL;
    for (uint32_t i = 0; i < n; ++i)
        if (arr[i] == nullptr || !aligned16(arr[i])) return THC_EINVAL;
    return THC_OK;
}

int thc_prepare(thc_ctx *ctx, const void *const *grads, uint32_t n, uint64_t d, float *scales,
                void *workspace, uint64_t workspace_bytes, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, n, &sz)) != THC_OK) return rc;
    if ((rc = check_ptr_array(grads, n)) != THC_OK) return rc;
    if (scales == nullptr || workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
    if (workspace_bytes < sz.workspace_bytes) return THC_EWORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t k = ctx->cfg.log2_block;
    if (ctx->cfg.range_mode == THC_RANGE_MINMAX) return THC_EUNSUPPORTED;   // thc_prepare_minmax
    PtrArray in;
    memset(&in, 0, sizeof in);
    for (uint32_t i = 0; i < n; ++i) in.p[i] = grads[i];
    const double t_p = ctx->cfg.t_p;
    const bool bf16 = ctx->cfg.in_dtype == THC_BF16;
    if (k <= (uint32_t)kSmallPrepLog2) {
        const uint64_t tiles = (sz.d_pad + (1u << kSmallPrepLog2) - 1) >> kSmallPrepLog2;
        if (tiles > 0x7FFFFFFFull) return THC_EUNSUPPORTED;
        if (bf16) THC_CUDA(launch_after(prepare_small_kernel<true>, dim3((unsigned)tiles), kThreads, 0, st, in, n, d, sz.d_pad, k, t_p, scales, ctx->dev));
        else THC_CUDA(launch_after(prepare_small_kernel<false>, dim3((unsigned)tiles), kThreads, 0, st, in, n, d, sz.d_pad, k, t_p, scales, ctx->dev));
        return THC_OK;
    }
    const uint32_t chunk_log2 = k < (uint32_t)kChunkLog2 ? k : (uint32_t)kChunkLog2;
    const uint64_t chunks_per_worker = sz.d_pad >> chunk_log2;
    const uint32_t chunks_per_block = 1u << (k - chunk_log2);
    if (chunks_per_worker > 0x7FFFFFFFull) return THC_EUNSUPPORTED;
    double *partial = static_cast<double *>(workspace);
    uint32_t *counters = sz.nblocks <= (uint64_t)kPrepCounters ? ctx->dev->prep_counters : nullptr;
    const dim3 grid((unsigned)chunks_per_worker, n);
    if (bf16)
        THC_CUDA(launch_after(prepare_partial_kernel<true>, grid, kThreads, 0, st, in, d, chunk_log2, chunks_per_worker, partial, counters,
                                                                chunks_per_block, t_p, k, scales, ctx->dev));
    else
        THC_CUDA(launch_after(prepare_partial_kernel<false>, grid, kThreads, 0, st, in, d, chunk_log2, chunks_per_worker, partial, counters,
                                                                 chunks_per_block, t_p, k, scales, ctx->dev));
    if (counters == nullptr) {
        THC_CUDA(launch_after(prepare_final_kernel, dim3((unsigned)((sz.nblocks + 3) / 4)), 128, 0, st,
            partial, n, sz.nblocks, chunks_per_block, chunks_per_worker, t_p, k, scales, ctx->dev));
    }
    return THC_OK;
}

// ---- persistent pipeline dispatch (RHT blocks of 2^16 .. 2^22 coordinates that block_kernel_serves leaves; 2^15 only
// after thc_debug_skip_tasks)
typedef void (*pipe_kernel_t)(const TmaMaps, PipeParams, PtrArrayP, MutPtrArrayP, MutPtrArrayP, PhiloxKeys);

template <int MODE, int KB>
static pipe_kernel_t pick_pipe_kernel_kb(uint32_t bits, bool identity)
{
    if constexpr (MODE == kRangeF32) {
        return thc_pipeline_kernel<MODE, 4, true, KB>;
    } else if constexpr (MODE == kAggDecompress) {
        return thc_pipeline_kernel<MODE, 4, true, KB>;     // one launch only for 4-bit indices (see the entry point)
    } else if constexpr (MODE == kErrorFeedback) {
        switch (bits) {
        case 1: return thc_pipeline_kernel<MODE, 1, true, KB>;
        case 2: return thc_pipeline_kernel<MODE, 2, true, KB>;
        case 3: return thc_pipeline_kernel<MODE, 3, true, KB>;
        case 4: return thc_pipeline_kernel<MODE, 4, true, KB>;
        default: return thc_pipeline_kernel<MODE, 8, true, KB>;
        }
    } else if constexpr (MODE != kCompressF32 && MODE != kCompressBF16 && MODE != kCompressF32Fused) {
        return thc_pipeline_kernel<MODE, 4, true, KB>;
    } else {
        switch (bits) {
        case 1: return identity ? thc_pipeline_kernel<MODE, 1, true, KB> : thc_pipeline_kernel<MODE, 1, false, KB>;
        case 2: return identity ? thc_pipeline_kernel<MODE, 2, true, KB> : thc_pipeline_kernel<MODE, 2, false, KB>;
        case 3: return identity ? thc_pipeline_kernel<MODE, 3, true, KB> : thc_pipeline_kernel<MODE, 3, false, KB>;
        case 4: return identity ? thc_pipeline_kernel<MODE, 4, true, KB> : thc_pipeline_kernel<MODE, 4, false, KB>;
        default: return thc_pipeline_kernel<MODE, 8, true, KB>;      // (the only table, see validate_config)
        }
    }
}

// The 2^20-coordinate block (the paper's 4 MB partition) gets the compile-time geometry in every mode.
template <int MODE>
static pipe_kernel_t pick_pipe_kernel(uint32_t bits, bool identity, uint32_t k)
{
    if constexpr (MODE == kCompressF32 || MODE == kCompressBF16) {
        // 2^21 and 2^22: geometry at compile time, pass B in two rounds (pass_b_low5, pass_b_high4).  4-bit
        // indices only, the width of the configurations with such blocks.  The others would gain as
        // much (4 x 2^26 fp32 coordinates, us: 2^21 b = 2 754 -> 638, b = 8 880 -> 786; 2^22 785 -> 674, 924 -> 833)
        // and their 32 kernels would take a build from 131 to 164 s.
        if (k == 21 && bits == 4)
            return identity ? thc_pipeline_kernel<MODE, 4, true, 8> : thc_pipeline_kernel<MODE, 4, false, 8>;
        if (k == 22 && bits == 4)
            return identity ? thc_pipeline_kernel<MODE, 4, true, 9> : thc_pipeline_kernel<MODE, 4, false, 9>;
    }
    return k == 20 ? pick_pipe_kernel_kb<MODE, 7>(bits, identity)
                   : pick_pipe_kernel_kb<MODE, 0>(bits, identity);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda).
typedef CUresult (*encode_tiled_t)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                   const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static encode_tiled_t get_encode_tiled()
{
    static const encode_tiled_t fn = []() -> encode_tiled_t {     // initialised once, thread-safe
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<encode_tiled_t>(p);
        return nullptr;
    }();
    return fn;
}

// A 2-D map over `rows` rows of `cols` 32-bit words (row pitch in bytes), box box_cols x
// box_rows (32 columns with the 128-byte swizzle, 16 with the 64-byte one).  The data type is
// UINT32 so that bits travel unchanged.
// With box_groups > 0 the rows are seen as cols / 32 groups of 32 words and the map is 3-D
// (word in group, group, row) with a box of 32 x box_groups x box_rows: one copy then brings
// box_rows rows of 32 * box_groups words each, and they land densely, row after row, in the
// 128-byte swizzle (16-byte chunk c at c ^ ((c >> 3) & 7)).
static int encode_map(CUtensorMap *map, const void *base, uint64_t cols, uint64_t rows,
                      uint64_t pitch_bytes, uint32_t box_rows, uint32_t box_cols = 32u, bool half_words = false,
                      uint32_t box_groups = 0u)
{
    encode_tiled_t enc = get_encode_tiled();
    if (enc == nullptr) return THC_ECUDA;
    if (box_groups != 0u) {
        const cuuint64_t dims3[3] = {32u, cols / 32u, rows};
        const cuuint64_t strides3[2] = {128u, pitch_bytes};
        const cuuint32_t box3[3] = {32u, box_groups, box_rows};
        const cuuint32_t estr3[3] = {1u, 1u, 1u};
        const CUresult r3 = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void *>(base), dims3, strides3,
                                box3, estr3, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        return r3 == CUDA_SUCCESS ? THC_OK : THC_ECUDA;
    }
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {pitch_bytes};
    const cuuint32_t box[2] = {box_cols, box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    // 16-bit elements (bf16 gradients as rows of 32: 64 bytes) or 32-bit words; rows of 64
    // bytes take the 64-byte swizzle
    const bool rows64 = half_words ? box_cols == 32u : box_cols == 16u;
    const CUresult r = enc(map, half_words ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_UINT32, 2,
                           const_cast<void *>(base), dims, strides,
                           box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           rows64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? THC_OK : THC_ECUDA;
}

// encode_map through the context's cache.
static int cached_map(const thc_ctx *ctx, CUtensorMap *map, const void *base, uint64_t cols, uint64_t rows,
                      uint64_t pitch_bytes, uint32_t box_rows, uint32_t box_cols = 32u, bool half_words = false,
                      uint32_t box_groups = 0u)
{
    std::lock_guard<std::mutex> lock(ctx->map_mutex);
    for (int i = 0; i < ctx->map_cache_used; ++i) {
        const thc_ctx::MapEntry &e = ctx->map_cache[i];
        if (e.base == base && e.cols == cols && e.rows == rows && e.pitch == pitch_bytes && e.box_rows == box_rows &&
            e.box_cols == box_cols && e.half == (half_words ? 1u : 0u) && e.groups == box_groups) {
            *map = e.map;
            return THC_OK;
        }
    }
    const int rc = encode_map(map, base, cols, rows, pitch_bytes, box_rows, box_cols, half_words, box_groups);
    if (rc != THC_OK) return rc;
    int slot = ctx->map_cache_used < thc_ctx::kMapCache ? ctx->map_cache_used++ : ctx->map_cache_next;
    ctx->map_cache_next = (slot + 1) % thc_ctx::kMapCache;
    thc_ctx::MapEntry &e = ctx->map_cache[slot];
    e.base = base; e.cols = cols; e.rows = rows; e.pitch = pitch_bytes; e.box_rows = box_rows; e.box_cols = box_cols;
    e.half = half_words ? 1u : 0u; e.groups = box_groups; e.map = *map;
    return THC_OK;
}

static int launch_pipeline(thc_ctx *ctx, pipe_kernel_t kern, bool compress_f32,
                           const thc_sizes_t &sz, uint64_t d, uint32_t n_local, uint32_t worker_base, uint32_t round, uint32_t divisor,
                           const float *scales, void *workspace, const PtrArrayP &in,
                           const MutPtrArrayP &out, const MutPtrArrayP &rot, cudaStream_t st,
                           float *fused_scales_out = nullptr, bool compress_bf16 = false, uint32_t agg_n = 0,
                           uint32_t *range_keys = nullptr, float *range_out = nullptr)
{
    const uint32_t k = ctx->cfg.log2_block;
    PipeParams P;
    memset(&P, 0, sizeof P);
    P.d = d;
    P.d_pad = sz.d_pad;
    P.wb_count = sz.nblocks * n_local;
    const uint64_t T = 1ull << (k - kPLog2);
    P.total_tasks = P.wb_count * T * 2;
    if (P.wb_count >= 0x7FFFFFFFull || P.total_tasks >= 0x7FFFFFFFull) return THC_EUNSUPPORTED;
    PipePlan pl = plan_pipeline(ctx, P.wb_count);
    // Compress of 2^22 blocks: pass B trails by two worker-blocks in a ring of four slots
    // (64 MB stay in L2 better than the planned six slots of 16 MB; the workspace holds those).
    if ((compress_f32 || compress_bf16) && k == 22 && pl.ring > 4) { pl.lag = 2; pl.ring = 4; }
    if (fused_scales_out != nullptr) {
        if (!plan_pipeline_fused(ctx, sz.nblocks, n_local, &pl)) return THC_EUNSUPPORTED;
        P.tile_sq = reinterpret_cast<double *>(static_cast<unsigned char *>(workspace) +
                                               ((uint64_t)pl.ring << k) * 4);
        P.fused_const = reinterpret_cast<float2 *>(P.tile_sq + P.wb_count * T);
        P.scales_out = fused_scales_out;
        P.t_p = ctx->cfg.t_p;
    }
    P.ring = static_cast<float *>(workspace);
    P.scales = scales;
    P.dev = ctx->dev;
    P.k = k;
    P.kb = k - kPLog2;
    P.n_local = n_local;
    P.lag = pl.lag;
    P.ring_slots = pl.ring;
    P.granularity = ctx->cfg.granularity;
    P.divisor = divisor;
    P.round = round;
    P.worker_base = worker_base;
    P.c_block = (float)(1.0 / sqrt((double)(1ull << k)));
    P.exact_range = ctx->cfg.range_mode == THC_RANGE_MINMAX ? 1u : 0u;
    P.nblocks = (uint32_t)sz.nblocks;
    P.agg_n = agg_n;
    P.agg_acc_bits = ctx->acc_bits;
    P.range_keys = range_keys;
    P.range_out = range_out;
    const uint64_t nblk_cached = sz.nblocks < (uint64_t)kBlockConstMax ? sz.nblocks : (uint64_t)kBlockConstMax;
    const size_t smem = (size_t)1024 + (size_t)2 * kPElems * 4 + kPSignWords * 4 +
                        (size_t)(ctx->cfg.granularity + 1) * kLutEntryBytes + (size_t)nblk_cached * 8;
    { const int rc = ensure_dynamic_smem(reinterpret_cast<const void *>(kern)); if (rc != THC_OK) return rc; }
    // Tensor maps: the ring (pass-B panels are fetched by TMA at every block size) and, for fp32 compress, every
    // worker's gradient viewed as rows of 32 floats (whole rows only; a ragged last tile is
    // loaded by the compute warps).
    TmaMaps maps;
    memset(&maps, 0, sizeof maps);
    P.b_swz_mask = 7u;
    if (k == 20) {
        const int rc = cached_map(ctx, &maps.ring, workspace, (uint64_t)kPElems,
                                  (uint64_t)pl.ring << (k - kPLog2), (uint64_t)kPElems * 4, 128u);
        if (rc != THC_OK) return rc;
    } else if (k == 22) {
        // panels of 512 rows x 16 columns: boxes of 16 x 256, 64-byte swizzle
        const int rc = cached_map(ctx, &maps.ring, workspace, (uint64_t)kPElems,
                                  (uint64_t)pl.ring << (k - kPLog2), (uint64_t)kPElems * 4, 256u, 16u);
        if (rc != THC_OK) return rc;
        P.b_swz_mask = 3u;
        P.b_tma = 2u;
    } else if (k == 21) {
        const int rc = cached_map(ctx, &maps.ring, workspace, (uint64_t)kPElems,
                                  (uint64_t)pl.ring << (k - kPLog2), (uint64_t)kPElems * 4, 256u);
        if (rc != THC_OK) return rc;
        P.b_tma = 1u;
    } else {
        // k = 15 .. 19: panels of 2^(k-13) rows x 2^(26-k) columns, one 3-D box each
        const uint32_t kb = k - kPLog2;
        const int rc = cached_map(ctx, &maps.ring, workspace, (uint64_t)kPElems,
                                  (uint64_t)pl.ring << kb, (uint64_t)kPElems * 4, 1u << kb, 32u, false, 1u << (8u - kb));
        if (rc != THC_OK) return rc;
        P.b_tma = 3u;
    }
    if (compress_f32 && (d >> 5) >= 256) {
        for (uint32_t i = 0; i < n_local; ++i) {
            const int rc = cached_map(ctx, &maps.in[i], in.p[i], 32u, d >> 5, 128u, 256u);
            if (rc != THC_OK) return rc;
        }
    }
    if (compress_bf16 && (d >> 5) >= 256) {
        for (uint32_t i = 0; i < n_local; ++i) {
            const int rc = cached_map(ctx, &maps.in[i], in.p[i], 32u, d >> 5, 64u, 256u, 32u, true);
            if (rc != THC_OK) return rc;
        }
    }
    THC_CUDA(launch_after(kern, dim3(pl.grid), kPCtaThreads, smem, st, maps, P, in, out, rot, ctx->keys));
    ctx->pipeline_next = false;
    return THC_OK;
}

// ---- blocks held in shared memory (see block_kernel_serves).  Blocks of up to 2^14 have no other kernel: for
// them thc_sizes reserves no ring, and below 2^13 the pipeline has no tile.
static bool use_block_kernel(const thc_ctx *ctx, uint64_t coords)
{
    const uint32_t k = ctx->cfg.log2_block;
    return k <= (uint32_t)kChunkLog2 || (!ctx->pipeline_next && block_kernel_serves(ctx, coords));
}

// CTAs (clusters) of a block kernel that the GPU holds at a time.  A tile of 2^13 with
// a table of more than 167 entries leaves room for three CTAs per SM instead of four: with 592 CTAs in the grid,
// each with a fixed share of the tasks, a quarter of them started when others had ended.  Compress with a 4-bit
// table of 256 entries, 592 against 444 CTAs: 4 x 2^22 coordinates in blocks of 2^12 37.7 -> 34.5 us, 4 x 2^24
// 123.7 -> 117.6, 8 x 3,000,001 in blocks of 2^13 50.7 -> 47.1; over 448 .. 3500 tiles 22 % faster to 5 % slower
// (near 700 and 1000 tiles, where 592 leave the shorter last round).  Of clusters of eight there are fewer than the
// SMs have room for, since a cluster stays within one GPC (2^16: 48 with such a table: 4 x 2^20 coordinates 28.1 -> 24.5 us).
// The runtime is asked where shared memory leaves less room than the kernel's registers do (four CTAs
// or two) and for the clusters of scales + compress, whose number depends on the workers: that adds some 0.5 us to a
// context's first call.  Elsewhere no more clusters are launched than there are (block_kernel_serves).
constexpr size_t kSmemPerSm = 228u << 10, kSmemPerCta = 1024u + 256u;     // reserved and static
static int resident_units(const thc_ctx *ctx, uint32_t entry, const void *kern, const cudaLaunchConfig_t &shape, uint32_t cluster, uint32_t *units)
{
    const uint32_t by_registers = shape.blockDim.x == 128u ? 4u : 2u;
    *units = (uint32_t)ctx->sm_count * by_registers / cluster;
    if (entry < (uint32_t)kPipeModes && shape.dynamicSmemBytes + kSmemPerCta <= kSmemPerSm / by_registers) return THC_OK;
    *units = ctx->resident[entry].load(std::memory_order_relaxed);
    if (*units != 0u) return THC_OK;
    int n = 0;
    if (cluster == 1u) {
        THC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, (int)shape.blockDim.x, shape.dynamicSmemBytes));
        n *= ctx->sm_count;
    } else {
        THC_CUDA(cudaOccupancyMaxActiveClusters(&n, kern, &shape));
    }
    *units = n > 0 ? (uint32_t)n : 1u;
    ctx->resident[entry].store(*units, std::memory_order_relaxed);
    return THC_OK;
}

// lut_bytes: table space in shared memory; keys: exact-range mode; agg_n: aggregate + decompress; scales_out: scales and
// compress in one launch.
static int launch_block(const thc_ctx *ctx, const void *kern, PipeMode mode, size_t lut_bytes, const thc_sizes_t &sz,
                        uint64_t d, uint32_t n_local, uint32_t worker_base, uint32_t round, uint32_t divisor,
                        const float *scales, const PtrArrayP &in, const MutPtrArrayP &out, const MutPtrArrayP &rot,
                        cudaStream_t st, uint32_t *keys = nullptr, uint32_t agg_n = 0, float *range_out = nullptr,
                        float *scales_out = nullptr)
{
    const uint32_t k = ctx->cfg.log2_block;
    BlockParams P;
    memset(&P, 0, sizeof P);
    const uint32_t tile_log2 = block_tile_log2(block_kind(k)), e = block_cluster_log2(block_kind(k));
    const size_t tile = (size_t)1 << tile_log2;
    const uint64_t units = e != 0u ? sz.nblocks : (sz.d_pad + tile - 1) >> tile_log2;
    if ((units << e) * n_local >= 0x7FFFFFFFull || sz.nblocks >= 0xFFFFFFFFull) return THC_EUNSUPPORTED;
    P.d = d;
    P.d_pad = sz.d_pad;
    P.scales = scales;
    P.dev = ctx->dev;
    P.tasks = (uint32_t)(scales_out != nullptr ? units : units * n_local);
    P.scales_out = scales_out;
    P.t_p = ctx->cfg.t_p;
    P.sqrt_block = sqrt((double)(1ull << k));
    P.n_local = n_local;
    P.k = k;
    P.granularity = ctx->cfg.granularity;
    P.divisor = divisor;
    P.round = round;
    P.worker_base = worker_base;
    P.c_block = (float)(1.0 / sqrt((double)(1ull << k)));
    P.exact_range = ctx->cfg.range_mode == THC_RANGE_MINMAX ? 1u : 0u;
    P.nblocks = (uint32_t)sz.nblocks;
    P.const_slots = k < tile_log2 ? 1u << (tile_log2 - k) : 1u;
    P.range_keys = keys;
    P.range_out = range_out;
    P.exited = &reinterpret_cast<PipeCounters *>(ctx->dev->counters)->exited;
    P.agg_n = agg_n;
    P.agg_chunk = 255u / ctx->cfg.granularity;
    P.agg_acc_bits = ctx->acc_bits;
    const size_t smem = (size_t)1024 + tile * 4 + tile / 4 + (size_t)P.const_slots * 16 + lut_bytes;
    { const int rc = ensure_dynamic_smem(kern); if (rc != THC_OK) return rc; }
    TmaMaps maps;
    if ((d >> 5) >= 256) {
        for (uint32_t i = 0; i < n_local; ++i) {
            int rc = THC_OK;
            if (mode == kCompressBF16 || mode == kCompressBF16Fused) rc = cached_map(ctx, &maps.in[i], in.p[i], 32u, d >> 5, 64u, 64u, 32u, true);
            else if (mode == kCompressF32 || mode == kCompressF32Fused || mode == kRangeF32) rc = cached_map(ctx, &maps.in[i], in.p[i], 32u, d >> 5, 128u, 256u);
            if (rc != THC_OK) return rc;
        }
    }
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    const uint32_t cluster = scales_out != nullptr ? n_local : 1u << e;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((unsigned)ctx->sm_count * 8u * cluster);
    cfg.blockDim = dim3((unsigned)(tile / 64));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = cluster != 1u ? 2 : 1;
    cudaLaunchConfig_t shape = cfg;
    shape.attrs = attr + 1;
    shape.numAttrs = 1;
    uint32_t resident = 0;
    { const int rc = resident_units(ctx, scales_out != nullptr ? kPipeModes + cluster : (uint32_t)mode,
                                                 kern, shape, cluster, &resident); if (rc != THC_OK) return rc; }
    cfg.gridDim = dim3((P.tasks < resident ? P.tasks : resident) * cluster);
    // Tasks claimed from a counter instead of dealt out in a fixed stride: the CTAs of an SM do not progress evenly,
    // and with fixed shares the mean CTA of a compress ended after four fifths of the time.  With few tasks to a CTA fixed
    // shares put the last ones on different SMs; in clusters the claim is read from the first CTA.  us, fixed / claimed,
    // 4 bits, by tasks to a CTA (cluster) that the GPU holds:
    //                               2.1          2.9          3.9          4.5          4.9          5.5          6.5          7.5
    //   tile 2^13  compress         20.7 / 22.0  26.6 / 28.5  34.1 / 33.9  38.3 / 39.9  41.5 / 42.3  45.7 / 44.8  53.4 / 53.3  60.9 / 60.2
    //              8 workers, bf16  19.5 / 20.9  25.7 / 25.8  33.4 / 33.4  37.7 / 39.4  41.6 / 43.6  45.6 / 45.1  53.4 / 54.0  61.3 / 60.8
    //   + scales   1 worker         22.7 / 23.8  29.9 / 31.9  38.8 / 38.1               47.5 / 46.5  51.4 / 52.8  60.0 / 59.1
    //              2 workers        23.7 / 25.1  31.1 / 31.9  39.8 / 39.7               48.8 / 47.5  52.0 / 53.7  61.1 / 62.3
    //              4 workers        22.9 / 24.5  31.6 / 32.8  41.1 / 42.4               50.0 / 49.2  53.0 / 55.1  65.1 / 64.2
    //              8 workers        22.9 / 24.2  31.2 / 32.5  41.0 / 42.7               50.1 / 50.4  56.3 / 55.6  65.7 / 64.6
    //                               6.5          7.5          8.5          10.5         13.5         17.5         24.5         40
    //              error feedback   66.9 / 67.8  76.5 / 76.6  86.0 / 86.0   103 / 104    130 / 130    168 / 166    234 / 228    384 / 374
    //              decompress                                 57.3 / 57.1  69.0 / 69.4  88.1 / 86.9   114 / 111    157 / 152    262 / 246
    //   tile 2^14  compress         56.0 / 53.4  63.4 / 62.4  71.3 / 67.0  86.1 / 83.6   108 / 105    138 / 132    190 / 183    303 / 296
    //              + 4 workers' scales  74.1 / 69.4  84.3 / 78.6  94.3 / 88.0
    //              error feedback   74.5 / 70.8  82.9 / 79.6  93.0 / 90.7   113 / 111    141 / 139    180 / 174    246 / 241    400 / 393
    //              decompress                                 68.4 / 69.1  83.6 / 82.1   105 / 104    135 / 132    186 / 182    302 / 290
    //   2 x 2^14   compress         78.0 / 79.0  89.3 / 91.2   100 / 104    123 / 122    157 / 155    202 / 198    282 / 275    458 / 441
    //   (cluster)  error feedback   96.2 / 98.0   111 / 112    125 / 127    152 / 155    193 / 196    248 / 250    344 / 343    561 / 550
    //              decompress                                  100 / 103    123 / 125    158 / 160    204 / 204    283 / 280    462 / 452
    //              aggregate + dec.                            101 / 104    123 / 126    158 / 162    204 / 207    284 / 284    463 / 456
    //   exact range     2^13       45.7 / 47.6               57.9 / 59.9  70.2 / 70.7  88.0 / 88.5   111 / 111    152 / 150
    //                   2^14       49.4 / 47.9               60.5 / 58.1  73.5 / 71.2  92.9 / 89.7   111 / 108    150 / 146
    //                   2 x 2^14   69.9 / 71.7               90.5 / 92.3   110 / 112    139 / 138    178 / 176    247 / 242
    const bool quantises = mode == kCompressF32 || mode == kCompressBF16, range = mode == kRangeF32;
    const uint32_t fixed = e != 0u ? (quantises || range ? 10u : 20u)
                         : tile_log2 != 13u ? 8u : scales_out != nullptr ? 6u : quantises ? 5u : range ? 16u : 8u;
    P.head = nullptr;
    if (P.tasks > (uint64_t)fixed * resident) {
        P.head = &reinterpret_cast<PipeCounters *>(ctx->dev->counters)->head;
        kern = block_kernel(mode, ctx->cfg.bits, ctx->identity, k, true);
        const int rc = ensure_dynamic_smem(kern);
        if (rc != THC_OK) return rc;
    }
    void *args[] = {&maps, &P, const_cast<PtrArrayP *>(&in), const_cast<MutPtrArrayP *>(&out), const_cast<MutPtrArrayP *>(&rot),
                    const_cast<PhiloxKeys *>(&ctx->keys)};
    THC_CUDA(cudaLaunchKernelExC(&cfg, kern, args));
    return THC_OK;
}

// Table space of a launch that quantises.
static size_t quant_lut_bytes(const thc_ctx *ctx)
{
    return ctx->identity ? 0 : (size_t)(ctx->cfg.granularity + 1) * kLutEntryBytes;
}

// thc_prepare in exact-range mode (Algorithm 1's preliminary stage on the rotated coordinates):
// one transform pass over all workers whose epilogue only takes the minimum and maximum, then
// the keys become the (lo, hi) planes of `scales`.  This costs about as much as the transform
// half of thc_compress: the price of a range that clamps nothing.
int thc_prepare_minmax(thc_ctx *ctx, const void *const *grads, uint32_t n, uint64_t d, uint32_t round,
                       float *scales, float *const *rotated, void *workspace, uint64_t workspace_bytes,
                       void *stream)
{
    int rc0 = check_launch_ctx(ctx);
    if (rc0 != THC_OK) return rc0;
    if (ctx->cfg.range_mode != THC_RANGE_MINMAX) return THC_EUNSUPPORTED;
    thc_sizes_t sz;
    if ((rc0 = thc_sizes(ctx, d, n, &sz)) != THC_OK) return rc0;
    if ((rc0 = check_ptr_array(grads, n)) != THC_OK) return rc0;
    if (scales == nullptr || workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
    if (workspace_bytes < sz.workspace_bytes) return THC_EWORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t k = ctx->cfg.log2_block;
    const bool in_block = use_block_kernel(ctx, sz.d_pad * n);
    // up to kPrepCounters blocks the keys are the context's own, zero between calls, and the last CTA
    // of the transform writes the ranges: one launch (three took 3.7 us more on 65 blocks)
    const bool own_keys = sz.nblocks <= (uint64_t)kPrepCounters;
    uint32_t *keys = own_keys ? ctx->dev->range_keys : static_cast<uint32_t *>(workspace);
    if (!own_keys) {
        if (!in_block) {
            const PipePlan pl = plan_pipeline(ctx, sz.nblocks * n);
            keys = reinterpret_cast<uint32_t *>(static_cast<unsigned char *>(workspace) + ((uint64_t)pl.ring << k) * 4);
        }
        THC_CUDA(cudaMemsetAsync(keys, 0, sz.nblocks * 8, st));
    }
    float *range_out = own_keys ? scales : nullptr;
    int rc;
    PtrArrayP pin;
    MutPtrArrayP pout, prot;
    memset(&pin, 0, sizeof pin);
    memset(&pout, 0, sizeof pout);
    memset(&prot, 0, sizeof prot);
    for (uint32_t i = 0; i < n; ++i) {
        pin.p[i] = grads[i];
        if (rotated != nullptr && rotated[i] != nullptr) {
            if (!aligned16(rotated[i])) return THC_EINVAL;
            prot.p[i] = rotated[i];
        }
    }
    if (in_block)
        rc = launch_block(ctx, block_kernel(kRangeF32, 4, true, ctx->cfg.log2_block), kRangeF32, 0, sz, d, n, 0, round, 1, scales, pin, pout,
                          prot, st, keys, 0, range_out);
    else
        rc = launch_pipeline(ctx, pick_pipe_kernel<kRangeF32>(4, true, k), true, sz, d, n, 0, round,
                             1, scales, workspace, pin, pout, prot, st, nullptr, false, 0, keys, range_out);
    if (rc != THC_OK) return rc;
    if (!own_keys) {
        THC_CUDA(launch_after(range_final_kernel, dim3((unsigned)((sz.nblocks + 255) / 256)), 256, 0, st, keys, sz.nblocks, scales, ctx->dev));
    }
    return THC_OK;
}

int thc_compress(thc_ctx *ctx, const void *const *grads, uint32_t n_local, uint32_t worker_base,
                 uint64_t d, uint32_t round, const float *scales, void *const *packed,
                 float *const *rotated, void *workspace, uint64_t workspace_bytes, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, n_local, &sz)) != THC_OK) return rc;
    if ((rc = check_ptr_array(grads, n_local)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n_local)) != THC_OK) return rc;
    if (scales == nullptr) return THC_EINVAL;
    if ((uint64_t)worker_base + n_local > 0xFFFFFFFFull) return THC_EINVAL;
    const uint32_t k = ctx->cfg.log2_block;
    if (k > (uint32_t)kChunkLog2) {
        if (workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
        if (workspace_bytes < sz.workspace_bytes) return THC_EWORKSPACE;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PtrArrayP in;
    MutPtrArrayP out, rot;
    memset(&in, 0, sizeof in);
    memset(&out, 0, sizeof out);
    memset(&rot, 0, sizeof rot);
    for (uint32_t i = 0; i < n_local; ++i) {
        in.p[i] = grads[i];
        out.p[i] = packed[i];
        if (rotated != nullptr && rotated[i] != nullptr) {
            if (!aligned16(rotated[i])) return THC_EINVAL;
            rot.p[i] = rotated[i];
        }
    }
    const bool bf16 = ctx->cfg.in_dtype == THC_BF16;
    if (use_block_kernel(ctx, sz.d_pad * n_local)) {
        const void *kern = bf16 ? block_kernel(kCompressBF16, ctx->cfg.bits, ctx->identity, ctx->cfg.log2_block)
                                   : block_kernel(kCompressF32, ctx->cfg.bits, ctx->identity, ctx->cfg.log2_block);
        return launch_block(ctx, kern, bf16 ? kCompressBF16 : kCompressF32, quant_lut_bytes(ctx), sz, d, n_local, worker_base,
                            round, 1, scales, in, out, rot, st);
    }
    pipe_kernel_t kern = bf16 ? pick_pipe_kernel<kCompressBF16>(ctx->cfg.bits, ctx->identity, k)
                              : pick_pipe_kernel<kCompressF32>(ctx->cfg.bits, ctx->identity, k);
    return launch_pipeline(ctx, kern, !bf16, sz, d, n_local, worker_base, round, 1, scales, workspace,
                           in, out, rot, st, nullptr, bf16);
}

// Scales and compress in one launch (see thc.h).  Falls back to the two separate calls where
// the fused kernel does not apply.
int thc_prepare_compress(thc_ctx *ctx, const void *const *grads, uint32_t n, uint32_t worker_base,
                         uint64_t d, uint32_t round, float *scales, void *const *packed,
                         float *const *rotated, void *workspace, uint64_t workspace_bytes, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, n, &sz)) != THC_OK) return rc;
    PipePlan pf;
    const bool in_block = block_scales_serve(ctx, sz.d_pad * n, n);
    if (!in_block && !plan_pipeline_fused(ctx, sz.nblocks, n, &pf)) {
        rc = thc_prepare(ctx, grads, n, d, scales, workspace, workspace_bytes, stream);
        if (rc != THC_OK) return rc;
        return thc_compress(ctx, grads, n, worker_base, d, round, scales, packed, rotated, workspace,
                            workspace_bytes, stream);
    }
    if ((rc = check_ptr_array(grads, n)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n)) != THC_OK) return rc;
    if (scales == nullptr || workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
    if ((uint64_t)worker_base + n > 0xFFFFFFFFull) return THC_EINVAL;
    if (workspace_bytes < sz.workspace_bytes) return THC_EWORKSPACE;
    PtrArrayP pin;
    MutPtrArrayP pout, prot;
    memset(&pin, 0, sizeof pin);
    memset(&pout, 0, sizeof pout);
    memset(&prot, 0, sizeof prot);
    for (uint32_t i = 0; i < n; ++i) {
        pin.p[i] = grads[i];
        pout.p[i] = packed[i];
        if (rotated != nullptr && rotated[i] != nullptr) {
            if (!aligned16(rotated[i])) return THC_EINVAL;
            prot.p[i] = rotated[i];
        }
    }
    if (in_block) {
        const PipeMode mode = ctx->cfg.in_dtype == THC_BF16 ? kCompressBF16Fused : kCompressF32Fused;
        return launch_block(ctx, block_kernel(mode, ctx->cfg.bits, ctx->identity, ctx->cfg.log2_block), mode, quant_lut_bytes(ctx), sz, d, n,
                            worker_base, round, 1, scales, pin, pout, prot, static_cast<cudaStream_t>(stream), nullptr, 0, nullptr, scales);
    }
    pipe_kernel_t kern = ctx->cfg.log2_block == 20 ? pick_pipe_kernel_kb<kCompressF32Fused, 7>(ctx->cfg.bits, ctx->identity)
                                                    : pick_pipe_kernel_kb<kCompressF32Fused, 0>(ctx->cfg.bits, ctx->identity);
    return launch_pipeline(ctx, kern, true, sz, d, n, worker_base, round, 1, scales, workspace, pin, pout,
                           prot, static_cast<cudaStream_t>(stream), scales);
}

int thc_decompress(thc_ctx *ctx, const void *sum, uint32_t divisor, uint64_t d, uint32_t round,
                   const float *scales, float *outp, void *workspace, uint64_t workspace_bytes,
                   void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, 1, &sz)) != THC_OK) return rc;
    if (sum == nullptr || outp == nullptr || scales == nullptr || divisor == 0) return THC_EINVAL;
    if (!aligned16(sum) || !aligned16(outp)) return THC_EINVAL;
    const uint32_t k = ctx->cfg.log2_block;
    if (k > (uint32_t)kChunkLog2) {
        if (workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
        if (workspace_bytes < pipeline_workspace_need(ctx, sz.nblocks, sz.nblocks)) return THC_EWORKSPACE;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t w = ctx->acc_bits;
    PtrArrayP pin;
    MutPtrArrayP pout, prot;
    memset(&pin, 0, sizeof pin);
    memset(&pout, 0, sizeof pout);
    memset(&prot, 0, sizeof prot);
    pin.p[0] = sum;
    pout.p[0] = outp;
    if (use_block_kernel(ctx, sz.d_pad)) {
        const void *kern = w == 8 ? block_kernel(kDecompress8, 4, true, ctx->cfg.log2_block)
                            : w == 16 ? block_kernel(kDecompress16, 4, true, ctx->cfg.log2_block)
                                      : block_kernel(kDecompress32, 4, true, ctx->cfg.log2_block);
        return launch_block(ctx, kern, w == 8 ? kDecompress8 : w == 16 ? kDecompress16 : kDecompress32, 0, sz, d, 1, 0, round,
                            divisor, scales, pin, pout, prot, st);
    }
    pipe_kernel_t kern = w == 8 ? pick_pipe_kernel<kDecompress8>(4, true, k)
                       : w == 16 ? pick_pipe_kernel<kDecompress16>(4, true, k)
                                 : pick_pipe_kernel<kDecompress32>(4, true, k);
    return launch_pipeline(ctx, kern, false, sz, d, 1, 0, round, divisor, scales, workspace, pin, pout,
                           prot, st);
}

// thc_aggregate followed by thc_decompress in one launch for the simulated cluster, whose workers'
// packed indices all sit in this GPU's memory (Algorithm 2: the PS line Y = sum_i T[Z_i] feeding
// the worker's estimate line and the inverse RHT): pass A of the inverse transform adds up the
// table values itself, so the sums need not travel through HBM; they are written only on request.
// Whether the two calls are faster where the sums are wanted too: a thread's first round waits for the indices of all
// workers, some at a time, and the pipeline and the tiles of 2^14 have fewer threads to cover that.  Two launches win
// where the tail is latency (few tiles) and where many workers' loads queue up, one launch where the tiles fill the
// GPU once.  (Pipeline, up to 2^24 coordinates: the two cross between 12 and 17 workers, by up to 4 % either way at 13
// to 16; the line is 12 for all of them.)  us, two calls / one:
//                     4 workers    8            13           14           16           17           20           24           32
//   2^ 8  3000        6.7 / 4.9    6.7 / 5.6                              7.3 / 6.9                              8.8 / 8.3    10.2 / 9.8
//   2^12  2^22       13.3 / 10.5  13.7 / 11.4                            19.2 / 15.9                            24.1 / 20.2   29.0 / 24.7
//   2^14  2^20        9.3 / 8.5    9.9 / 9.5   11.4 / 11.7  11.5 / 12.1  11.7 / 12.2  12.6 / 13.0  12.9 / 13.6  13.4 / 14.6   15.1 / 17.0
//         2^22       14.0 / 11.6  15.2 / 13.2  20.1 / 16.8  20.4 / 17.6  20.9 / 18.1  23.7 / 19.4  24.2 / 20.6  25.6 / 22.4   30.4 / 26.3
//         2^24       46.1 / 40.7  48.3 / 48.5  69.6 / 62.9  70.8 / 66.1  73.0 / 68.4  80.9 / 73.5  83.0 / 80.5  87.5 / 90.0    101 / 115
//         2^26        155 / 137    164 / 162    243 / 209    246 / 220    259 / 230    289 / 242    301 / 262    323 / 301     383 / 397
//   2^15  2^20       12.3 / 11.6  12.8 / 12.6  14.5 / 14.8  14.7 / 15.3  14.9 / 15.3  15.8 / 16.1  16.0 / 16.6  16.5 / 17.7   18.2 / 20.1
//         2^22       19.3 / 16.1  20.2 / 17.5  25.1 / 21.0  25.4 / 21.6  26.1 / 22.3  28.7 / 23.5  29.3 / 24.7  30.7 / 26.2   35.6 / 30.3
//         2^24       55.8 / 50.0  58.0 / 58.1  81.3 / 72.0  82.8 / 75.2  84.8 / 76.0  93.1 / 80.7  94.5 / 85.0  98.7 / 95.1    112 / 119
//   2^16  2^20       13.2 / 12.5  13.8 / 13.3  15.3 / 14.9  15.4 / 15.3  15.6 / 15.3  16.6 / 15.8  16.9 / 16.4  17.3 / 17.4   18.9 / 19.4   (clusters)
//   2^17  2^20       13.7 / 14.0  14.3 / 15.0  16.2 / 17.1  16.4 / 17.7  16.6 / 17.7  17.5 / 18.5  17.8 / 19.0  18.3 / 20.0   19.9 / 22.4   (clusters)
//         11 blocks  15.2 / 14.8  15.6 / 15.7  18.0 / 18.0  18.1 / 18.5  18.2 / 18.6  19.7 / 19.4  19.8 / 19.9  20.2 / 21.0   22.1 / 23.4
//         15 blocks  15.6 / 14.9  16.1 / 15.9  18.5 / 18.2  18.6 / 18.7  18.9 / 18.7  20.2 / 19.5  20.5 / 20.0  21.1 / 21.1   23.9 / 23.5
//   2^16  2^24       62.5 / 55.8  64.9 / 62.8  83.1 / 80.1  84.2 / 82.6  86.8 / 88.8  94.7 / 94.6  96.4 / 104    101 / 117     115 / 143   (pipeline)
//   2^18  2^26        205 / 194    215 / 218    288 / 284    293 / 291    304 / 312    330 / 329    338 / 360    358 / 405     408 / 499
//   2^20  2^22       26.3 / 23.7  26.8 / 25.5  31.4 / 30.2  31.9 / 31.1  32.5 / 32.3  35.8 / 34.3  36.1 / 37.2  38.5 / 42.0   42.9 / 52.7
//         25.6 M     86.8 / 75.7  90.8 / 86.5   120 / 115    122 / 118    126 / 127    138 / 136    141 / 148    149 / 166     171 / 202
//   2^21  2^24       67.5 / 58.7  70.0 / 67.2  88.2 / 89.2  89.0 / 92.3  92.0 / 99.0  99.3 / 105    102 / 113    106 / 125     120 / 150
//         2^26        236 / 211    247 / 238    315 / 304    318 / 309    329 / 328    358 / 346    366 / 369    384 / 406     439 / 497
//   2^22  2^24       75.5 / 64.6  77.5 / 72.0  95.4 / 92.7  96.1 / 96.2  99.0 / 103    107 / 109    109 / 118    113 / 130     128 / 152
//         2^26        271 / 235    282 / 255    349 / 313    353 / 322    365 / 342    392 / 361    399 / 387    417 / 429     472 / 524
static bool two_call_tail(const thc_ctx *ctx, uint64_t d_pad, uint32_t n)
{
    const uint32_t k = ctx->cfg.log2_block;
    if (use_block_kernel(ctx, d_pad)) {
        if (k == 14u || k == 15u) return d_pad <= (1ull << 20) ? n > 16u : d_pad > (1ull << 22) && n > 24u;
        return k == 17u && (d_pad <= 9ull << 17 || n > 13u);
    }
    return n > (d_pad <= (1ull << 24) ? 12u : k == 22u ? 18u : 14u);
}

int thc_aggregate_decompress(thc_ctx *ctx, const void *const *packed, uint32_t n, uint64_t d, uint32_t round,
                             const float *scales, float *outp, void *sum_or_null, void *workspace,
                             uint64_t workspace_bytes, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    if (n == 0 || n > ctx->cfg.workers) return THC_EINVAL;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, 1, &sz)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n)) != THC_OK) return rc;
    if (outp == nullptr || scales == nullptr || !aligned16(outp)) return THC_EINVAL;
    if (sum_or_null != nullptr && !aligned16(sum_or_null)) return THC_EINVAL;
    const uint32_t k = ctx->cfg.log2_block;
    // index widths without the byte-lane look-up (there the one launch is slower than the two), and see
    // two_call_tail: the sums go to the caller's buffer or take the end of the workspace
    const bool two_calls = ctx->cfg.bits != 4 || ctx->cfg.granularity >= 128 || sz.d_pad % 32 != 0 ||
                           (sum_or_null != nullptr && two_call_tail(ctx, sz.d_pad, n));
    // What is refused is refused before the first launch.  Without a buffer room for the sums is asked for where
    // the one launch needs no workspace too: the same rule for all configurations.
    uint64_t ws_left = workspace_bytes;
    if (sum_or_null == nullptr && (two_calls || k <= (uint32_t)kChunkLog2)) {
        const uint64_t room = round_up(sz.sum_bytes, 256);
        if (workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
        if (workspace_bytes < room) return THC_EWORKSPACE;
        ws_left = (workspace_bytes - room) & ~(uint64_t)255;
    }
    if (k > (uint32_t)kChunkLog2) {
        if (workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
        if (ws_left < pipeline_workspace_need(ctx, sz.nblocks, sz.nblocks)) return THC_EWORKSPACE;
    }
    if (two_calls) {
        void *sum = sum_or_null != nullptr ? sum_or_null : static_cast<unsigned char *>(workspace) + ws_left;
        if ((rc = thc_aggregate(ctx, packed, n, d, sum, stream)) != THC_OK) return rc;
        return thc_decompress(ctx, sum, n, d, round, scales, outp, workspace, ws_left, stream);
    }
    PtrArrayP pin;
    MutPtrArrayP pout, prot;
    memset(&pin, 0, sizeof pin);
    memset(&pout, 0, sizeof pout);
    memset(&prot, 0, sizeof prot);
    for (uint32_t i = 0; i < n; ++i) pin.p[i] = packed[i];
    pout.p[0] = outp;
    pout.p[1] = sum_or_null;
    if (use_block_kernel(ctx, sz.d_pad))
        return launch_block(ctx, block_kernel(kAggDecompress, 4, true, ctx->cfg.log2_block), kAggDecompress, 0, sz, d, 1, 0, round, n, scales,
                            pin, pout, prot, static_cast<cudaStream_t>(stream), nullptr, n);
    pipe_kernel_t kern = pick_pipe_kernel<kAggDecompress>(ctx->cfg.bits, true, k);
    return launch_pipeline(ctx, kern, false, sz, d, 1, 0, round, n, scales, workspace, pin, pout, prot,
                           static_cast<cudaStream_t>(stream), nullptr, false, n);
}

int thc_quantize_rotated(thc_ctx *ctx, const float *const *rotated, uint32_t n_local,
                         uint32_t worker_base, uint64_t d, uint32_t round, const float *scales,
                         void *const *packed, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, n_local, &sz)) != THC_OK) return rc;
    if ((rc = check_ptr_array(reinterpret_cast<const void *const *>(rotated), n_local)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n_local)) != THC_OK) return rc;
    if (scales == nullptr) return THC_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PtrArray in;
    MutPtrArray out;
    memset(&in, 0, sizeof in);
    memset(&out, 0, sizeof out);
    for (uint32_t i = 0; i < n_local; ++i) { in.p[i] = rotated[i]; out.p[i] = packed[i]; }
    const uint64_t units = sz.d_pad / 8;
    uint64_t blocks = (units + kThreads - 1) / kThreads;
    const uint64_t cap = (uint64_t)ctx->sm_count * 16;
    if (blocks > cap) blocks = cap;
    const dim3 grid((unsigned)blocks, n_local);
    const uint32_t k = ctx->cfg.log2_block, g = ctx->cfg.granularity;
    const size_t qr_smem = (size_t)(g + 1) * kLutEntryBytes + (size_t)kQrBlockCache * 8;
#define THC_QR(B, I) THC_CUDA(launch_after(quantize_rotated_kernel<B, I>, grid, kThreads, qr_smem, st, \
        in, out, sz.d_pad, k, g, round, worker_base,                         \
        ctx->cfg.range_mode == THC_RANGE_MINMAX ? 1u : 0u, scales, ctx->dev, ctx->keys))
    switch (ctx->cfg.bits) {
    case 1: if (ctx->identity) THC_QR(1, true); else THC_QR(1, false); break;
    case 2: if (ctx->identity) THC_QR(2, true); else THC_QR(2, false); break;
    case 3: if (ctx->identity) THC_QR(3, true); else THC_QR(3, false); break;
    case 4: if (ctx->identity) THC_QR(4, true); else THC_QR(4, false); break;
    default: THC_QR(8, true); break;              // (the only table, see validate_config)
    }
#undef THC_QR
    return THC_OK;
}

int thc_aggregate(thc_ctx *ctx, const void *const *packed, uint32_t n, uint64_t d, void *sum,
                  void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    if (n == 0 || n > ctx->cfg.workers) return THC_EINVAL;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, n, &sz)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n)) != THC_OK) return rc;
    if (sum == nullptr || !aligned16(sum)) return THC_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    PtrArray in;
    memset(&in, 0, sizeof in);
    for (uint32_t i = 0; i < n; ++i) in.p[i] = packed[i];
    const uint64_t units = sz.d_pad / 32;       // the kernel finishes a tail of 8..24 itself
    uint64_t blocks = (units + kThreads - 1) / kThreads;
    if (blocks == 0) blocks = 1;
    const uint64_t cap = (uint64_t)ctx->sm_count * 16;
    if (blocks > cap) blocks = cap;
    unsigned char *s = static_cast<unsigned char *>(sum);
    if (ctx->cfg.bits == 4 && ctx->acc_bits == 8 && ctx->cfg.granularity < 128 && sz.d_pad % 32 == 0) {
        const uint64_t units32 = sz.d_pad / 32;
        uint64_t nb = (units32 + kThreads - 1) / kThreads;
        const uint64_t cap32 = (uint64_t)ctx->sm_count * 64;     // a unit or two per thread: no uneven tail
        if (nb > cap32) nb = cap32;
        THC_CUDA(launch_after(aggregate_b4w8_kernel, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, ctx->dev,
                                                                  reinterpret_cast<uint4 *>(s)));
        return THC_OK;
    }
    const uint32_t bits = ctx->cfg.bits, g = ctx->cfg.granularity, w = ctx->acc_bits;
    if (bits == 4 && w == 16 && g < 128 && sz.d_pad % 32 == 0) {
        const uint64_t units32 = sz.d_pad / 32;
        uint64_t nb = (units32 + kThreads - 1) / kThreads;
        if (nb > (uint64_t)ctx->sm_count * 64) nb = (uint64_t)ctx->sm_count * 64;
        uint4 *s4 = reinterpret_cast<uint4 *>(s);
        if (g <= 31) THC_CUDA(launch_after(aggregate_b4w16_kernel<8>, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, ctx->dev, s4));
        else if (g <= 63) THC_CUDA(launch_after(aggregate_b4w16_kernel<4>, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, ctx->dev, s4));
        else THC_CUDA(launch_after(aggregate_b4w16_kernel<2>, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, ctx->dev, s4));
        return THC_OK;
    }
    if ((bits == 1 || (bits == 2 && ctx->identity)) && w == 8 && sz.d_pad % 32 == 0) {
        const uint64_t units32 = sz.d_pad / 32;
        uint64_t nb = (units32 + kThreads - 1) / kThreads;
        if (nb > (uint64_t)ctx->sm_count * 8) nb = (uint64_t)ctx->sm_count * 8;
        if (bits == 1)
            THC_CUDA(launch_after(aggregate_small_w8_kernel<1>, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, g,
                                                                            reinterpret_cast<uint4 *>(s)));
        else
            THC_CUDA(launch_after(aggregate_small_w8_kernel<2>, dim3((unsigned)nb), kThreads, 0, st, in, n, units32, 1u,
                                                                            reinterpret_cast<uint4 *>(s)));
        return THC_OK;
    }
    if (bits == 3 && w <= 16 && sz.d_pad % 64 == 0) {
        const uint64_t units64 = sz.d_pad / 64;
        uint64_t nb = (units64 + 127) / 128;
        if (nb > (uint64_t)ctx->sm_count * 64) nb = (uint64_t)ctx->sm_count * 64;
        uint4 *s4 = reinterpret_cast<uint4 *>(s);
        const uint32_t chunk = w == 8 ? n : 255u / g;
        if (w == 8) THC_CUDA(launch_after(aggregate_b3_kernel<8>, dim3((unsigned)nb), 128, 0, st, in, n, units64, chunk, ctx->dev, s4));
        else THC_CUDA(launch_after(aggregate_b3_kernel<16>, dim3((unsigned)nb), 128, 0, st, in, n, units64, chunk, ctx->dev, s4));
        return THC_OK;
    }
    if (bits == 8 && ctx->identity && w == 16 && sz.d_pad % 16 == 0) {
        const uint64_t units16 = sz.d_pad / 16;
        uint64_t nb = (units16 + kThreads - 1) / kThreads;
        if (nb > (uint64_t)ctx->sm_count * 8) nb = (uint64_t)ctx->sm_count * 8;
        THC_CUDA(launch_after(aggregate_b8w16_kernel, dim3((unsigned)nb), kThreads, 0, st, in, n, units16, reinterpret_cast<uint4 *>(s)));
        return THC_OK;
    }
#define THC_AG(B, W) THC_CUDA(launch_after(aggregate_kernel<B, W>, dim3((unsigned)blocks), kThreads, 0, st, in, n, units, sz.d_pad, ctx->dev, s))
#define THC_AGW(B)                                       \
    do {                                                 \
        if (ctx->acc_bits == 8) THC_AG(B, 8);            \
        else if (ctx->acc_bits == 16) THC_AG(B, 16);     \
        else THC_AG(B, 32);                              \
    } while (0)
    switch (ctx->cfg.bits) {
    case 1: THC_AGW(1); break;
    case 2: THC_AGW(2); break;
    case 3: THC_AGW(3); break;
    case 4: THC_AGW(4); break;
    default: THC_AGW(8); break;
    }
#undef THC_AGW
#undef THC_AG
    return THC_OK;
}

int thc_error_feedback(thc_ctx *ctx, const void *const *grads, const void *const *packed,
                       uint32_t n_local, uint64_t d, uint32_t round, const float *scales,
                       float *const *ef, void *workspace, uint64_t workspace_bytes, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    if (ctx->cfg.in_dtype != THC_F32) return THC_EUNSUPPORTED;
    thc_sizes_t sz;
    if ((rc = thc_sizes(ctx, d, 1, &sz)) != THC_OK) return rc;
    if (n_local == 0 || n_local > THC_MAX_WORKERS) return THC_EINVAL;
    if ((rc = check_ptr_array(grads, n_local)) != THC_OK) return rc;
    if ((rc = check_ptr_array(packed, n_local)) != THC_OK) return rc;
    if ((rc = check_ptr_array(reinterpret_cast<const void *const *>(ef), n_local)) != THC_OK) return rc;
    if (scales == nullptr || workspace == nullptr || !aligned16(workspace)) return THC_EINVAL;
    if (workspace_bytes < sz.workspace_bytes) return THC_EWORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // one launch for all workers: indices in, x_i - RHT^-1(X_i) out
    thc_sizes_t szn;
    if ((rc = thc_sizes(ctx, d, n_local, &szn)) != THC_OK) return rc;
    if (ctx->cfg.log2_block > (uint32_t)kChunkLog2 && workspace_bytes < szn.workspace_bytes) return THC_EWORKSPACE;
    PtrArrayP pin;
    MutPtrArrayP pout, px;
    memset(&pin, 0, sizeof pin);
    memset(&pout, 0, sizeof pout);
    memset(&px, 0, sizeof px);
    for (uint32_t i = 0; i < n_local; ++i) {
        pin.p[i] = packed[i];
        pout.p[i] = ef[i];
        px.p[i] = const_cast<void *>(grads[i]);
    }
    const uint32_t bits = ctx->cfg.bits;
    if (use_block_kernel(ctx, sz.d_pad * n_local))
        return launch_block(ctx, block_kernel(kErrorFeedback, bits, true, ctx->cfg.log2_block), kErrorFeedback,
                            ((size_t)4 << bits) * (bits <= 4 ? 32 : 8), szn, d, n_local, 0, round, 1, scales, pin, pout, px, st);
    pipe_kernel_t kern = pick_pipe_kernel<kErrorFeedback>(bits, true, ctx->cfg.log2_block);
    return launch_pipeline(ctx, kern, false, szn, d, n_local, 0, round, 1, scales, workspace, pin, pout, px, st);
}

int thc_accumulate_error(thc_ctx *ctx, float *const *grads, const float *const *ef, uint32_t n_local,
                         uint64_t d, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    if (ctx->cfg.in_dtype != THC_F32) return THC_EUNSUPPORTED;
    if (n_local == 0 || n_local > THC_MAX_WORKERS || d == 0) return THC_EINVAL;
    if ((rc = check_ptr_array(reinterpret_cast<const void *const *>(grads), n_local)) != THC_OK) return rc;
    if ((rc = check_ptr_array(reinterpret_cast<const void *const *>(ef), n_local)) != THC_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint64_t blocks = (d / 4 + kThreads * kAccUnits - 1) / (kThreads * kAccUnits);
    if (blocks > 0x7FFFFFFFull) return THC_EUNSUPPORTED;
    MutPtrArray x;
    PtrArray e;
    memset(&x, 0, sizeof x);
    memset(&e, 0, sizeof e);
    // buffers that overlap (one gradient that takes several residuals) are added in the order given
    const auto overlap = [d](const float *a, const float *b) { return a < b + d && b < a + d; };
    bool apart = true;
    for (uint32_t i = 0; i < n_local; ++i)
        for (uint32_t j = 0; j < n_local; ++j)
            if (i != j && (overlap(grads[i], grads[j]) || overlap(grads[i], ef[j]))) apart = false;
    const uint32_t per_launch = apart ? n_local : 1u;
    for (uint32_t i0 = 0; i0 < n_local; i0 += per_launch) {
        for (uint32_t i = 0; i < per_launch; ++i) { x.p[i] = grads[i0 + i]; e.p[i] = ef[i0 + i]; }
        THC_CUDA(launch_after(accumulate_kernel, dim3((unsigned)(blocks ? blocks : 1), per_launch), kThreads, 0, st, x, e, d));
    }
    return THC_OK;
}

int thc_debug_skip_tasks(thc_ctx *ctx, uint32_t count)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    THC_CUDA(cudaDeviceSynchronize());
    // (blocks that have no pipeline claim their tiles from the same counter: a start that no pipeline launch takes
    // up and clears would make the next such launch leave tiles out)
    if (ctx->cfg.log2_block <= (uint32_t)kChunkLog2) return THC_OK;
    PipeCounters *pc = reinterpret_cast<PipeCounters *>(ctx->dev->counters);
    THC_CUDA(cudaMemcpy(&pc->head, &count, sizeof count, cudaMemcpyHostToDevice));
    ctx->pipeline_next = true;
    return THC_OK;
}

int thc_status(thc_ctx *ctx, uint32_t *flags, void *stream)
{
    int rc = check_launch_ctx(ctx);
    if (rc != THC_OK) return rc;
    if (flags == nullptr) return THC_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    THC_CUDA(cudaMemcpyAsync(flags, &ctx->dev->status, 4, cudaMemcpyDeviceToHost, st));
    THC_CUDA(cudaMemsetAsync(&ctx->dev->status, 0, 4, st));
    THC_CUDA(cudaStreamSynchronize(st));
    return THC_OK;
}

