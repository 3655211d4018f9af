// RHT blocks of 2^3 .. 2^17 coordinates: transform, quantise or de-quantise without an intermediate
// in global memory.
//
// A CTA holds a tile of consecutive coordinates of one worker in shared memory: 2^13 of them (one
// block, or several small ones; 128 threads, four CTAs per SM) or 2^14 (256 threads, two CTAs).  A
// block of 2^15 is held by a cluster of two tiles of 2^14, one of 2^16 (2^17) by eight of 2^13 (2^14); the CTAs
// exchange the last stages through distributed shared memory.  A thread owns 64 coordinates (64
// registers) at a time:
//   round 1  strides 1 .. 32: two rows of 32 coordinates per lane, straight after the load
//            (sign flip or de-quantisation in registers)
//   round 2  strides 64 .. 512 (1024 in the tile of 2^14), inside the warp's 2048 coordinates: only
//            a warp barrier in between
//   last     the three strides above on eight rows of a unit of eight coordinates, then the epilogue
//            on the registers.  In a cluster these three stages are a round in place, and the
//            last round takes the strides between the tiles: each thread gathers the same
//            eight-coordinate unit from all CTAs and finishes 1 / C of the positions of every tile.
// Stages above the block size are left out.  Few tiles per CTA are dealt out in a fixed stride,
// more are claimed from a counter (see launch_block); as soon as the last round holds the tile in registers
// the next tile's TMA copy is started, so the
// epilogue hides it.
//
// What bounds it.  Timers in the kernel, 4 x 2^26 coordinates in blocks of 2^12, 4 bits, before the quantiser was
// packed: per tile a CTA spent 2190 cycles on the load and the block constants, 2350 on round 1, 1650 on round 2 and its
// barrier, 1230 on the last round and 5480 on the epilogue (Philox and the quantiser, bound by instruction issue), with
// four CTAs side by side on an SM; with fixed shares of the tiles the CTAs ran for 371 us of 465 on average, hence the counter.
// Now (five rounds through shared memory with a block barrier between them in front): blocks of 2^12 compress
// 669 -> 400 us, decompress 156 -> 93 us, error feedback 1310 -> 499 us; 2^14 681 -> 408, 155 -> 111,
// 1316 -> 531 us.  In a cluster the gather binds (a tile of every CTA crosses the SM-to-SM network: 8740
// cycles for the last round of a tile of 2^15 where one of 2^14 takes 1580): 2^15 is as fast as the
// two-pass pipeline on large inputs (611 us; error feedback 985 -> 758 us) and takes 9.3 instead of 13.1 us on
// a few blocks; 2^16 and 2^17 pay only there (see block_kernel_serves).
#include "thc_block.h"

namespace thc {

// ------------------------------------------------------------------------ clusters
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 cluster_load(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ double cluster_load_f64(uint32_t addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t cluster_load_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// ------------------------------------------------------------------------ round 1
// A warp owns 64 rows of 8 chunks (32 coordinates); row r, chunk c sits at r*8 + (c ^ (r & 7)).  Lane l
// owns rows 2l and 2l+1, 64 consecutive coordinates.  Lanes with bit 2 set take row 2l+1 first:
// with that the eight lanes of a quarter warp are on rows of eight different XOR patterns and every
// 128-bit access is free of bank conflicts.  v[0..7] is the first row taken, v[8..15] the other one.
struct LowRows {
    int first;          // row (within the warp's 64) of v[0..7]; the other one is first ^ 1
    float s;            // -1 where v[0..7] is the upper row
};
__device__ __forceinline__ LowRows low_rows(int lane)
{
    LowRows r;
    const int h = (lane >> 2) & 1;
    r.first = 2 * lane + h;
    r.s = h ? -1.0f : 1.0f;
    return r;
}
__device__ __forceinline__ float4 *low_chunk(float4 *wtile, const LowRows &lr, int m)
{
    const int row = m < 8 ? lr.first : lr.first ^ 1;
    return wtile + row * 8 + ((m & 7) ^ (row & 7));
}

// The stages of strides 1 .. 32 that lie inside the block, and the store back.  (Variants side by
// side: stages under a condition, in place in 64 registers, cost the compiler 40 spilled ones.)
__device__ __forceinline__ void low_stages_store(float4 *wtile, const LowRows &lr, float4 (&v)[16], uint32_t k)
{
    if (k >= 6u) {
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = stages01(v[m]);
#pragma unroll
        for (int t = 0; t < 3; ++t) {
#pragma unroll
            for (int m = 0; m < 16; ++m)
                if (!(m & (1 << t))) butterfly(v[m], v[m | (1 << t)]);
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) swapped_butterfly(v[m], v[m + 8], lr.s);
#pragma unroll
        for (int m = 0; m < 16; ++m) *low_chunk(wtile, lr, m) = v[m];
        return;
    }
    // blocks of 8, 16 or 32 coordinates: a row at a time
#pragma unroll
    for (int m = 0; m < 16; ++m) *low_chunk(wtile, lr, m) = stages01(v[m]);
#pragma unroll 1
    for (int g = 0; g < 2; ++g) {
        float4 *row = wtile + (lr.first ^ g) * 8;
        const int x = (lr.first ^ g) & 7;
        float4 w[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) w[m] = row[m ^ x];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            if (k > 2u + t) {
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (!(m & (1 << t))) butterfly(w[m], w[m | (1 << t)]);
            }
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) row[m ^ x] = w[m];
    }
}

// ... of a gradient.  fp32 rows lie in the tile; the bf16 rows of a warp (64 rows of 64 bytes in the
// 64-byte swizzle) in the upper half of its 8 KB, and are widened exactly.
// With SQ the sum of squares of the lane's 64 inputs (fp64, four interleaved partial sums combined
// in a fixed order) is returned.
template <bool BF16, bool SQ>
__device__ __forceinline__ double low_round_gradient(float4 *wtile, const uint32_t *wsw, int lane, uint32_t k)
{
    const LowRows lr = low_rows(lane);
    float4 v[16];
    if (BF16) {
        const uint4 *stage = reinterpret_cast<const uint4 *>(wtile) + 256;
        uint4 raw[8];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int row = lr.first ^ g;
#pragma unroll
            for (int q = 0; q < 4; ++q) raw[4 * g + q] = stage[row * 4 + (q ^ ((row >> 1) & 3))];
        }
        __syncwarp();                              // the fp32 rows overlap other lanes' bf16 rows
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 t4 = raw[i];
            v[2 * i] = make_float4(__uint_as_float(t4.x << 16), __uint_as_float(t4.x & 0xFFFF0000u),
                                   __uint_as_float(t4.y << 16), __uint_as_float(t4.y & 0xFFFF0000u));
            v[2 * i + 1] = make_float4(__uint_as_float(t4.z << 16), __uint_as_float(t4.z & 0xFFFF0000u),
                                       __uint_as_float(t4.w << 16), __uint_as_float(t4.w & 0xFFFF0000u));
        }
    } else {
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = *low_chunk(wtile, lr, m);
    }
    double sq = 0.0;
    if (SQ) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            a0 = fma((double)v[m].x, (double)v[m].x, a0);
            a1 = fma((double)v[m].y, (double)v[m].y, a1);
            a2 = fma((double)v[m].z, (double)v[m].z, a2);
            a3 = fma((double)v[m].w, (double)v[m].w, a3);
        }
        sq = (a0 + a1) + (a2 + a3);
    }
    const uint32_t w0 = wsw[lr.first], w1 = wsw[lr.first ^ 1];
#pragma unroll
    for (int m = 0; m < 8; ++m) { v[m] = flip4(v[m], w0 >> (m * 4)); v[8 + m] = flip4(v[8 + m], w1 >> (m * 4)); }
    low_stages_store(wtile, lr, v, k);
    return sq;
}

// (step, base) of the estimate line for chunk m of a row: rows of 32 coordinates hold several blocks
// only below 2^5.
struct DecodeConst {
    const float2 *blk;         // of the blocks of the tile
    float2 row0, row1;
    uint32_t k;
};
__device__ __forceinline__ DecodeConst decode_const(const float2 *blk, const LowRows &lr, int warp, uint32_t k)
{
    DecodeConst c;
    c.blk = blk; c.k = k;
    const uint32_t r0 = (uint32_t)(64 * warp + lr.first), r1 = r0 ^ 1u;
    c.row0 = blk[k >= 13u ? 0u : (r0 * 32u) >> k];
    c.row1 = blk[k >= 13u ? 0u : (r1 * 32u) >> k];
    return c;
}
__device__ __forceinline__ float2 chunk_const(const DecodeConst &c, const LowRows &lr, int warp, int m)
{
    if (c.k >= 5u) return m < 8 ? c.row0 : c.row1;
    const uint32_t row = (uint32_t)(64 * warp + (m < 8 ? lr.first : lr.first ^ 1));
    return c.blk[(row * 32u + 4u * (m & 7)) >> c.k];
}

// ... of the inverse transform: the thread fetches its two rows straight from global memory and
// de-quantises them in registers: sums Y -> m + Y (M - m)/(g n), or own indices
// z -> m + T[z] (M - m)/g  (Algorithm 2).  A row of 32 coordinates is IN_BITS 32-bit words; src is the
// warp's first row, `rows` how many of the warp's rows exist (below 64 in the last tile of small blocks).
template <int MODE, int BITS, int FREP>
__device__ __forceinline__ void low_round_inverse(float4 *wtile, const unsigned char *src, int coords, const float2 *blk,
                                                  const float *ft, int lane, int warp, uint32_t k)
{
    constexpr int IN_BITS = MODE == kDecompress8 ? 8 : MODE == kDecompress16 ? 16
                            : MODE == kDecompress32 ? 32 : BITS;
    const LowRows lr = low_rows(lane);
    const DecodeConst dc = decode_const(blk, lr, warp, k);
    float4 v[16];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int row = lr.first ^ g;
        uint32_t w[IN_BITS];
#pragma unroll
        for (int q = 0; q < IN_BITS; ++q) w[q] = 0u;
        const unsigned char *p = src + (size_t)row * (IN_BITS * 4);
        if (row * 32 + 32 <= coords) {
            if constexpr (IN_BITS >= 4) {
#pragma unroll
                for (int q = 0; q < IN_BITS / 4; ++q) {
                    const uint4 t4 = ld_global(reinterpret_cast<const uint4 *>(p) + q);
                    w[4 * q] = t4.x; w[4 * q + 1] = t4.y; w[4 * q + 2] = t4.z; w[4 * q + 3] = t4.w;
                }
            } else if constexpr (IN_BITS == 2) {
                const uint2 t2 = ld_global(reinterpret_cast<const uint2 *>(p));
                w[0] = t2.x; w[1] = t2.y;
            } else {
#pragma unroll
                for (int q = 0; q < IN_BITS; ++q) w[q] = ld_global(reinterpret_cast<const uint32_t *>(p) + q);
            }
        } else if (row * 32 < coords) {
            // 8, 16 or 24 coordinates (blocks of 2^3 and 2^4): byte by byte
            const int bytes = (coords - row * 32) * IN_BITS / 8;
#pragma unroll
            for (int q = 0; q < IN_BITS; ++q)
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    if (4 * q + y < bytes) w[q] |= (uint32_t)ld_global(p + 4 * q + y) << (8 * y);
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float2 bc = chunk_const(dc, lr, warp, 8 * g + m);
            float sv[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int bit = (m * 4 + e) * IN_BITS;
                const uint32_t nxt = w[((bit >> 5) + 1) < IN_BITS ? (bit >> 5) + 1 : (bit >> 5)];
                const uint32_t val = IN_BITS == 32 ? w[bit >> 5]
                                     : __funnelshift_r(w[bit >> 5], nxt, bit & 31) & ((1u << (IN_BITS & 31)) - 1u);
                float yf;
                if (MODE == kErrorFeedback) yf = ft[val * FREP];
                else if (MODE == kDecompress32) yf = (float)val;
                else yf = __uint_as_float(0x4B000000u | val) - 8388608.0f;
                sv[e] = fmaf(yf, bc.x, bc.y);
            }
            v[8 * g + m] = make_float4(sv[0], sv[1], sv[2], sv[3]);
        }
    }
    low_stages_store(wtile, lr, v, k);
}

// The sums of one row of 32 coordinates (exact in floats), acc_bits each, to coordinate j.
__device__ __forceinline__ void store_row_sums(void *sum_out, size_t j, uint32_t acc_bits, const float4 *v)
{
    if (acc_bits == 8) {
        uint4 *o = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(sum_out) + j);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t ww[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 f = v[4 * q + c];
                ww[c] = (uint32_t)f.x | ((uint32_t)f.y << 8) | ((uint32_t)f.z << 16) | ((uint32_t)f.w << 24);
            }
            o[q] = make_uint4(ww[0], ww[1], ww[2], ww[3]);
        }
    } else if (acc_bits == 16) {
        uint4 *o = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(sum_out) + 2 * j);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 a = v[2 * q], b = v[2 * q + 1];
            o[q] = make_uint4((uint32_t)a.x | ((uint32_t)a.y << 16), (uint32_t)a.z | ((uint32_t)a.w << 16),
                              (uint32_t)b.x | ((uint32_t)b.y << 16), (uint32_t)b.z | ((uint32_t)b.w << 16));
        }
    } else {
        uint4 *o = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(sum_out) + 4 * j);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] = make_uint4((uint32_t)v[q].x, (uint32_t)v[q].y, (uint32_t)v[q].z, (uint32_t)v[q].w);
    }
}

// ... of thc_aggregate_decompress: the PS line and the estimate line of Algorithm 2 in one place.  The
// thread fetches the packed indices of its two rows from every worker, adds up the table values
// (in byte lanes, then exactly in floats: the sums stay below 2^24 and equal the integer sums
// thc_aggregate writes), optionally writes the sums, and goes on with v = m + Y (M - m)/(g n).
// 4-bit indices and table values below 128 only, four look-ups per byte-permute instruction (see
// aggregate_b4w8_kernel), `chunk` workers at a time so that no byte overflows.
__device__ __forceinline__ void low_round_aggregate(float4 *wtile, const PtrArrayP &in, uint32_t agg_n, size_t byte_off, int coords,
                                                    const float2 *blk, void *sum_out, size_t coord_off, uint32_t acc_bits,
                                                    int lane, int warp, const uint32_t (&tb)[4], uint32_t chunk, uint32_t k)
{
    const LowRows lr = low_rows(lane);
    const DecodeConst dc = decode_const(blk, lr, warp, k);
    float4 v[16];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int row = lr.first ^ g;
        float4 *vg = v + 8 * g;
#pragma unroll
        for (int m = 0; m < 8; ++m) vg[m] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row * 32 < coords) {
#pragma unroll 1
            for (uint32_t i0 = 0; i0 < agg_n; i0 += chunk) {
                uint32_t acc[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[q] = 0u;
                const uint32_t i1 = min(agg_n, i0 + chunk);
#pragma unroll 4
                for (uint32_t i = i0; i < i1; ++i) {
                    const unsigned char *src = static_cast<const unsigned char *>(in.p[i]) + byte_off;
                    const uint4 t4 = ld_global(reinterpret_cast<const uint4 *>(src + (size_t)row * 16));
                    const uint32_t words[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const uint32_t a = words[h], b = a ^ 0x88888888u;
                        acc[2 * h] += prmt(tb[0], tb[1], a) + prmt(tb[2], tb[3], b);
                        acc[2 * h + 1] += prmt(tb[0], tb[1], a >> 16) + prmt(tb[2], tb[3], b >> 16);
                    }
                }
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const uint32_t wv = acc[m];
                    vg[m].x += __uint_as_float(__byte_perm(wv, 0x4B000000u, 0x7440)) - 8388608.0f;
                    vg[m].y += __uint_as_float(__byte_perm(wv, 0x4B000000u, 0x7441)) - 8388608.0f;
                    vg[m].z += __uint_as_float(__byte_perm(wv, 0x4B000000u, 0x7442)) - 8388608.0f;
                    vg[m].w += __uint_as_float(__byte_perm(wv, 0x4B000000u, 0x7443)) - 8388608.0f;
                }
            }
            if (sum_out != nullptr) store_row_sums(sum_out, coord_off + (size_t)row * 32, acc_bits, vg);
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float2 bc = chunk_const(dc, lr, warp, 8 * g + m);
            vg[m].x = fmaf(vg[m].x, bc.x, bc.y); vg[m].y = fmaf(vg[m].y, bc.x, bc.y);
            vg[m].z = fmaf(vg[m].z, bc.x, bc.y); vg[m].w = fmaf(vg[m].w, bc.x, bc.y);
        }
    }
    low_stages_store(wtile, lr, v, k);
}

// ------------------------------------------------------------------------ round 2
// Strides 64 .. 512 (row bits 1 .. 4), in place inside the warp's 64 rows: lane (bit 5 of the row, bit 0 of
// the row, chunk).
template <int STAGES>
__device__ __forceinline__ void mid_round(float4 *wtile, int lane)
{
    const int cc = lane & 7, r0 = ((lane >> 3) & 1) | ((lane >> 4) << 5);
    float4 *q[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) q[x] = wtile + r0 * 8 + (cc ^ (r0 & 1) ^ (2 * x));
    float4 v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = q[m & 3][16 * m];
#pragma unroll
    for (int t = 0; t < STAGES; ++t) {
#pragma unroll
        for (int m = 0; m < 16; ++m)
            if (!(m & (1 << t))) butterfly(v[m], v[m | (1 << t)]);
    }
#pragma unroll
    for (int m = 0; m < 16; ++m) q[m & 3][16 * m] = v[m];
}

// Five strides, 64 .. 1024: lane l owns the pair of coordinates 2l, 2l+1 of each of the warp's 32 groups of
// 64; a half warp's 64-bit access is one row of 128 bytes.
__device__ __forceinline__ void mid_round5(float4 *wtile, int lane)
{
    unsigned char *b = reinterpret_cast<unsigned char *>(wtile) + (lane >> 4) * 128 + (lane & 1) * 8;
    const int c0 = ((lane >> 1) & 7) ^ (lane >> 4);
    float2 *p[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) p[x] = reinterpret_cast<float2 *>(b + ((c0 ^ (2 * x)) << 4));
    float2 v[32];
#pragma unroll
    for (int g = 0; g < 32; ++g) v[g] = p[g & 3][g * 32];
#pragma unroll
    for (int t = 0; t < 5; ++t) {
#pragma unroll
        for (int g = 0; g < 32; ++g)
            if (!(g & (1 << t))) {
                const float2 a = v[g], c = v[g | (1 << t)];
                v[g] = add2(a, c);
                v[g | (1 << t)] = sub2(a, c);
            }
    }
#pragma unroll
    for (int g = 0; g < 32; ++g) p[g & 3][g * 32] = v[g];
}

// ------------------------------------------------------------------------ last round
// Stages on eight rows of two chunks.
template <int STAGES>
__device__ __forceinline__ void unit_stages(float4 (&a)[8], float4 (&b)[8])
{
#pragma unroll
    for (int t = 0; t < STAGES; ++t) {
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if (!(m & (1 << t))) {
                butterfly(a[m], a[m | (1 << t)]);
                butterfly(b[m], b[m | (1 << t)]);
            }
    }
}
template <int STAGES, int STEP>
__device__ __forceinline__ void unit_load(const float4 *pa, const float4 *pb, float4 (&a)[8], float4 (&b)[8])
{
#pragma unroll
    for (int m = 0; m < 8; ++m) { a[m] = pa[m * STEP]; b[m] = pb[m * STEP]; }
    unit_stages<STAGES>(a, b);
}
// The same from the tiles of a cluster: 2^STAGES tiles, row of the first, STEP rows further for each
// 2^STAGES-th register.  `own` is the address of the own tile.
template <int STAGES, int STEP>
__device__ __forceinline__ void unit_gather(uint32_t own, uint32_t row, uint32_t ca, uint32_t cb, float4 (&a)[8], float4 (&b)[8])
{
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const uint32_t base = cluster_map(own + (row + STEP * (m >> STAGES)) * 128u, m & ((1 << STAGES) - 1));
        a[m] = cluster_load(base + ca);
        b[m] = cluster_load(base + cb);
    }
}

// ------------------------------------------------------------------------ scales
// Scales and compress in one launch: the sums of squares come from round 1's registers, go to shared memory and are
// exchanged between the workers' CTAs while round 2 runs; the scales are ready before the epilogue, which alone needs
// them.  What it adds to a compress (4 x 2^25 coordinates in 2^12 blocks: 202 -> 246 us) is the conversion to fp64, which runs at an
// eighth of the issue rate and fills its own unit in round 1, three dispatch slots per coordinate, and the
// wait for the slowest of the cluster; the launch it replaces took 83 us.
// Scales of the tile's blocks (Section 5.3: M = t_p max_i ||x_i|| / sqrt(B)) from the sums of squares in the shared memory of
// the n_local CTAs of the cluster, and the quantiser's constants into `bc`.  sq: address of the own sums, one per
// block or, from 2^11 on, per 2^11 coordinates; they are added in ascending order.  Every CTA does it for itself;
// `store`: this one writes the scales.
template <int TILE_LOG2>
__device__ __forceinline__ void block_scales(const BlockParams &P, uint32_t sq, uint32_t blk0, float2 *bc, bool store, int tid)
{
    const uint32_t k = P.k, blocks = 1u << (TILE_LOG2 - k);
    double s = 0.0;                                    // largest sum of squares; a NaN sticks
    uint32_t b;
    bool live;
    if (k <= 10u) {
        b = (uint32_t)tid;                             // a thread per block
        live = b < blocks;
        if (live) {
            for (uint32_t i = 0; i < P.n_local; ++i) {
                const double v = cluster_load_f64(cluster_map(sq + 8u * b, i));
                if (v > s || v != v) s = v;
            }
        }
    } else {
        b = (uint32_t)tid >> 5;                        // a warp per block, a lane per worker
        live = b < blocks;
        const uint32_t lane = (uint32_t)tid & 31u, parts = 1u << (k - 11u);
        if (live && lane < P.n_local) {
            const uint32_t a = cluster_map(sq + 8u * parts * b, lane);
#pragma unroll 4
            for (uint32_t c = 0; c < parts; ++c) s += cluster_load_f64(a + 8u * c);
        }
#pragma unroll
        for (int off = 1; off < (int)kScalesMaxWorkers; off <<= 1) {
            const double v = __shfl_xor_sync(0xFFFFFFFFu, s, off);
            if (v > s || v != v) s = v;
        }
        live = live && lane == 0u;
    }
    if (!live) return;
    float M = (float)(P.t_p * sqrt(s) / P.sqrt_block);
    uint32_t flags = 0;
    if (!isfinite(M)) { M = 0.0f; flags |= THC_STATUS_NONFINITE; }
    if (M == 0.0f) flags |= THC_STATUS_ZERO_BLOCK;
    bc[b] = compress_constants(BlockRange{-M, M});
    if (store && blk0 + b < P.nblocks) {
        P.scales_out[blk0 + b] = M;
        if (flags) atomicOr(&P.dev->status, flags);
    }
}

// ------------------------------------------------------------------------ the kernel
// KIND: see block_kind.  CLAIMS: tasks can be claimed from P.head (see block_claims).
template <int MODE, int BITS, bool IDENTITY, int KIND, bool CLAIMS>
__global__ void __launch_bounds__(block_tile_log2(KIND) == 13 ? 128 : 256, block_tile_log2(KIND) == 13 ? 4 : 2)
thc_block_kernel(const __grid_constant__ TmaMaps maps, const __grid_constant__ BlockParams P,
                 const __grid_constant__ PtrArrayP in, const __grid_constant__ MutPtrArrayP outp,
                 const __grid_constant__ MutPtrArrayP rotated, const __grid_constant__ PhiloxKeys keys)
{
    constexpr int kBLog2 = block_tile_log2(KIND);
    constexpr uint32_t E = block_cluster_log2(KIND), C = 1u << E;
    constexpr bool CLUSTER = E != 0u;
    constexpr int kBElems = 1 << kBLog2;
    constexpr int kBThreads = kBElems / 64;
    constexpr int kBSignWords = kBElems / 32;
    constexpr int kBRowStep = kBSignWords / 8;         // rows between the registers of the last round
    constexpr bool kEF = MODE == kErrorFeedback;
    constexpr bool kRange = MODE == kRangeF32;
    // Scales in the same launch: the n_local CTAs of a cluster hold the same tile of all workers and exchange
    // its sums of squares.
    constexpr bool kScales = MODE == kCompressF32Fused || MODE == kCompressBF16Fused;
    constexpr bool kBF16In = MODE == kCompressBF16 || MODE == kCompressBF16Fused;
    constexpr bool kF32In = MODE == kCompressF32 || MODE == kCompressF32Fused || kRange;
    constexpr bool kForward = kF32In || kBF16In;
    constexpr bool kQuant = kForward && !kRange;
    constexpr int kFRep = BITS <= 4 ? 32 : 8;
    extern __shared__ __align__(1024) unsigned char block_smem_raw[];
    // TMA's 128-byte swizzle needs the tile on a 1024-byte boundary of the shared address space; the
    // launch reserves 1 KB of slack for this round-up.
    unsigned char *smem = block_smem_raw +
        ((1024u - ((uint32_t)__cvta_generic_to_shared(block_smem_raw) & 1023u)) & 1023u);
    float4 *tile = reinterpret_cast<float4 *>(smem);
    uint32_t *sw = reinterpret_cast<uint32_t *>(smem + kBElems * 4);                  // two slots by task parity
    float2 *blk_const = reinterpret_cast<float2 *>(smem + kBElems * 4 + 2 * kBSignWords * 4);   // likewise
    unsigned char *lut = smem + kBElems * 4 + 2 * kBSignWords * 4 + (size_t)P.const_slots * 16;
    __shared__ __align__(8) uint64_t s_full;
    __shared__ uint32_t s_next[2];                     // the task after this one
    __shared__ double s_sq[2][!kScales ? 1 : KIND == 0 ? kBElems >> kScalesMinLog2 : kBElems >> 11];    // sums of squares, by task parity

    const int thread = threadIdx.x;
    const uint32_t k = P.k;
    const uint32_t group = kScales ? P.n_local : C;    // CTAs that take a task together
    const uint32_t rank = kScales ? blockIdx.x % group : CLUSTER ? blockIdx.x & (C - 1u) : 0u;
    const uint64_t d_rows32 = P.d >> 5;

    // tasks: tile (cluster: block) x worker, worker minor.  Dealt out in a fixed stride, or, where P.head is
    // given, claimed from it after the first two.
    const uint32_t groups = kScales ? gridDim.x / group : gridDim.x >> E;
    uint32_t task = kScales ? blockIdx.x / group : blockIdx.x >> E;
    uint32_t unit = task, wl = kScales ? rank : 0u;
    constexpr bool kVectors = !kScales && (kForward || kEF);      // (the others have one, or one to a CTA)
    const uint32_t unit_step = groups / P.n_local, wl_step = groups - unit_step * P.n_local;
    auto split_task = [&]() {
        unit = task;
        if (kVectors) {
            unit = task / P.n_local;
            wl = task - unit * P.n_local;
        }
    };
    split_task();
    auto tile_coord = [&](uint32_t u) -> uint64_t { return ((uint64_t)((u << E) + (CLUSTER ? rank : 0u))) << kBLog2; };
    // Thread 0: whole tiles of a gradient come by TMA.
    auto by_tma = [&](uint32_t u) -> bool { return kForward && (tile_coord(u) >> 5) + kBSignWords <= d_rows32; };
    auto start_load = [&](uint32_t u, uint32_t w) {
        const int row = (int)(tile_coord(u) >> 5);
        const uint64_t policy = make_evict_first_policy();         // gradients are read once
        if (kF32In) {
            mbar_expect_tx(&s_full, kBElems * 4);
            for (int q = 0; q < kBSignWords / 256; ++q) tma_load_2d(tile + 2048 * q, &maps.in[w], 0, row + 256 * q, &s_full, policy);
        } else {
            // every warp's 4 KB of bf16 into the upper half of its own 8 KB of the buffer
            mbar_expect_tx(&s_full, kBElems * 2);
#pragma unroll 1
            for (int q = 0; q < kBThreads / 32; ++q)
                tma_load_2d(tile + 512 * q + 256, &maps.in[w], 0, row + 64 * q, &s_full, policy);
        }
    };
    // The inverse modes read the tile's sums or indices (error feedback: and x) from global memory:
    // pull the lines into L2.
    auto prefetch_inputs = [&](uint32_t u, uint32_t w) {
        constexpr int kInBits = MODE == kDecompress8 ? 8 : MODE == kDecompress16 ? 16 : MODE == kDecompress32 ? 32 : BITS;
        const uint64_t j = tile_coord(u);
        const uint64_t first = j * kInBits / 8, limit = P.d_pad * kInBits / 8;
        const uint32_t sources = MODE == kAggDecompress ? P.agg_n : 1u;
        for (uint32_t i = 0; i < sources; ++i) {
            const unsigned char *src = static_cast<const unsigned char *>(in.p[MODE == kAggDecompress ? i : kEF ? w : 0]);
            for (uint32_t l = thread; l < (uint32_t)kBElems * kInBits / 8 / 128; l += kBThreads)
                if (first + 128ull * l < limit) prefetch_l2(src + first + 128ull * l);
        }
        if (kEF) {
            const float *x = static_cast<const float *>(rotated.p[w]);
            for (uint32_t l = thread; l < (uint32_t)kBElems / 32; l += kBThreads)
                if (j + 32ull * l < P.d) prefetch_l2(x + j + 32ull * l);
        }
    };

    if (thread == 0) {
        mbar_init(&s_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (kQuant && !IDENTITY) lut_fill(lut, P.dev, P.granularity, thread, kBThreads);
    if (kEF) {
        // table values as floats, one copy per lane (8 copies for 8-bit indices)
        for (int i = thread; i < (1 << BITS) * kFRep; i += kBThreads)
            reinterpret_cast<float *>(lut)[i] = (float)P.dev->table[i / kFRep];
    }
    uint32_t agg_tb[4] = {0u, 0u, 0u, 0u};             // the table as 16 bytes
    if (MODE == kAggDecompress) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            agg_tb[q] = P.dev->table[4 * q] | (P.dev->table[4 * q + 1] << 8) | (P.dev->table[4 * q + 2] << 16) |
                        (P.dev->table[4 * q + 3] << 24);
    }
    depend_on_previous();
    if (task < P.tasks) {
        if (thread == 0 && by_tma(unit)) start_load(unit, wl);
        if (!kForward) prefetch_inputs(unit, wl);
    }
    __syncthreads();

    uint32_t uses = 0;                                 // TMA loads waited for
    for (uint32_t n = 0; task < P.tasks; ++n) {
        // (opaque, so that the addresses of all rounds are not kept in registers over the whole loop)
        int tid = thread;
        asm volatile("" : "+r"(tid));
        const int lane = tid & 31, warp = tid >> 5;
        float4 *wtile = tile + 512 * warp;
        const uint32_t par = n & 1u;
        const uint64_t j0 = tile_coord(unit);
        // the task after this one, handed round by the barrier in front of the last round
        const bool claims = CLAIMS && P.head != nullptr && task >= groups && tid == 0 && rank == 0u;
        uint32_t claimed = 0u;
        if (claims) claimed = groups * 2u + atomicAdd(P.head, 1u);
        // ---- constants of the tile's blocks
        float2 *bc = blk_const + par * P.const_slots;
        const uint32_t blk0 = (uint32_t)(j0 >> k);
        if (!kRange && !kScales) {
            for (uint32_t b = tid; b < P.const_slots; b += kBThreads) {
                float2 c = make_float2(0.f, 0.f);
                if (blk0 + b < P.nblocks) {
                    const BlockRange br = block_range(P.scales, blk0 + b, P.nblocks, P.exact_range);
                    c = kForward ? compress_constants(br) : decode_constants(br, P.granularity, P.divisor);
                }
                bc[b] = c;
            }
        }
        // ---- sign words: of the warp's own rows (compress), or of the positions the thread finishes
        if (kForward) {
            if (lane < 16)
                *reinterpret_cast<uint4 *>(sw + 64 * warp + 4 * lane) = sign_call(j0 + 2048u * warp + 128u * lane, P.round, keys);
            __syncwarp();
        } else if (tid < kBSignWords / 4) {
            // cluster: 1 / C of every tile, in order of the tiles
            const uint32_t per = (uint32_t)(kBSignWords / 4) >> E, from = (uint32_t)tid / per, c = (uint32_t)tid - from * per;
            const uint64_t j = !CLUSTER ? j0 + 128u * tid
                                       : ((uint64_t)unit << k) + ((uint64_t)from << kBLog2) + (rank << (kBLog2 - E)) + 128u * c;
            *reinterpret_cast<uint4 *>(sw + kBSignWords * par + 4 * tid) = sign_call(j, P.round, keys);
        }
        if (!kForward) __syncthreads();                // the constants

        // ---- round 1
        if constexpr (kForward) {
            const bool tma = by_tma(unit);
            if (tma) {
                if (!mbar_wait(&s_full, uses & 1u)) atomicOr(&P.dev->status, THC_STATUS_WAIT_TIMEOUT);
                ++uses;
            } else {
                // the ragged last tile of a gradient, zero behind its end: a warp loads its own rows
                const uint64_t jw = j0 + 2048u * warp;
                if (kF32In) {
                    const float *x = static_cast<const float *>(in.p[wl]);
#pragma unroll 4
                    for (int i = 0; i < 16; ++i) {
                        const int c = lane + 32 * i;
                        wtile[c ^ ((c >> 3) & 7)] = load_f32x4_masked(x, jw + 4u * c, P.d);
                    }
                } else {
                    const uint16_t *x = static_cast<const uint16_t *>(in.p[wl]);
#pragma unroll 1
                    for (int i = 0; i < 8; ++i) {
                        const int u = lane + 32 * i;
                        const uint64_t j = jw + 8u * u;
                        uint32_t w[4] = {0, 0, 0, 0};
                        if (j + 8 <= P.d) {
                            const uint4 q4 = ld_global(reinterpret_cast<const uint4 *>(x + j));
                            w[0] = q4.x; w[1] = q4.y; w[2] = q4.z; w[3] = q4.w;
                        } else {
                            for (int e = 0; e < 8; ++e)
                                if (j + e < P.d) w[e >> 1] |= (uint32_t)ld_global(x + j + e) << ((e & 1) * 16);
                        }
                        const int c = 2 * u;
                        wtile[c ^ ((c >> 3) & 7)] = make_float4(__uint_as_float(w[0] << 16), __uint_as_float(w[0] & 0xFFFF0000u),
                                                                __uint_as_float(w[1] << 16), __uint_as_float(w[1] & 0xFFFF0000u));
                        wtile[(c + 1) ^ ((c >> 3) & 7)] = make_float4(__uint_as_float(w[2] << 16), __uint_as_float(w[2] & 0xFFFF0000u),
                                                                      __uint_as_float(w[3] << 16), __uint_as_float(w[3] & 0xFFFF0000u));
                    }
                }
                __syncwarp();
            }
            double sq;
            if (kBF16In && tma) sq = low_round_gradient<true, kScales>(wtile, sw + 64 * warp, lane, k);
            else sq = low_round_gradient<false, kScales>(wtile, sw + 64 * warp, lane, k);
            if constexpr (kScales) {
                // a lane has 64 consecutive coordinates: 2^(k-6) lanes to a block, at most the warp
                const uint32_t parts_log2 = min(k, 11u);
                for (uint32_t b = 0; b + 6u < parts_log2; ++b) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, 1 << b);
                if ((lane & ((1 << (parts_log2 - 6u)) - 1)) == 0) s_sq[par][(2048u * warp + 64u * lane) >> parts_log2] = sq;
                if (claims) s_next[par] = claimed;
                __syncwarp();
                cluster_arrive();
            }
        } else {
            const uint64_t jw = j0 + 2048u * warp;
            const int coords = jw + 2048u <= P.d_pad ? 2048 : jw < P.d_pad ? (int)(P.d_pad - jw) : 0;
            if constexpr (MODE == kAggDecompress) {
                low_round_aggregate(wtile, in, P.agg_n, jw / 2, coords, bc, outp.p[1], jw, P.agg_acc_bits, lane, warp, agg_tb,
                                    P.agg_chunk, k);
            } else {
                constexpr int kInBits = MODE == kDecompress8 ? 8 : MODE == kDecompress16 ? 16 : MODE == kDecompress32 ? 32 : BITS;
                const unsigned char *src = static_cast<const unsigned char *>(in.p[kEF ? wl : 0]) + jw * kInBits / 8;
                low_round_inverse<MODE, BITS, kFRep>(wtile, src, coords, bc, reinterpret_cast<const float *>(lut) + (tid & (kFRep - 1)),
                                                     lane, warp, k);
            }
        }
        // ---- round 2
        __syncwarp();
        if constexpr (KIND == 3) {
            mid_round<4>(wtile, lane);
        } else if constexpr (KIND == 0) {
            switch (k) {
            case 3: case 4: case 5: case 6: break;
            case 7: mid_round<1>(wtile, lane); break;
            case 8: mid_round<2>(wtile, lane); break;
            case 9: mid_round<3>(wtile, lane); break;
            default: mid_round<4>(wtile, lane); break;
            }
        } else {
            mid_round5(wtile, lane);
        }
        if (!kScales && claims) s_next[0] = claimed;
        __syncthreads();

        // ---- last round.  Thread (rl, u) owns the unit u of eight coordinates of rows rl + kBRowStep m: lanes 0-7 of
        // a quarter warp cover four units of two adjacent rows, whose XOR patterns differ in bit 0.
        const int rl = tid >> 2, u = tid & 3, x = rl & 7;
        float4 a[8], b[8];
        float4 *pa = tile + rl * 8 + ((2 * u) ^ x), *pb = tile + rl * 8 + ((2 * u + 1) ^ x);
        if constexpr (KIND == 0) {
            switch (k) {
            case 13: unit_load<3, 8 * kBRowStep>(pa, pb, a, b); break;
            case 12: unit_load<2, 8 * kBRowStep>(pa, pb, a, b); break;
            case 11: unit_load<1, 8 * kBRowStep>(pa, pb, a, b); break;
            default: unit_load<0, 8 * kBRowStep>(pa, pb, a, b); break;
            }
        } else {
            unit_load<3, 8 * kBRowStep>(pa, pb, a, b);
        }
        if constexpr (CLUSTER) {
            // back in place, then one position from all tiles
#pragma unroll
            for (int m = 0; m < 8; ++m) { pa[m * 8 * kBRowStep] = a[m]; pb[m * 8 * kBRowStep] = b[m]; }
            cluster_arrive();
            cluster_wait();
            const uint32_t own = (uint32_t)__cvta_generic_to_shared(tile);
            const uint32_t row = (rank << (kBLog2 - 5 - E)) + (uint32_t)rl, ca = (uint32_t)((2 * u) ^ x) << 4, cb = (uint32_t)((2 * u + 1) ^ x) << 4;
            unit_gather<E, kBRowStep>(own, row, ca, cb, a, b);
        }
        uint32_t next_task = 0u;
        if constexpr (kScales) {
            // every worker's sums of squares of this tile are in place
            cluster_wait();
            if (CLAIMS && P.head != nullptr && task >= groups) next_task = cluster_load_u32(cluster_map((uint32_t)__cvta_generic_to_shared(&s_next[par]), 0));
            block_scales<kBLog2>(P, (uint32_t)__cvta_generic_to_shared(s_sq[par]), blk0, bc, wl == 0u, tid);
        }
        // ---- the tile is in registers: start the next task's load
        const uint32_t cur_wl = wl;
        const uint64_t j_out = !CLUSTER ? j0 + 32u * rl + 8u * u
                                       : ((uint64_t)unit << k) + ((uint64_t)rank << (kBLog2 - E)) + 32u * rl + 8u * u;
        // (the task after the next one is stored behind the barrier below; a cluster reads its first CTA's)
        if (!CLAIMS) {
            task += groups;
            if (kVectors) {
                unit += unit_step;
                wl += wl_step;
                if (wl >= P.n_local) { wl -= P.n_local; ++unit; }
            } else {
                unit = task;
            }
        } else {
            if (task < groups || P.head == nullptr) task += groups;
            else if (kScales) task = next_task;
            else if (!CLUSTER) task = s_next[0];
            else task = cluster_load_u32(cluster_map((uint32_t)__cvta_generic_to_shared(&s_next[0]), 0));
            if (task < P.tasks) split_task();
        }
        fence_proxy_async();                           // these reads before the next load's writes
        if (!CLUSTER) {
            __syncthreads();
            if (task < P.tasks) {
                if (tid == 0 && by_tma(unit)) start_load(unit, wl);
                if (!kForward) prefetch_inputs(unit, wl);
            }
        } else {
            cluster_arrive();                          // waited for after the first half of the epilogue
        }
        if (CLUSTER) {
            unit_stages<E>(a, b);
        }

        // ---- epilogue: two iterations over four rows (unrolled over all eight it does not fit the instruction
        // cache); the second iteration's rows move down the register arrays
        const float gf = (float)P.granularity;
        const uint32_t my_lut = lut_lane_addr(lut, tid);
        // Offsets from the thread's first unit fit 32 bits; the rounding calls of a tile (of a cluster's block)
        // share the high word of their counter (see EpilogueCtx).
        const uint64_t limit = kForward ? P.d_pad : P.d;
        const uint32_t left = j_out >= limit ? 0u : (uint32_t)min(limit - j_out, (uint64_t)1 << 31);
        const uint32_t call_lo = (uint32_t)(j_out >> 3), call_hi = (uint32_t)(j_out >> 35);
        float *rot = kForward ? static_cast<float *>(rotated.p[cur_wl]) : nullptr;
        if (rot != nullptr) rot += j_out;
        unsigned char *packed = kQuant ? static_cast<unsigned char *>(outp.p[cur_wl]) + j_out / 8 * BITS : nullptr;
        uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll 1
        for (uint32_t half = 0; half < 2; ++half) {
#pragma unroll
            for (uint32_t mm = 0; mm < 4; ++mm) {
                const uint32_t m = 4u * half + mm;
                const uint32_t off = ((m & (C - 1u)) << kBLog2) + (m >> E) * (32u * kBRowStep);
                const float4 ra = scale4(a[mm], P.c_block), rb = scale4(b[mm], P.c_block);
                if (kForward) {
                    if (rot != nullptr && off < left) {
                        *reinterpret_cast<float4 *>(rot + off) = ra;
                        *reinterpret_cast<float4 *>(rot + off + 4) = rb;
                    }
                    const float r[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
                    if constexpr (kRange) {
                        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
                        if (off < left) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const uint32_t key = float_key(r[e]);
                                lo = min(lo, key);
                                hi = max(hi, key);
                            }
                        }
                        if (KIND != 0 || k >= (uint32_t)kBLog2) {
                            kmin = min(kmin, lo);
                            kmax = max(kmax, hi);
                        } else {
                            // a warp's units of one m are 256 consecutive coordinates
                            if (k >= 8u) {
                                lo = __reduce_min_sync(0xFFFFFFFFu, lo);
                                hi = __reduce_max_sync(0xFFFFFFFFu, hi);
                            }
                            if (off < left && (k < 8u || lane == 0)) add_range(P.range_keys, P.nblocks, (j_out + off) >> k, lo, hi);
                        }
                    } else {
                        const float2 kc = bc[KIND != 0 ? 0u : ((32u * rl + 8u * u + off) >> k)];
                        const uint4 rnd = philox4x32_10(call_lo + (off >> 3), call_hi, P.worker_base + cur_wl, P.round, keys);
                        const uint64_t z = quantize8<BITS, IDENTITY>(r, kc.x, kc.y, gf, rnd, my_lut);
                        if (off < left) store_unit<BITS>(packed, off, z);
                    }
                } else if (off < left) {
                    float *out = static_cast<float *>(outp.p[kEF ? cur_wl : 0]) + j_out;
                    const float *xs = kEF ? static_cast<const float *>(rotated.p[cur_wl]) + j_out : nullptr;
                    const uint32_t word = ((m & (C - 1u)) << (kBLog2 - 5 - E)) + (uint32_t)rl + kBRowStep * (m >> E);
                    const uint32_t bits = sw[kBSignWords * par + word] >> (8 * u);
                    float4 oa = flip4(ra, bits), ob = flip4(rb, bits >> 4);
                    if (off + 8 <= left) {
                        if (kEF) {
                            const float4 xa = ld_global_once(reinterpret_cast<const float4 *>(xs + off));
                            const float4 xb = ld_global_once(reinterpret_cast<const float4 *>(xs + off + 4));
                            oa = make_float4(xa.x - oa.x, xa.y - oa.y, xa.z - oa.z, xa.w - oa.w);
                            ob = make_float4(xb.x - ob.x, xb.y - ob.y, xb.z - ob.z, xb.w - ob.w);
                        }
                        *reinterpret_cast<float4 *>(out + off) = oa;
                        *reinterpret_cast<float4 *>(out + off + 4) = ob;
                    } else {
                        const float o[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
                        for (int e = 0; e < 8; ++e)
                            if (off + e < left) out[off + e] = kEF ? xs[off + e] - o[e] : o[e];
                    }
                }
            }
            if (CLUSTER && half == 0u) {
                cluster_wait();                        // every CTA has gathered: the tile is free
                if (task < P.tasks) {
                    if (tid == 0 && by_tma(unit)) start_load(unit, wl);
                    if (!kForward) prefetch_inputs(unit, wl);
                }
            }
#pragma unroll
            for (int mm = 0; mm < 4; ++mm) { a[mm] = a[mm + 4]; b[mm] = b[mm + 4]; }
        }
        if (kRange && (KIND != 0 || k >= (uint32_t)kBLog2)) {
            kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
            kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
            if (lane == 0) add_range(P.range_keys, P.nblocks, j_out >> k, kmin, kmax);
        }
    }
    if (kScales) { cluster_arrive(); cluster_wait(); }  // (the others read this CTA's sums)
    // the last CTA clears the task counter for the next launch and finishes the ranges
    if ((CLAIMS && P.head != nullptr) || (kRange && P.range_out != nullptr)) {
        __shared__ uint32_t s_left;
        __threadfence();
        __syncthreads();
        if (thread == 0) s_left = atomicAdd(P.exited, 1u);
        __syncthreads();
        if (s_left == gridDim.x - 1) {
            __threadfence();
            if (kRange && P.range_out != nullptr) finish_ranges(P.range_keys, P.nblocks, P.range_out, P.dev, thread, kBThreads);
            if (thread == 0) {
                if (CLAIMS && P.head != nullptr) *P.head = 0u;
                *P.exited = 0u;
            }
        }
    }
}

// Which kernels can claim their tasks.  The claim costs error feedback, the exact range and aggregate + decompress 0.1 to
// 0.4 us a launch even where nothing is claimed (with / without, 4 bits: error feedback of 2 x 3000 in 2^11 blocks
// 5.46 / 5.06 us, of 4 x 3 M in 2^12 28.1 / 27.7; range 6.17 / 5.88; aggregate + decompress 4.85 / 4.65): they have a kernel
// of each.  Compress loses 0.1 us (and has most of the kernels), decompress is level.  Clusters of eight have two tasks
// each at most and claim none: compress, error feedback and the range do without the code (bf16 with 3 bits, seven blocks of
// 2^17 from two workers, 14.6 / 13.5 us), decompress and the tail are 0.2 to 0.5 us of 11 to 13 faster as compiled with it.
constexpr bool block_claims(int mode, int kind, bool wanted)
{
    const bool both = mode == kErrorFeedback || mode == kRangeF32 || mode == kAggDecompress;
    const bool inverse = mode == kDecompress8 || mode == kDecompress16 || mode == kDecompress32 || mode == kAggDecompress;
    return kind < 3 ? wanted || !both : inverse;
}

template <int MODE, int KIND, bool WANTED>
static const void *pick(uint32_t bits, bool identity)
{
#define THC_BLK(B, I) reinterpret_cast<const void *>(thc_block_kernel<MODE, B, I, KIND, block_claims(MODE, KIND, WANTED)>)
    constexpr bool fused = MODE == kCompressF32Fused || MODE == kCompressBF16Fused;
    if constexpr (fused && KIND > 1) {
        return nullptr;
    } else if constexpr (MODE == kErrorFeedback) {
        switch (bits) {
        case 1: return THC_BLK(1, true);
        case 2: return THC_BLK(2, true);
        case 3: return THC_BLK(3, true);
        case 4: return THC_BLK(4, true);
        default: return THC_BLK(8, true);
        }
    } else if constexpr (MODE == kCompressF32 || MODE == kCompressBF16 || fused) {
        switch (bits) {
        case 1: return identity ? THC_BLK(1, true) : THC_BLK(1, false);
        case 2: return identity ? THC_BLK(2, true) : THC_BLK(2, false);
        case 3: return identity ? THC_BLK(3, true) : THC_BLK(3, false);
        case 4: return identity ? THC_BLK(4, true) : THC_BLK(4, false);
        default: return THC_BLK(8, true);              // (the only table there is)
        }
    } else {
        return THC_BLK(4, true);
    }
#undef THC_BLK
}

template <int KIND, bool WANTED>
static const void *pick_mode(PipeMode mode, uint32_t bits, bool identity)
{
    switch (mode) {
    case kCompressF32: return pick<kCompressF32, KIND, WANTED>(bits, identity);
    case kCompressBF16: return pick<kCompressBF16, KIND, WANTED>(bits, identity);
    case kCompressF32Fused: return pick<kCompressF32Fused, KIND, WANTED>(bits, identity);
    case kCompressBF16Fused: return pick<kCompressBF16Fused, KIND, WANTED>(bits, identity);
    case kDecompress8: return pick<kDecompress8, KIND, WANTED>(bits, identity);
    case kDecompress16: return pick<kDecompress16, KIND, WANTED>(bits, identity);
    case kDecompress32: return pick<kDecompress32, KIND, WANTED>(bits, identity);
    case kErrorFeedback: return pick<kErrorFeedback, KIND, WANTED>(bits, identity);
    case kRangeF32: return pick<kRangeF32, KIND, WANTED>(bits, identity);
    case kAggDecompress: return pick<kAggDecompress, KIND, WANTED>(bits, identity);
    default: return nullptr;
    }
}

const void *block_kernel(PipeMode mode, uint32_t bits, bool identity, uint32_t k, bool claims)
{
    if (claims) {
        switch (block_kind(k)) {
        case 0: return pick_mode<0, true>(mode, bits, identity);
        case 1: return pick_mode<1, true>(mode, bits, identity);
        case 2: return pick_mode<2, true>(mode, bits, identity);
        default: break;
        }
    }
    switch (block_kind(k)) {
    case 0: return pick_mode<0, false>(mode, bits, identity);
    case 1: return pick_mode<1, false>(mode, bits, identity);
    case 2: return pick_mode<2, false>(mode, bits, identity);
    case 3: return pick_mode<3, false>(mode, bits, identity);
    default: return pick_mode<4, false>(mode, bits, identity);
    }
}

}  // namespace thc
