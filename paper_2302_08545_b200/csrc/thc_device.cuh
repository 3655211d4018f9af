// Device-side building blocks of libthc: counter RNG, packed-fp32 butterflies, the
// swizzled shared-memory Hadamard rounds and the per-coordinate quantiser.
//
// Arithmetic contract (what makes results reproducible bit for bit):
//   * every fp32 operation is a single IEEE round-to-nearest operation; the file is
//     compiled with -fmad=false, so only the fmaf() calls written here are fused;
//   * the Hadamard transform is radix-2 with stages in ascending stride order and one
//     multiplication by (float)(1/sqrt(B)) at the end (THC paper, Section 5.1: the RHT is
//     (1/sqrt d) H D x; the paper fixes no evaluation order, this is the library's);
//   * random bits come from Philox4x32-10 keyed by the shared seed.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/thc.h"

namespace thc {

constexpr int kChunkLog2 = 14;                 // coordinates whose squares one CTA sums (prepare)
constexpr int kThreads = 256;

constexpr int kPrepCounters = 4096;

// Lives in the context's device block.
struct DeviceBlock {
    uint32_t status;             // THC_STATUS_* bits
    uint32_t pad_[31];
    uint32_t counters[5632];     // scheduling counters (self-resetting), 128-byte aligned
    uint32_t prep_counters[kPrepCounters];     // chunks done per RHT block in thc_prepare (self-resetting)
    uint32_t range_keys[2 * kPrepCounters];    // exact range, up to as many blocks (self-resetting)
    uint4    lut[256];           // by floor(u*g): (-T[z0] as float, 65536/(T[z0+1]-T[z0]), z0, 0)
    uint32_t table[256];         // T
};

// ------------------------------------------------------------------------ dependent launches
// Every kernel is launched so that it may start before the launch before it is complete (launch_after in
// thc.cu): the launch itself, the tables and the barriers are set up while the other's writes drain.  Each CTA
// calls depend_on_previous() before it touches anything that a launch writes; it returns when the previous
// launch, which called it too, is complete and its writes are visible.  No kernel releases the next one
// early (griddepcontrol.launch_dependents): CTAs that move in beside a kernel with another split of
// shared memory and L1 keep that split (a pipeline kernel next to a streaming one: 8 us of 144 lost).
__device__ __forceinline__ void depend_on_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of what other launches wrote: volatile and coherent, so that none of them is moved in front of
// depend_on_previous() (loads through the read-only path may be).
__device__ __forceinline__ uint4 ld_global(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_global_once(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_global_once(const float4 *p)
{
    const uint4 v = ld_global_once(reinterpret_cast<const uint4 *>(p));
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
__device__ __forceinline__ uint2 ld_global(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const uint16_t *p)
{
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_global(const unsigned char *p)
{
    uint32_t v;
    asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_global(const float *p) { return __uint_as_float(ld_global(reinterpret_cast<const uint32_t *>(p))); }

struct PhiloxKeys { uint32_t k[20]; };         // the ten round keys, precomputed on the host

// Philox4x32-10 (Salmon et al., SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               const PhiloxKeys &keys)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * (uint64_t)c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * (uint64_t)c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ keys.k[2 * r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ keys.k[2 * r + 1];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
    }
    return make_uint4(c0, c1, c2, c3);
}

// Sign diagonal D of the RHT (Section 5.1; "D^r" in Algorithm 3): one Philox call covers
// 128 consecutive padded coordinates, counter = (j/128 lo, j/128 hi, 0xFFFFFFFF, round).
__device__ __forceinline__ uint4 sign_call(uint64_t j, uint32_t round, const PhiloxKeys &keys)
{
    const uint64_t call = j >> 7;
    return philox4x32_10((uint32_t)call, (uint32_t)(call >> 32), 0xFFFFFFFFu, round, keys);
}

// Rounding variates (Section 4.1 needs one uniform per coordinate; Appendix A.2 asks that
// workers draw independently): one call covers 8 consecutive coordinates, 16 bits each,
// counter = (j/8 lo, j/8 hi, worker, round).
__device__ __forceinline__ uint4 round_call(uint64_t j, uint32_t worker, uint32_t round,
                                            const PhiloxKeys &keys)
{
    const uint64_t call = j >> 3;
    return philox4x32_10((uint32_t)call, (uint32_t)(call >> 32), worker, round, keys);
}

// ------------------------------------------------------------------------ clamp range
// Range [lo, hi] of an RHT block (Algorithm 2's m and M).  Norm mode (Section 5.3): the
// scales array holds M per block and m = -M.  Exact mode (Algorithm 1's preliminary stage
// applied to the rotated coordinates): it holds nblocks minima followed by nblocks maxima.
struct BlockRange { float lo, hi; };

__device__ __forceinline__ BlockRange block_range(const float *scales, uint64_t r, uint64_t nblocks,
                                                  uint32_t exact)
{
    BlockRange b;
    if (exact) { b.lo = ld_global(scales + r); b.hi = ld_global(scales + nblocks + r); }
    else { b.hi = ld_global(scales + r); b.lo = -b.hi; }
    return b;
}

// (kappa, offset) of u = sat(fma(r, kappa, offset)): 1/(hi - lo) and -lo/(hi - lo), which for
// lo = -hi are 1/(2M) and exactly 1/2; (0, 0) marks a degenerate block (every index 0).
__device__ __forceinline__ float2 compress_constants(BlockRange b)
{
    if (!(b.hi > b.lo) || !isfinite(b.hi) || !isfinite(b.lo)) return make_float2(0.f, 0.f);
    const double w = (double)b.hi - (double)b.lo;
    return make_float2((float)(1.0 / w), (float)(-(double)b.lo / w));
}

// (step, base) of v = fma(Y, step, base): (hi - lo)/(g * divisor) and lo; (0, 0) for a
// degenerate block (decodes to zeros).  hi == lo (a constant block: every index is 0) gives
// step 0 and base lo: the estimate line of Algorithm 2 with M = m.
__device__ __forceinline__ float2 decode_constants(BlockRange b, uint32_t g, uint32_t divisor)
{
    if (!(b.hi >= b.lo) || !isfinite(b.hi) || !isfinite(b.lo)) return make_float2(0.f, 0.f);
    const double w = (double)b.hi - (double)b.lo;
    return make_float2((float)(w / ((double)g * (double)divisor)), b.lo);
}

// Order-preserving map of fp32 bit patterns onto unsigned integers (for atomic min / max).
__device__ __forceinline__ uint32_t float_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return u ^ ((u >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k)
{
    return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xFFFFFFFFu));
}

// Exact range: the keys are nblocks complements of the smallest key, then nblocks largest keys, so that
// both start at 0 and are raised by atomicMax.
__device__ __forceinline__ void add_range(uint32_t *keys, uint64_t nblocks, uint64_t r, uint32_t kmin, uint32_t kmax)
{
    atomicMax(keys + r, ~kmin);
    atomicMax(keys + nblocks + r, kmax);
}

// The keys of block r become its minimum and maximum in `scales` and are 0 again.  A block with a
// non-finite rotated coordinate gets (0, 0) and THC_STATUS_NONFINITE.
__device__ __forceinline__ void finish_range(uint32_t *keys, uint64_t nblocks, uint64_t r, float *scales, DeviceBlock *dev)
{
    float lo = key_float(~__ldcg(keys + r)), hi = key_float(__ldcg(keys + nblocks + r));
    keys[r] = 0u;
    keys[nblocks + r] = 0u;
    uint32_t flags = 0;
    if (!isfinite(lo) || !isfinite(hi)) { lo = 0.0f; hi = 0.0f; flags |= THC_STATUS_NONFINITE; }
    if (hi == 0.0f && lo == 0.0f) flags |= THC_STATUS_ZERO_BLOCK;   // a constant block decodes exactly
    scales[r] = lo;
    scales[nblocks + r] = hi;
    if (flags) atomicOr(&dev->status, flags);
}
__device__ __forceinline__ void finish_ranges(uint32_t *keys, uint64_t nblocks, float *scales, DeviceBlock *dev, int tid, int threads)
{
    for (uint64_t r = tid; r < nblocks; r += threads) finish_range(keys, nblocks, r, scales, dev);
}

// ---------------------------------------------------------------- packed fp32 arithmetic
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// a - b as fma(b, -1, a): one rounding of the exact difference, i.e. the same result as a
// subtraction, expressed with the packed intrinsic so that the compiler keeps operands in
// register pairs.
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}

// One radix-2 butterfly on four independent columns: (a, b) <- (a + b, a - b).
__device__ __forceinline__ void butterfly(float4 &a, float4 &b)
{
    const float2 alo = make_float2(a.x, a.y), ahi = make_float2(a.z, a.w);
    const float2 blo = make_float2(b.x, b.y), bhi = make_float2(b.z, b.w);
    const float2 slo = add2(alo, blo), shi = add2(ahi, bhi);
    const float2 dlo = sub2(alo, blo), dhi = sub2(ahi, bhi);
    a = make_float4(slo.x, slo.y, shi.x, shi.y);
    b = make_float4(dlo.x, dlo.y, dhi.x, dhi.y);
}

// Stages of stride 1 and 2 inside one 16-byte chunk (coordinates 4q .. 4q+3).
__device__ __forceinline__ float4 stages01(float4 v)
{
    const float x = v.x + v.y, y = v.x - v.y, z = v.z + v.w, w = v.z - v.w;
    const float2 s = add2(make_float2(x, y), make_float2(z, w));
    const float2 d = sub2(make_float2(x, y), make_float2(z, w));
    return make_float4(s.x, s.y, d.x, d.y);
}

__device__ __forceinline__ float4 scale4(float4 v, float c)
{
    const float2 c2 = make_float2(c, c);
    const float2 lo = __fmul2_rn(make_float2(v.x, v.y), c2);
    const float2 hi = __fmul2_rn(make_float2(v.z, v.w), c2);
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Flip the signs of a chunk by bits [0,4) of `bits` (bit e set -> element e negated).
__device__ __forceinline__ float4 flip4(float4 v, uint32_t bits)
{
    v.x = __uint_as_float(__float_as_uint(v.x) ^ ((bits << 31) & 0x80000000u));
    v.y = __uint_as_float(__float_as_uint(v.y) ^ ((bits << 30) & 0x80000000u));
    v.z = __uint_as_float(__float_as_uint(v.z) ^ ((bits << 29) & 0x80000000u));
    v.w = __uint_as_float(__float_as_uint(v.w) ^ ((bits << 28) & 0x80000000u));
    return v;
}

// --------------------------------------------------------------------------- quantiser
// The quantiser's table in shared memory, indexed by f = floor(u g): what the rounding rule
// needs about the table interval [T[z0], T[z0+1]] that holds f.  Consecutive entries are 128
// bytes apart and every entry is replicated over lanes so that a warp's look-ups (random f per
// lane) never meet in a bank: 16 copies of 8 bytes (R16 = 65536 / gap as fp32, bf16(-T[z0]) << 16 | z0: table
// values up to 255 are exact in bf16).  Indices of 8 bits need none: 256 rising values up to g <= 255 are the identity.
constexpr int kLutEntryBytes = 128;

__device__ __forceinline__ void lut_fill(unsigned char *lut, const DeviceBlock *dev, uint32_t g, int tid, int nthreads)
{
    for (int idx = tid; idx < (int)(g + 1) * 16; idx += nthreads) {
        const uint4 e = dev->lut[idx / 16];
        reinterpret_cast<uint2 *>(lut)[idx] = make_uint2(e.y, (e.x & 0xFFFF0000u) | e.z);
    }
}

// Shared-space byte address of this lane's copy of entry 0, minus 0x4B000000 * 128: the bits of
// the float 2^23 + f, times 128, plus this value is the address of entry f.
__device__ __forceinline__ uint32_t lut_lane_addr(const unsigned char *lut, int lane)
{
    return (uint32_t)__cvta_generic_to_shared(lut) + (uint32_t)(lane & 15) * 8u - 0x4B000000u * (uint32_t)kLutEntryBytes;
}

// Stochastic quantisation of four consecutive rotated coordinates to table indices
// (Algorithm 2, worker lines; Section 4.1 for the rounding rule):
//   u = sat(fma(r, kappa, offset))          position in [m, M] on the unit interval, truncated
//   f = floor(u * g)                         (one round-down fma onto 2^23; exact)
//   z0 = index of the table value at or below u*g, delta = fma(u, g, -T[z0])
//   up iff u16 < RN(2^16 delta / gap)        (one fma onto 2^23, integer compare)
// kappa = 1/(2M) and offset = 1/2; kappa = offset = 0 encodes a degenerate block (index 0).
// w0, w1: the four 16-bit variates.  `lut_addr` comes from lut_lane_addr (unused for the identity
// table).  Returns the indices packed BITS apiece, coordinate 0 in the low bits: the compare is the
// carry of an addition, and a multiply-add with carry shifts the indices so far, appends z0 and
// adds it.  What is added for z0 is a whole word of which only the low half (table) or the low 24 bits
// (identity: the bits of 2^23 + f) mean anything, so the bits above 4 BITS are not defined (join_units
// cuts them off; 8 bits: the one 0x4B000000 that is left is taken off here).
// Bound by dispatch slots.  What allows it is packed, two coordinates to an instruction; the variates are
// inverted two at a time.  Cycles per coordinate of an SM's 128 lanes, alone, 12 warps per SM: 4 bits
// 12.9 -> 11.5, 2 bits identity 10.5 -> 8.0, 1 bit 10.5 -> 4.5 (its f is 0 below u = 1, where 2^16 u is
// above every variate, so the carry is the index).
template <int BITS, bool IDENTITY>
__device__ __forceinline__ uint32_t quantize4(float r0, float r1, float r2, float r3, float kappa, float offset,
                                              float gf, uint32_t w0, uint32_t w1, uint32_t lut_addr)
{
    static_assert(IDENTITY || BITS <= 4, "8 bits: identity");
    const float r[4] = {r0, r1, r2, r3};
    const uint32_t words[2] = {w0, w1};
    const float2 big = make_float2(8388608.0f, 8388608.0f), g2 = make_float2(gf, gf);
    uint32_t acc = 0u;
#pragma unroll
    for (int p = 1; p >= 0; --p) {
        float2 u, tau;
        asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(u.x) : "f"(r[2 * p]), "f"(kappa), "f"(offset));
        asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(u.y) : "f"(r[2 * p + 1]), "f"(kappa), "f"(offset));
        uint32_t zw[2] = {0u, 0u};
        if (IDENTITY && BITS == 1) {
            tau = __ffma2_rn(u, make_float2(65536.0f, 65536.0f), big);
        } else {
            const float2 t = __ffma2_rd(u, g2, big);           // 2^23 + floor(u * g)
            if (IDENTITY) {
                const float2 delta = __ffma2_rn(u, g2, __ffma2_rn(t, make_float2(-1.0f, -1.0f), big));
                tau = __ffma2_rn(delta, make_float2(65536.0f, 65536.0f), big);
                zw[0] = __float_as_uint(t.x);
                zw[1] = __float_as_uint(t.y);
            } else {
                const float tf[2] = {t.x, t.y};
                float nt[2], r16[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t a = __float_as_uint(tf[e]) * (uint32_t)kLutEntryBytes + lut_addr;
                    uint32_t x, y;
                    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x), "=r"(y) : "r"(a));
                    nt[e] = __uint_as_float(y & 0xFFFF0000u);
                    zw[e] = y;
                    r16[e] = __uint_as_float(x);
                }
                const float2 delta = __ffma2_rn(u, g2, make_float2(nt[0], nt[1]));
                tau.x = fmaf(delta.x, r16[0], 8388608.0f);
                tau.y = fmaf(delta.y, r16[1], 8388608.0f);
            }
        }
        const float tauf[2] = {tau.x, tau.y};
        const uint32_t inv = ~words[p];
#pragma unroll
        for (int e = 1; e >= 0; --e) {
            // ~ of the bits of 2^23 + u16
            const uint32_t nub = __byte_perm(inv, 0xB4FFFFFFu, e ? 0x7632 : 0x7610);
            // carry out of tau + ~ub: ub < tau
            if (IDENTITY && BITS == 1)
                asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %0, %0;\n\t}"
                    : "+r"(acc) : "r"(__float_as_uint(tauf[e])), "r"(nub));
            else
                asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\tmadc.lo.u32 %0, %0, %4, %3;\n\t}"
                    : "+r"(acc) : "r"(__float_as_uint(tauf[e])), "r"(nub), "r"(zw[e]), "n"(1 << BITS));
        }
    }
    return IDENTITY && BITS == 8 ? acc - 0x4B000000u : acc;
}

// Two groups of four indices as one unit of eight, coordinate 0 in the low bits.
template <int BITS>
__device__ __forceinline__ uint64_t join_units(uint32_t lo, uint32_t hi)
{
    if constexpr (BITS == 8) {
        return (uint64_t)lo | ((uint64_t)hi << 32);
    } else if constexpr (BITS == 4) {
        return (uint64_t)__byte_perm(lo, hi, 0x5410);
    } else {
        constexpr uint32_t mask = (1u << (4 * BITS)) - 1u;
        return (uint64_t)((lo & mask) | ((hi & mask) << (4 * BITS)));
    }
}

// Eight consecutive coordinates (see quantize4).
template <int BITS, bool IDENTITY>
__device__ __forceinline__ uint64_t quantize8(const float (&r)[8], float kappa, float offset,
                                              float gf, uint4 rnd, uint32_t lut_addr)
{
    const uint32_t lo = quantize4<BITS, IDENTITY>(r[0], r[1], r[2], r[3], kappa, offset, gf, rnd.x, rnd.y, lut_addr);
    const uint32_t hi = quantize4<BITS, IDENTITY>(r[4], r[5], r[6], r[7], kappa, offset, gf, rnd.z, rnd.w, lut_addr);
    return join_units<BITS>(lo, hi);
}

// Eight 3-bit indices (24 bits, coordinate 0 in the low bits) go to bytes 3 (j/8) .. +2.
__device__ __forceinline__ void store_packed3(unsigned char *pk, uint64_t j, uint32_t z)
{
    unsigned char *p = pk + 3 * (j >> 3);
    p[0] = (unsigned char)z;
    p[1] = (unsigned char)(z >> 8);
    p[2] = (unsigned char)(z >> 16);
}

// The eight indices of coordinates j .. j+7 (j a multiple of 8) to their place in the stream.
template <int BITS>
__device__ __forceinline__ void store_unit(unsigned char *pk, uint64_t j, uint64_t z)
{
    if constexpr (BITS == 8) *reinterpret_cast<uint2 *>(pk + j) = make_uint2((uint32_t)z, (uint32_t)(z >> 32));
    else if constexpr (BITS == 4) *reinterpret_cast<uint32_t *>(pk + j / 2) = (uint32_t)z;
    else if constexpr (BITS == 3) store_packed3(pk, j, (uint32_t)z);
    else if constexpr (BITS == 2) *reinterpret_cast<uint16_t *>(pk + j / 4) = (uint16_t)z;
    else pk[j / 8] = (unsigned char)z;
}

// ------------------------------------------------------------------------ small helpers
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

__device__ __forceinline__ float4 load_f32x4_masked(const float *x, uint64_t j, uint64_t d)
{
    if (j + 4 <= d) return ld_global_once(reinterpret_cast<const float4 *>(x + j));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j + 0 < d) v.x = ld_global(x + j + 0);
    if (j + 1 < d) v.y = ld_global(x + j + 1);
    if (j + 2 < d) v.z = ld_global(x + j + 2);
    if (j + 3 < d) v.w = ld_global(x + j + 3);
    return v;
}

// Geometry of a tile: 2^row_log2 rows, row_stride coordinates apart, of 2^col_log2 consecutive ones.
struct TileGeom {
    uint64_t row_stride;
    uint32_t row_log2, col_log2;
    uint32_t round;
};

// Sign words of every row of the tile, 32 coordinates per word.
__device__ __forceinline__ void fill_sign_words(uint32_t *sw, const TileGeom &g, uint64_t base,
                                                const PhiloxKeys &keys, int tid,
                                                int nthreads = kThreads)
{
    const int cols = 1 << g.col_log2;
    const int words_per_row = max(1, cols >> 5);
    const int calls_per_row = max(1, cols >> 7);
    const int rows = 1 << g.row_log2;
    const int words_per_call = min(4, words_per_row);
    for (int q = tid; q < rows * calls_per_row; q += nthreads) {
        const int row = q / calls_per_row;
        const int cr = q - row * calls_per_row;
        const uint64_t j0 = base + (uint64_t)row * g.row_stride + (uint64_t)cr * 128;
        const uint4 ph = sign_call(j0, g.round, keys);
        const int first = (int)((j0 >> 5) & 3);
        for (int wi = 0; wi < words_per_call; ++wi) {
            const int src = first + wi;
            const uint32_t w = src == 0 ? ph.x : src == 1 ? ph.y : src == 2 ? ph.z : ph.w;
            sw[row * words_per_row + cr * 4 + wi] = w;
        }
    }
}

}  // namespace thc
