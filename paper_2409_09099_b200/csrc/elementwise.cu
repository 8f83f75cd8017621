// HBM-bound kernels of the S-STE linear layer: beta (Eq. 5), the fused
// projection + scale + 2:4 compression (Eq. 4, Sec. 4.2), the fused MVUE +
// compression of the output gradient (Sec. 5.1) and the FP8 scaling helpers
// (Sec. 5.2).  Every fp32 step is a single rounded operation (no FMA
// contraction) in a fixed order, so results are reproducible bit for bit.
#include "common.cuh"

namespace {

constexpr int EW_THREADS = 256;
constexpr int PC_ROWS = 32;                                  // rows of W per project+compress CTA
constexpr int PC_CHUNKS = PC_ROWS * 16 / EW_THREADS;         // 16-byte chunks per thread

// ---------------------------------------------------------------- an amax that the kernel in front has found

// The amax a kernel quantises with.  scratch NULL: it is in *amax.  Otherwise the kernel in front of this one has left it in
// *scratch only (as the bits of a non-negative fp32); this kernel publishes it in *amax, and the product behind it empties
// the scratch.  That keeps the amax kernel free of a last block's chain of atomics and fences, which was 2 of the 3-4 us
// that a small tensor's took.  (Counting this kernel's blocks to empty it here made them queue up at that address:
// project + compress of 45 M weights 35 -> 85 us.)
struct AmaxIn { float *amax; const unsigned int *scratch; };
__device__ __forceinline__ float amax_take(const AmaxIn &a, bool publish)
{
    if (!a.scratch) return *a.amax;
    const float v = __uint_as_float(*a.scratch);
    if (publish) *a.amax = v;
    return v;
}

// ---------------------------------------------------------------- two fp32 values per instruction

// Two fp32 values in one register pair: one instruction per operation for both (sm_100 f32x2), each lane a single
// rounded operation, subnormals included.
using f32x2 = unsigned long long;
// byte permute with the selector as the instruction takes it (four nibbles in the low half)
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }
// a <= b, a >= b as 1.0f / 0.0f (0 if either is a NaN), one instruction
__device__ __forceinline__ float one_if_le(float a, float b)
{
    float r;
    asm("set.le.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// ---------------------------------------------------------------- packed bf16, and bf16 terms of 32-bit sums

// halves of a and b equal: all ones (0 if either is a NaN)
__device__ __forceinline__ uint32_t bf_eq2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("set.eq.u32.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// half HI of a in a 32-bit sum, rounded once
template <int HI>
__device__ __forceinline__ float mix_add(uint32_t a, float c)
{
    float r;
    if (HI) asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tadd.rn.f32.bf16 %0, h, %2;\n\t}" : "=f"(r) : "r"(a), "f"(c));
    else asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %1;\n\tadd.rn.f32.bf16 %0, l, %2;\n\t}" : "=f"(r) : "r"(a), "f"(c));
    return r;
}

// ---------------------------------------------------------------- group of four: S_soft + kept pair

struct SoftGroup {
    float w[4];       // beta * S_soft (times the FP8 scale), pruned entries +0
    uint32_t p0, p1;  // kept positions, p0 < p1
};

// w01 = a0 | a1 << 16, w23 = a2 | a3 << 16 (bf16 bit patterns).  Written for instruction count (the kernel
// is bound by instruction issue): the threshold t = second-smallest magnitude comes from packed 16-bit
// min/max on the magnitude bits (bf16 magnitudes order like unsigned integers), sign(a)(|a| - t) is the single
// subtraction a - copysign(t, a), and the kept pair is the top two of four integer keys
// (magnitude << 2 | 3 - index: magnitude descending, index ascending; pairwise distinct) found with a
// seven-operation min/max network.
// MODE 0: the method's projection of a group with values that are not finite (project_group takes the others); MODE 1:
// interpolated threshold t = (1 - gamma) |t2| + gamma |t3| (Sec. 4.1); MODE 2: hard thresholding (Eq. 2), the kept pair
// unchanged.
template <bool FP8, int MODE>
__device__ __forceinline__ SoftGroup soft_group(uint32_t w01, uint32_t w23, float beta, float wscale, float gamma)
{
    SoftGroup r;
    const uint32_t m01 = w01 & 0x7fff7fffu, m23 = w23 & 0x7fff7fffu;
    // second-smallest of the four magnitudes, in both halves of t2
    const uint32_t lo = __vminu2(m01, m23), hi = __vmaxu2(m01, m23);
    const uint32_t lmax = __vmaxu2(lo, __byte_perm(lo, 0, 0x1032));
    const uint32_t hmin = __vminu2(hi, __byte_perm(hi, 0, 0x1032));
    const uint32_t t2 = __vminu2(lmax, hmin);
    uint32_t tb = t2 << 16;                             // fp32 bits of t
    if (MODE == 1) {                                    // third-smallest magnitude: the other of (lmax, hmin)
        const float t3 = __uint_as_float(__vmaxu2(lmax, hmin) << 16);
        tb = __float_as_uint(__fadd_rn(__fmul_rn(__fsub_rn(1.0f, gamma), __uint_as_float(tb)), __fmul_rn(gamma, t3)));
    }
    const float t = __uint_as_float(tb);
    const uint32_t ab[4] = {w01 << 16, w01 & 0xffff0000u, w23 << 16, w23 & 0xffff0000u};
    if (MODE != 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = __uint_as_float(ab[i]);
            const float st = __uint_as_float(tb | (ab[i] & 0x80000000u));     // copysign(t, a)
            float w = __fmul_rn(__fsub_rn(a, st), beta);                        // sign(a) (|a| - t) beta
            if (FP8) w = __fmul_rn(w, wscale);
            r.w[i] = (fabsf(a) > t) ? w : 0.0f;
        }
    }
    const uint32_t k0 = (m01 & 0xffffu) * 4u + 3u, k1 = (m01 >> 16) * 4u + 2u;
    const uint32_t k2 = (m23 & 0xffffu) * 4u + 1u, k3 = (m23 >> 16) * 4u;
    const uint32_t a = max(k0, k1), b = min(k0, k1), c = max(k2, k3), d = min(k2, k3);
    const uint32_t top1 = max(a, c), top2 = max(min(a, c), max(b, d));
    const uint32_t i1 = (top1 & 3u) ^ 3u, i2 = (top2 & 3u) ^ 3u;
    r.p0 = min(i1, i2);
    r.p1 = max(i1, i2);
    if (MODE == 2) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = __uint_as_float(ab[i]);
            float w = __fmul_rn(a, beta);
            if (FP8) w = __fmul_rn(w, wscale);
            const bool kept = (static_cast<uint32_t>(i) == r.p0) || (static_cast<uint32_t>(i) == r.p1);
            r.w[i] = (kept && fabsf(a) > 0.0f) ? w : 0.0f;      // a kept zero is +0 like every pruned entry
        }
    }
    return r;
}

// What the six comparisons of a group's magnitudes (i < j: m_i >= m_j, so that ties go to the lower index) come to, by table:
//   x: byte-permute selector of the two kept halfwords | kept nibble p0 | p1 << 2 in bits 16-19 | selector of the threshold's
//      halfword (the third in rank, the second-smallest magnitude) into the upper half of a word, in bits 24-31
//   y: 0x80 in byte i where position i is kept
// Entry number: bit k of the comparison (0,1) (0,2) (0,3) (1,2) (1,3) (2,3).  Codes that no order gives are filled alike.
constexpr int PROJECT_ENTRIES = 64;
struct ProjectTable { uint2 e[PROJECT_ENTRIES]; };
constexpr ProjectTable project_table()
{
    ProjectTable t{};
    for (int n = 0; n < PROJECT_ENTRIES; ++n) {
        int wins[4] = {0, 0, 0, 0}, k = 0;
        for (int i = 0; i < 4; ++i)
            for (int j = i + 1; j < 4; ++j, ++k) ++wins[(n >> k) & 1 ? i : j];
        int order[4] = {0, 1, 2, 3};       // by wins, descending (they are 3, 2, 1, 0 for every order of magnitudes)
        for (int a = 0; a < 4; ++a)
            for (int b = a + 1; b < 4; ++b)
                if (wins[order[b]] > wins[order[a]]) { const int o = order[a]; order[a] = order[b]; order[b] = o; }
        const int p0 = order[0] < order[1] ? order[0] : order[1], p1 = order[0] < order[1] ? order[1] : order[0], th = order[2];
        t.e[n].x = (0x1010u + 0x22u * p0 + 0x2200u * p1) | (static_cast<uint32_t>(p0 | (p1 << 2)) << 16) |
                   (static_cast<uint32_t>((2 * th) | ((2 * th + 1) << 4)) << 24);
        t.e[n].y = (0x80u << (8 * p0)) | (0x80u << (8 * p1));
    }
    return t;
}
__device__ const ProjectTable project_table_dev = project_table();

// The method's projection of one group by that table: w01 = a0 | a1 << 16, w23 = a2 | a3 << 16; v: the values before the
// cast, right in the kept positions only (a kept |a| = t gives +0: the fma adds +0 to an exact zero of either sign).
// The kernel is bound by instruction issue: sums and products run for two values at once, comparisons give 1.0 / 0.0 and are
// added up as subnormal floats whose bit pattern is the byte offset of the table entry (about 40 instructions per group,
// 84 with the rank by integer keys).
struct Projected { uint2 e; f32x2 v01, v23; };
template <bool FP8>
__device__ __forceinline__ Projected project_group(uint32_t w01, uint32_t w23, f32x2 beta2, f32x2 wscale2, const uint8_t *lut)
{
    const uint32_t a0 = w01 << 16, a1 = w01 & 0xffff0000u, a2 = w23 << 16, a3 = w23 & 0xffff0000u;
    const float m0 = fabsf(__uint_as_float(a0)), m1 = fabsf(__uint_as_float(a1));
    const float m2 = fabsf(__uint_as_float(a2)), m3 = fabsf(__uint_as_float(a3));
    constexpr int UNIT = 8;
    auto unit2 = [](int lo, int hi) { return pack2(__int_as_float(UNIT << lo), __int_as_float(UNIT << hi)); };
    f32x2 off2 = mul2(pack2(one_if_le(m1, m0), one_if_le(m2, m0)), unit2(0, 1));
    off2 = fma2(pack2(one_if_le(m3, m0), one_if_le(m2, m1)), unit2(2, 3), off2);
    off2 = fma2(pack2(one_if_le(m3, m1), one_if_le(m3, m2)), unit2(4, 5), off2);
    float o0, o1;
    unpack2(off2, o0, o1);
    Projected r;
    r.e = *reinterpret_cast<const uint2 *>(lut + __float_as_uint(o0) + __float_as_uint(o1));
    const uint32_t t = prmt(w01, w23, r.e.x >> 16) & 0x7fff0000u;         // fp32 bits of the threshold
    // sign(a) (|a| - t) as the single subtraction a - copysign(t, a)
    auto st = [&](uint32_t a) { return __uint_as_float((~a & 0x80000000u) | t); };       // -copysign(t, a)
    const f32x2 zero2 = both(0.0f);
    r.v01 = fma2(add2(pack2(__uint_as_float(a0), __uint_as_float(a1)), pack2(st(a0), st(a1))), beta2, zero2);
    r.v23 = fma2(add2(pack2(__uint_as_float(a2), __uint_as_float(a3)), pack2(st(a2), st(a3))), beta2, zero2);
    if (FP8) {
        r.v01 = mul2(r.v01, wscale2);
        r.v23 = mul2(r.v23, wscale2);
    }
    return r;
}

// ---------------------------------------------------------------- project + compress

// The two groups of eight consecutive features after the projection: kept values packed (bf16: 32 bits, FP8: 16 bits per group),
// all values packed (bf16: two words, FP8: word 0 per group), the metadata byte.
struct ProjectedChunk { uint32_t kept[2], dn[2][2], mbyte; };

// By rank on integer keys (soft_group), whatever the values.
template <bool FP8, int MODE>
__device__ __forceinline__ ProjectedChunk project_by_keys(const uint4 &in, float beta, float wscale, float gamma)
{
    const uint32_t raw[4] = {in.x, in.y, in.z, in.w};
    ProjectedChunk o;
    o.mbyte = 0;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const SoftGroup s = soft_group<FP8, MODE>(raw[2 * g], raw[2 * g + 1], beta, wscale, gamma);
        if (FP8) {
            const uint32_t e01 = __nv_cvt_float2_to_fp8x2(make_float2(s.w[0], s.w[1]), __NV_SATFINITE, __NV_E4M3);
            const uint32_t e23 = __nv_cvt_float2_to_fp8x2(make_float2(s.w[2], s.w[3]), __NV_SATFINITE, __NV_E4M3);
            o.dn[g][0] = e01 | (e23 << 16);
            o.kept[g] = __byte_perm(o.dn[g][0], 0, s.p0 | (s.p1 << 4) | 0x4400u);
        } else {
            const __nv_bfloat162 d01 = __floats2bfloat162_rn(s.w[0], s.w[1]);
            const __nv_bfloat162 d23 = __floats2bfloat162_rn(s.w[2], s.w[3]);
            o.dn[g][0] = *reinterpret_cast<const uint32_t *>(&d01);
            o.dn[g][1] = *reinterpret_cast<const uint32_t *>(&d23);
            // halfword p0 -> low half, halfword p1 -> high half
            o.kept[g] = __byte_perm(o.dn[g][0], o.dn[g][1], 0x1010u + 0x22u * s.p0 + 0x2200u * s.p1);
        }
        o.mbyte |= (s.p0 | (s.p1 << 2)) << (4 * g);
    }
    return o;
}

// Chunk c (of PC_ROWS x 16) of CTA (kb, rb) to where it belongs.
template <bool FP8>
__device__ __forceinline__ void put_chunk(const ProjectedChunk &o, int c, int kb, int rb, size_t row_chunks, void *vals,
                                          uint8_t *meta_s, void *dense)
{
    const int row = c >> 4, kc = c & 15;
    const uint32_t k = 8u * kc;
    const uint32_t arow = (rb & 3) * PC_ROWS + row;   // row inside the 128-row atom
    meta_s[(FP8 ? sste_meta_atom_byte8(arow, k) : sste_meta_atom_byte16(arow, k)) - 512u * (rb & 3)] = static_cast<uint8_t>(o.mbyte);
    const size_t chunk = (static_cast<size_t>(rb) * PC_ROWS + row) * row_chunks + kb * 16 + kc;   // in units of 8 input features
    if (FP8) {
        reinterpret_cast<uint32_t *>(vals)[chunk] = o.kept[0] | (o.kept[1] << 16);
        if (dense) reinterpret_cast<uint2 *>(dense)[chunk] = make_uint2(o.dn[0][0], o.dn[1][0]);
    } else {
        reinterpret_cast<uint2 *>(vals)[chunk] = make_uint2(o.kept[0], o.kept[1]);
        if (dense) reinterpret_cast<uint4 *>(dense)[chunk] = make_uint4(o.dn[0][0], o.dn[0][1], o.dn[1][0], o.dn[1][1]);
    }
}

// What the projection of a tile (32 rows x 128 features of W: a quarter of a metadata atom, 512 contiguous bytes of its image)
// needs besides its values; a thread handles two chunks of eight consecutive features.
struct ProjectOut {
    const uint4 *W;
    size_t row_chunks;
    float beta, wscale, gamma;
    void *vals;
    uint8_t *meta;
    void *dense;
};
__device__ __forceinline__ const uint4 *project_src(const uint4 *W, size_t row_chunks, int kb, int rb, int c)
{
    return W + (static_cast<size_t>(rb) * PC_ROWS + (c >> 4)) * row_chunks + kb * 16 + (c & 15);
}
// A tile's groups once more, by keys (the method's projection of values that are not all finite; all threads).
template <bool FP8>
__device__ __noinline__ void project_any_values(const uint4 *W, int kb, int rb, size_t row_chunks, float beta, float wscale, void *vals,
                                                uint8_t *meta_s, void *dense)
{
    for (int c = threadIdx.x; c < PC_ROWS * 16; c += EW_THREADS)
        put_chunk<FP8>(project_by_keys<FP8, 0>(*project_src(W, row_chunks, kb, rb, c), beta, wscale, 0.0f), c, kb, rb, row_chunks, vals,
                       meta_s, dense);
}
// One tile (all threads of the block); in: its chunks c = i * EW_THREADS + tid; meta_s: 512 bytes, lut: the table (MODE 0).
template <bool FP8, int MODE>
__device__ __forceinline__ void project_tile(const uint4 (&in)[PC_CHUNKS], int kb, int rb, const ProjectOut &p, uint8_t *meta_s,
                                             const uint2 *lut)
{
    const int tid = threadIdx.x;
    const f32x2 beta2 = both(p.beta), wscale2 = both(p.wscale);
    // An infinity or a NaN in a group or in a scale makes the sum of its values one (so may huge values, which only costs
    // time): the table's order of magnitudes is for numbers, and inf - inf is not the 0 of |a| = t.  Nor is a product with
    // beta = 0 (-0 for a negative value, which the fma's + 0 loses).
    bool plain = p.beta != 0.0f;
#pragma unroll
    for (int i = 0; i < PC_CHUNKS; ++i) {
        ProjectedChunk o;
        if (MODE == 0) {
            const uint32_t raw[4] = {in[i].x, in[i].y, in[i].z, in[i].w};
            f32x2 sum;
            o.mbyte = 0;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const Projected s = project_group<FP8>(raw[2 * g], raw[2 * g + 1], beta2, wscale2, reinterpret_cast<const uint8_t *>(lut));
                const uint32_t nib = (s.e.x >> 16) & 0xfu;
                sum = g == 0 ? add2(s.v01, s.v23) : add2(sum, add2(s.v01, s.v23));
                float v[4];
                unpack2(s.v01, v[0], v[1]);
                unpack2(s.v23, v[2], v[3]);
                // masks of the kept positions: the selector's high bit replicates a byte's sign bit
                if (FP8) {
                    const uint32_t e01 = __nv_cvt_float2_to_fp8x2(make_float2(v[0], v[1]), __NV_SATFINITE, __NV_E4M3);
                    const uint32_t e23 = __nv_cvt_float2_to_fp8x2(make_float2(v[2], v[3]), __NV_SATFINITE, __NV_E4M3);
                    const uint32_t all = prmt(e01, e23, 0x5410);
                    o.dn[g][0] = all & prmt(s.e.y, 0, 0xba98);
                    o.kept[g] = prmt(all, 0, 0x4400u | (nib & 3u) | ((nib & 12u) << 2));
                } else {
                    const __nv_bfloat162 d01 = __floats2bfloat162_rn(v[0], v[1]), d23 = __floats2bfloat162_rn(v[2], v[3]);
                    const uint32_t w01 = *reinterpret_cast<const uint32_t *>(&d01), w23 = *reinterpret_cast<const uint32_t *>(&d23);
                    o.dn[g][0] = w01 & prmt(s.e.y, 0, 0x9988);
                    o.dn[g][1] = w23 & prmt(s.e.y, 0, 0xbbaa);
                    o.kept[g] = prmt(w01, w23, s.e.x);
                }
                o.mbyte |= nib << (4 * g);
            }
            float lo, hi;
            unpack2(sum, lo, hi);
            plain = plain && fabsf(lo + hi) < INFINITY;
        } else {
            o = project_by_keys<FP8, MODE>(in[i], p.beta, p.wscale, p.gamma);
        }
        put_chunk<FP8>(o, i * EW_THREADS + tid, kb, rb, p.row_chunks, p.vals, meta_s, p.dense);
    }
    if (MODE != 0) {
        __syncthreads();
    } else if (!__syncthreads_and(plain)) {
        project_any_values<FP8>(p.W, kb, rb, p.row_chunks, p.beta, p.wscale, p.vals, meta_s, p.dense);
        __syncthreads();
    }
    if (tid < 32) {
        const size_t atom = static_cast<size_t>(rb >> 2) * (p.row_chunks / 16) + kb;
        reinterpret_cast<uint4 *>(p.meta + atom * 2048 + 512 * (rb & 3))[tid] = reinterpret_cast<const uint4 *>(meta_s)[tid];
    }
}

// One CTA: one tile.  Small tiles keep even the 2.4 M-element GPT-2 weights spread over several CTAs per SM.
template <bool FP8, int MODE>
__global__ void __launch_bounds__(EW_THREADS)
project_compress_kernel(const uint4 *__restrict__ W, int I, const float *__restrict__ beta_dev,
                        const float *__restrict__ w_amax_dev, float gamma, void *__restrict__ vals,
                        uint8_t *__restrict__ meta, void *__restrict__ dense)
{
    __shared__ __align__(16) uint8_t meta_s[512];
    __shared__ uint2 lut[PROJECT_ENTRIES];
    const int tid = threadIdx.x;
    const int kb = blockIdx.x, rb = blockIdx.y;
    sste_pdl_trigger();
    if (MODE == 0) {
        if (tid < PROJECT_ENTRIES) lut[tid] = project_table_dev.e[tid];
        __syncthreads();                         // the table is in place
    }
    sste_pdl_wait(W, beta_dev, w_amax_dev);
    const size_t row_chunks = static_cast<size_t>(I) / 8;
    const ProjectOut p{W, row_chunks, *beta_dev, FP8 ? sste_scale_from_amax(*w_amax_dev, 448.0f) : 1.0f, gamma, vals, meta, dense};
    uint4 in[PC_CHUNKS];
#pragma unroll
    for (int i = 0; i < PC_CHUNKS; ++i) in[i] = sste_ld_once(project_src(W, row_chunks, kb, rb, i * EW_THREADS + tid));
    project_tile<FP8, MODE>(in, kb, rb, p, meta_s, lut);
}

// ---------------------------------------------------------------- beta

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// fp64 sums of <w, s> and <s, s>, s = S_soft(w) in exact arithmetic; per-block partials are
// combined by the last block in a fixed order.
// L1 = false: beta = <w, S_soft(w)> / ||S_soft(w)||^2 (Eq. 5); L1 = true: ||w||_1 / ||S_soft(w)||_1 (Sec. 4.2,
// the rescaling the method replaces).
template <bool L1>
__global__ void __launch_bounds__(EW_THREADS)
beta_kernel(const uint4 *__restrict__ W, size_t n_chunks, double *__restrict__ partials,
            unsigned int *__restrict__ counter, float *__restrict__ beta_dev, unsigned int *__restrict__ status)
{
    __shared__ double red[2][EW_THREADS / 32];
    __shared__ bool is_last;
    sste_pdl_trigger();
    sste_pdl_wait(W);
    double num = 0.0, den = 0.0;
    for (size_t c = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; c < n_chunks;
         c += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        const uint4 v = sste_ld_once(W + c);
        const uint32_t raw[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const uint32_t bits[4] = {raw[2 * g] & 0xffffu, raw[2 * g] >> 16, raw[2 * g + 1] & 0xffffu,
                                      raw[2 * g + 1] >> 16};
            double a[4], m[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = static_cast<double>(sste_bf16_bits_to_f32(bits[i]));
                m[i] = fabs(a[i]);
            }
            const double lo1 = fmin(m[0], m[1]), hi1 = fmax(m[0], m[1]);
            const double lo2 = fmin(m[2], m[3]), hi2 = fmax(m[2], m[3]);
            const double t = fmin(fmax(lo1, lo2), fmin(hi1, hi2));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double d = m[i] - t;
                if (L1) {
                    num += m[i];
                    if (d > 0.0) den += d;
                } else if (d > 0.0) {
                    const double s = copysign(d, a[i]);
                    num += a[i] * s;
                    den += s * s;
                }
            }
        }
    }
    num = warp_sum(num);
    den = warp_sum(den);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { red[0][warp] = num; red[1][warp] = den; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double bn = 0.0, bd = 0.0;
        for (int w = 0; w < EW_THREADS / 32; ++w) { bn += red[0][w]; bd += red[1][w]; }
        partials[2 * blockIdx.x] = bn;
        partials[2 * blockIdx.x + 1] = bd;
        __threadfence();
        const unsigned int ticket = atomicAdd(counter, 1u);
        is_last = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (is_last && threadIdx.x < 32) {
        __threadfence();
        double tn = 0.0, td = 0.0;
        for (unsigned int b = threadIdx.x; b < gridDim.x; b += 32) {
            tn += __ldcg(partials + 2 * b);
            td += __ldcg(partials + 2 * b + 1);
        }
        tn = warp_sum(tn);
        td = warp_sum(td);
        if (threadIdx.x == 0) {
            if (td == 0.0) {
                *beta_dev = 1.0f;
                atomicCAS(status, 0u, static_cast<unsigned int>(SSTE_ERR_DEGENERATE));
            } else {
                *beta_dev = static_cast<float>(tn / td);
            }
            *counter = 0u;
        }
    }
}

// ---------------------------------------------------------------- Philox4x32-10

__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                              uint32_t k1, uint32_t out[4])
{
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * c0;   // one wide multiply gives both halves
        const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * c2;
        const uint32_t n0 = static_cast<uint32_t>(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n2 = static_cast<uint32_t>(p0 >> 32) ^ c3 ^ k1;
        c0 = n0; c1 = static_cast<uint32_t>(p1); c2 = n2; c3 = static_cast<uint32_t>(p0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// ---------------------------------------------------------------- MVUE of two groups

// What a group's draw comes to, by table: the kept positions q0 < q1 and how to pick their bits.
//   x: byte-permute selector over (a0 a1 | a2 a3) for the two kept elements | (q0 | q1 << 2) << 16
//      (bf16: both halfwords; FP8: the two upper bytes, which carry the signs)
//   y: bf16: which bits of the kept halfwords stay (the rest comes from bf16(h)); FP8: selector of the two result bytes
//      among (e5m2(h), e5m2(max)) | mask of the sign bits to keep << 16
// Entry number: 8 * set + pattern.  Sets 0 to 3: unclipped (alike), set 7 - x: clipped at position x.  Pattern: which sums
// lie above a point, 3 [c0 > p] + 2 [c1 > p] + [c1 > q] + [c2 > q] for the points p <= q and the cumulative sums c0 <= c1 <= c2,
// different for each of the eight cases that can be.  (Unclipped, whether c0 lies above q does not matter: the second kept
// position is above the first.  Clipped, both points are one.)  A clipped group without another nonzero element comes out as
// [c0 > p] = [c1 > p] = 1, [c1 > q] = [c2 > q] = 0, which no single point does.
constexpr int MVUE_ENTRIES = 64;
struct MvueTable { uint2 e[MVUE_ENTRIES]; };
constexpr uint2 mvue_entry(bool FP8, int n)
{
    const int pattern = n % 8, set = n / 8, x = set < 4 ? -1 : 7 - set;      // x: the kept position that keeps its own value
    const int above_p = pattern < 2 ? 0 : pattern < 5 ? 1 : 2;
    const int above_q = pattern == 4 || pattern == 7 ? 2 : pattern == 1 || pattern == 3 || pattern == 6 ? 1 : 0;
    const int a = 2 - above_p, b = 2 - above_q;
    int q0 = 0, q1 = 0;
    bool zero = false;             // the other kept value is +0
    if (x < 0) {
        q0 = a;
        q1 = 1 + (a > b ? a : b);
    } else {
        zero = a == 0 && b == 2;
        const int j = zero ? (x == 0 ? 1 : 0) : a == 2 ? 1 + b : a;
        q0 = x < j ? x : j;
        q1 = x < j ? j : x;
    }
    uint2 e{0, 0};
    const uint32_t nib = static_cast<uint32_t>(q0 | (q1 << 2)) << 16;
    if (FP8) {
        e.x = static_cast<uint32_t>((2 * q0 + 1) | ((2 * q1 + 1) << 4)) | nib;
        const uint32_t s0 = (zero && q0 != x) ? 0u : 0x80u, s1 = (zero && q1 != x) ? 0u : 0x8000u;
        e.y = (q0 == x ? 0x01u : 0u) | (q1 == x ? 0x10u : 0u) | ((s0 | s1) << 16);
    } else {
        e.x = 0x1010u + 0x22u * q0 + 0x2200u * q1 + nib;
        const uint32_t s0 = q0 == x ? 0xffffu : zero ? 0u : 0x8000u, s1 = q1 == x ? 0xffffu : zero ? 0u : 0x8000u;
        e.y = s0 | (s1 << 16);
    }
    return e;
}
constexpr MvueTable mvue_table(bool FP8)
{
    MvueTable t{};
    for (int n = 0; n < MVUE_ENTRIES; ++n) t.e[n] = mvue_entry(FP8, n);
    return t;
}
__device__ const MvueTable mvue_table_bf16 = mvue_table(false), mvue_table_fp8 = mvue_table(true);

struct MvuePair {
    uint2 e0, e1;     // table entries of the two groups
    f32x2 h;          // magnitude of a kept value other than a clipped maximum
    uint32_t mx;      // largest magnitudes, packed bf16; from MVUE_HUGE on the rest may not hold (mvue_group does)
};
// bf16 bits of 2^126: four smaller magnitudes have a finite sum, and neither infinities nor NaNs are smaller
constexpr uint32_t MVUE_HUGE = 0x7e80u;

// Inclusion probabilities p_i = min(1, c |a_i|) with sum 2, kept values a_i / p_i, systematic sampling
// with one uniform u.  With x the first largest magnitude and rest the sum of the others:
//   clipped   (m_x >= rest): x is kept as is; one other element j, chosen with probability m_j / rest
//                            by the point u*rest on the others' cumulative sums (kept below rest), carries
//                            sign(a_j)*rest;
//   unclipped (m_x <  rest): the points u*S/2 and u*S/2 + S/2 on the cumulative sums pick two elements,
//                            both carry sign(a_j)*S/2.
// Two groups at a time: w[i] holds token i's bf16 values of the columns in its halves.  The kernel is bound by instruction
// issue, the half-rate pipe of integer, compare, select and convert instructions first, so the rule is written for that: the
// maximum is found and left out by masks on packed pairs, a sum takes its bf16 terms as they are (one instruction on the FMA pipe,
// no conversion in front), comparisons with the points are integer differences whose sign bytes a dot product turns into the
// byte offset of the table entry that holds the kept pair.  (minus_one is -1 in a way the compiler does not see: multiply-adds with
// it leave the busy pipe to the others.)  No branches; every fp32 step is a single rounded operation in the oracle's order.
__device__ __forceinline__ MvuePair mvue_pair(const uint32_t (&w)[4], uint32_t k_lo, uint32_t k_hi, int minus_one, const uint8_t *lut)
{
    uint32_t m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = w[i] & 0x7fff7fffu;
    const uint32_t mx = __vmaxu2(__vimax3_u16x2(m[0], m[1], m[2]), m[3]);
    // equal to the maximum; z: the magnitudes without the first that is
    const uint32_t e0 = bf_eq2(m[0], mx), e1 = bf_eq2(m[1], mx), e2 = bf_eq2(m[2], mx), e01 = e0 | e1;
    const uint32_t z[4] = {m[0] & ~e0, m[1] & ~(e1 & ~e0), m[2] & ~(e2 & ~e01), m[3] & (e01 | e2)};
    const float rest0 = mix_add<0>(z[3], mix_add<0>(z[2], mix_add<0>(z[1], mix_add<0>(z[0], 0.0f))));
    const float rest1 = mix_add<1>(z[3], mix_add<1>(z[2], mix_add<1>(z[1], mix_add<1>(z[0], 0.0f))));
    // rest above the maximum: nothing is clipped
    const float t0 = mix_add<0>(mx, -rest0), t1 = mix_add<1>(mx, -rest1);
    const uint32_t open = prmt(__float_as_uint(t0), __float_as_uint(t1), 0xffbb), open1 = open & 0x3f803f80u;
    // cumulative sums the points fall into: clipped without the maximum, otherwise with it
    uint32_t v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = z[i] | (m[i] & open);
    const float c00 = mix_add<0>(v[0], 0.0f), c01 = mix_add<1>(v[0], 0.0f);
    const float c10 = mix_add<0>(v[1], c00), c11 = mix_add<1>(v[1], c01);
    const float c20 = mix_add<0>(v[2], c10), c21 = mix_add<1>(v[2], c11);
    const f32x2 total = pack2(mix_add<0>(v[3], c20), mix_add<1>(v[3], c21));
    const f32x2 open2 = pack2(mix_add<0>(open1, 0.0f), mix_add<1>(open1, 0.0f));      // 1 where not clipped
    const f32x2 h = mul2(total, fma2(open2, both(-0.5f), both(1.0f)));                // rest, or half of the sum
    // k is the uniform's 24 bits in the upper bits of a word: k * 2^-32 is exact
    const f32x2 u = mul2(pack2(__uint2float_rn(k_lo & 0xffffff00u), __uint2float_rn(k_hi & 0xffffff00u)), both(0x1p-32f));
    // Clipped: a point that rounding put AT rest (possible only when u * rest is subnormal) counts as just below it,
    // which selects the last other element of nonzero magnitude: minimum of the bit patterns with rest's minus one.
    // rest == 0 gives the first point the pattern -1, below every sum, and the second a NaN's (0x7fffffff), above every sum.
    // Not clipped: the bound is out of reach.
    float b0, b1, r0, r1, q0, q1;
    unpack2(fma2(open2, both(3.402823466e38f), h), b0, b1);
    unpack2(mul2(u, h), r0, r1);
    const int p0 = __viaddmin_s32(__float_as_int(b0), -1, __float_as_int(r0));
    const int p1 = __viaddmin_s32(__float_as_int(b1), -1, __float_as_int(r1));
    unpack2(fma2(h, open2, pack2(__int_as_float(p0), __int_as_float(p1))), q0, q1);
    // per half: 3 - x, less 4 where not clipped
    const uint32_t code = (e01 & 0x00020002u) | ((e0 | (e2 & ~e1)) & ~0x00020002u);
    const uint32_t set = (code & 0x00030003u) | (open & ~0x00030003u);
    // sign bytes of (point - sum), -1 where the sum is above, times -24, -16, -8, -8
    auto offset = [&](uint32_t set_weight, int p, int q, int c0, int c1, int c2) -> uint32_t {
        auto minus = [&](int x, int y) {
            uint32_t r;
            asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(y), "r"(minus_one), "r"(x));
            return r;
        };
        const uint32_t a = prmt(minus(p, c0), minus(p, c1), 0x00fb), b = prmt(minus(q, c1), minus(q, c2), 0x00fb);
        return static_cast<uint32_t>(__dp4a(static_cast<int>(b), 0x0000f8f8, __dp4a(static_cast<int>(a), 0x0000f0e8, __dp4a(static_cast<int>(set), static_cast<int>(set_weight), 256))));
    };
    static_assert(sizeof(uint2) * 8 == 64, "bytes of a set: the weight of a set's number");
    const uint32_t o0 = offset(0x00000040u, p0, __float_as_int(q0), __float_as_int(c00), __float_as_int(c10), __float_as_int(c20));
    const uint32_t o1 = offset(0x00400000u, p1, __float_as_int(q1), __float_as_int(c01), __float_as_int(c11), __float_as_int(c21));
    MvuePair g;
    g.e0 = *reinterpret_cast<const uint2 *>(lut + o0);
    g.e1 = *reinterpret_cast<const uint2 *>(lut + o1);
    g.h = h;
    g.mx = mx;
    return g;
}

// a <= b as an integer mask (all ones / zero)
__device__ __forceinline__ int fset_le(float a, float b)
{
    int r;
    asm("set.le.s32.f32 %0, %1, %2;" : "=r"(r) : "f"(a), "f"(b));
    return r;
}

// The same rule for one group of any values, by selections: p01 = a0 | a1 << 16, p23 = a2 | a3 << 16 (bf16), u the uniform.
// Sums may overflow; comparisons with a NaN are false, and a NaN is never the maximum.
struct MvueGroup {
    uint32_t q0, q1;  // kept positions q0 < q1
    float v0, v1;     // their values before the cast
};
__device__ __forceinline__ MvueGroup mvue_group(uint32_t p01, uint32_t p23, float u)
{
    const float m0 = fabsf(__uint_as_float(p01 << 16)), m1 = fabsf(__uint_as_float(p01 & 0xffff0000u));
    const float m2 = fabsf(__uint_as_float(p23 << 16)), m3 = fabsf(__uint_as_float(p23 & 0xffff0000u));
    const float mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
    const bool e0 = (m0 == mx), e1 = !e0 && (m1 == mx), e2 = !e0 && !e1 && (m2 == mx), e3 = !e0 && !e1 && !e2;
    const uint32_t xi = e0 ? 0u : e1 ? 1u : e2 ? 2u : 3u;
    // cumulative sums without the maximum and with it
    const float z0 = e0 ? 0.0f : m0, z1 = __fadd_rn(z0, e1 ? 0.0f : m1), z2 = __fadd_rn(z1, e2 ? 0.0f : m2);
    const float rest = __fadd_rn(z2, e3 ? 0.0f : m3);
    const float s1 = __fadd_rn(m0, m1), s2 = __fadd_rn(s1, m2), s3 = __fadd_rn(s2, m3);
    const bool clipped = (mx >= rest);
    const float h = clipped ? rest : __fmul_rn(0.5f, s3);
    const float c0 = clipped ? z0 : m0, c1 = clipped ? z1 : s1, c2 = clipped ? z2 : s2;
    const float r1 = __fmul_rn(u, h), r2 = __fadd_rn(r1, h);
    // (a point AT rest counts as just below it; rest == 0 makes the bound a NaN, which fminf passes over)
    const float r1c = clipped ? fminf(r1, __uint_as_float(__float_as_uint(rest) - 1u)) : r1;
    const int j1 = -(fset_le(c0, r1c) + fset_le(c1, r1c) + fset_le(c2, r1c));
    const int n2 = -(fset_le(c0, r2) + fset_le(c1, r2) + fset_le(c2, r2));
    const uint32_t ia = static_cast<uint32_t>(!clipped ? min(j1, 2) : rest == 0.0f ? (e0 ? 1 : 0) : j1);
    const uint32_t ib = clipped ? xi : static_cast<uint32_t>(min(max(j1 + 1, n2), 3));
    // bf16 bits of a_ia and a_ib in the upper half (lower half: don't care)
    const uint32_t sa = __byte_perm(p01, p23, ia * 0x2200u + 0x1000u), sb = __byte_perm(p01, p23, ib * 0x2200u + 0x1000u);
    const uint32_t hb = __float_as_uint(h), sgn = (hb == 0u) ? 0u : 0x80000000u;
    const float va = __uint_as_float((sa & sgn) | hb);
    const float vb = __uint_as_float(clipped ? (sb & 0xffff0000u) : ((sb & sgn) | hb));
    const bool swap = ia > ib;
    return MvueGroup{min(ia, ib), max(ia, ib), swap ? vb : va, swap ? va : vb};
}

// Word (bf16) / halfword (FP8) in shared memory of column jl's results for token group tgl of G: the lanes of a store spread over
// the banks, and sixteen bytes of a column stay together.
template <bool FP8, int G>
__device__ __forceinline__ int mvue_slot(int jl, int tgl)
{
    const int jc = jl >> 3;
    if (G == 32) return jl * 32 + (tgl ^ (FP8 ? 8 * (jc & 3) : 4 * (jc & 7)));
    return FP8 ? jl * 16 + (tgl ^ (8 * (jc & 1))) : (jl ^ (jc >> 2)) * 16 + (tgl ^ (4 * (jc & 3)));
}

// Metadata bytes of a thread's eight columns (nibs: a nibble per column).  Two token groups share a byte (lanes that differ in bit
// 3) and the byte behind it belongs to the next two (bit 4): the four lanes exchange, and each writes two columns' two bytes.
template <bool FP8>
__device__ __forceinline__ void mvue_put_meta(uint32_t nibs, int jc, int tgl, uint8_t *meta_s)
{
    const bool odd = tgl & 1, upper = tgl & 2;
    const uint32_t other = __shfl_xor_sync(0xffffffffu, nibs, 8);
    const uint32_t lo = odd ? other : nibs, hi = odd ? nibs : other;       // of the even token group, of the odd one
    // bytes of the even columns (low nibbles of each byte of nibs) in the lane of the even group, of the odd ones in the other
    const uint32_t v = odd ? ((lo >> 4) & 0x0f0f0f0fu) | (hi & 0xf0f0f0f0u) : (lo & 0x0f0f0f0fu) | ((hi << 4) & 0xf0f0f0f0u);
    const uint32_t w = __shfl_xor_sync(0xffffffffu, v, 16);
    const uint32_t two = prmt(v, w, upper ? 0x3726u : 0x5140u);            // columns 0, 1 of the four or 2, 3: (first byte, second byte)
    const uint32_t k = 4u * (tgl & ~3), jl = jc * 8 + (upper ? 4 : 0) + (odd ? 1 : 0);
    *reinterpret_cast<uint16_t *>(meta_s + (FP8 ? sste_meta_atom_byte8(jl, k) : sste_meta_atom_byte16(jl, k))) = static_cast<uint16_t>(two);
    *reinterpret_cast<uint16_t *>(meta_s + (FP8 ? sste_meta_atom_byte8(jl + 2, k) : sste_meta_atom_byte16(jl + 2, k))) = static_cast<uint16_t>(two >> 16);
}

// A block's groups by that rule (mvue_kernel's rare path; all threads): rows of dY or of its padded copy from `src` on, group
// g0 + e of the thread uses word (g0 + e) & 3 of Philox block (g0 + e) >> 2.
template <bool FP8, int G>
__device__ __noinline__ void mvue_any_values(const uint4 *src, size_t row_chunks, uint64_t g0, uint32_t tensor_id, uint32_t step,
                                             uint32_t key0, uint32_t key1, float gscale, uint32_t *vals_s, uint8_t *meta_s,
                                             uint2 *dense_q)
{
    const int lane = threadIdx.x & 31, jc = lane & 7, tgl = (threadIdx.x >> 5) * 4 + (lane >> 3);
    uint32_t nibs = 0, rnd[4];
#pragma unroll 1
    for (int e = 0; e < 8; ++e) {
        const uint64_t g = g0 + e;
        philox4x32_10(static_cast<uint32_t>(g >> 2), static_cast<uint32_t>(g >> 34), tensor_id, step, key0, key1, rnd);
        const uint32_t r01 = (g & 1u) ? rnd[1] : rnd[0], r23 = (g & 1u) ? rnd[3] : rnd[2], k = (g & 2u) ? r23 : r01;
        uint32_t a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = reinterpret_cast<const uint16_t *>(src + i * row_chunks)[e];
        const MvueGroup r = mvue_group(a[0] | (a[1] << 16), a[2] | (a[3] << 16), __uint2float_rn(k >> 8) * 0x1p-24f);
        nibs |= (r.q0 | (r.q1 << 2)) << (4 * e);
        if (FP8) {
            reinterpret_cast<uint16_t *>(vals_s)[mvue_slot<true, G>(jc * 8 + e, tgl)] = static_cast<uint16_t>(__nv_cvt_float2_to_fp8x2(
                make_float2(__fmul_rn(r.v0, gscale), __fmul_rn(r.v1, gscale)), __NV_SATFINITE, __NV_E5M2));
            if (dense_q) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    reinterpret_cast<uint8_t *>(dense_q + i * row_chunks)[e] =
                        static_cast<uint8_t>(sste_f32_to_e5m2(__fmul_rn(sste_bf16_bits_to_f32(a[i]), gscale)));
            }
        } else {
            const __nv_bfloat162 pair = __floats2bfloat162_rn(r.v0, r.v1);
            vals_s[mvue_slot<false, G>(jc * 8 + e, tgl)] = *reinterpret_cast<const uint32_t *>(&pair);
        }
    }
    mvue_put_meta<FP8>(nibs, jc, tgl, meta_s);
}

// The group rule on explicit inputs (test / debug): group i = four bf16 values a[4 i .. 4 i + 3] and the uniform
// u[i] = k[i] * 2^-24; out: kept positions (q0 | q1 << 2) and the two fp32 values before the cast.
__global__ void __launch_bounds__(EW_THREADS)
mvue_groups_kernel(const uint2 *__restrict__ a, const uint32_t *__restrict__ k24, size_t n, uint32_t *__restrict__ pos,
                   float2 *__restrict__ val)
{
    __shared__ uint2 lut[MVUE_ENTRIES];
    if (threadIdx.x < MVUE_ENTRIES) lut[threadIdx.x] = mvue_table_bf16.e[threadIdx.x];
    __syncthreads();
    sste_pdl_trigger();
    sste_pdl_wait(a, k24);
    for (size_t i = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; i < n;
         i += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        const uint2 g = a[i];
        const uint32_t k = k24[i] << 8;
        // the group in the low halves, its mirror image (an unrelated group) in the high ones
        const uint32_t w[4] = {__byte_perm(g.x, g.y, 0x7610), __byte_perm(g.x, g.y, 0x5432), __byte_perm(g.y, g.x, 0x7610),
                               __byte_perm(g.y, g.x, 0x5432)};
        const MvuePair r = mvue_pair(w, k, ~k, -static_cast<int>(gridDim.z), reinterpret_cast<const uint8_t *>(lut));
        float h, other;
        unpack2(r.h, h, other);
        if ((r.mx & 0xffffu) >= MVUE_HUGE) {
            const MvueGroup any = mvue_group(g.x, g.y, __uint2float_rn(k >> 8) * 0x1p-24f);
            pos[i] = any.q0 | (any.q1 << 2);
            val[i] = make_float2(any.v0, any.v1);
            continue;
        }
        const uint32_t kept = prmt(g.x, g.y, r.e0.x), mask = r.e0.y;
        pos[i] = (r.e0.x >> 16) & 0xfu;
        auto value = [&](uint32_t bits, uint32_t m) {      // bf16 bits of the kept element, its mask
            return m == 0xffffu ? __uint_as_float(bits << 16) : __uint_as_float(((bits & m) << 16) | __float_as_uint(h));
        };
        val[i] = make_float2(value(kept & 0xffffu, mask & 0xffffu), value(kept >> 16, mask >> 16));
    }
}

// ---------------------------------------------------------------- rows of any length, eight elements at a time

// Eight elements from element offset `first` (may be anything) of the array [begin, end) of elements counted from the
// 16-byte aligned address `base`; the caller has checked begin <= first, first + 8 <= end.
__device__ __forceinline__ bool load8_fits(size_t first, size_t begin, size_t end)
{
    // the aligned vectors touched lie inside the array
    return (first & ~static_cast<size_t>(7)) >= begin && ((first + 7) | 7) < end;
}
// the eight elements from element `sh` of the two consecutive vectors a, b on
__device__ __forceinline__ uint4 shift8(const uint4 &a, const uint4 &b, uint32_t sh)
{
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t u[6], t[5], o[4];
#pragma unroll
    for (int k = 0; k < 6; ++k) u[k] = (sh & 4u) ? w[k + 2] : w[k];
#pragma unroll
    for (int k = 0; k < 5; ++k) t[k] = (sh & 2u) ? u[k + 1] : u[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = __funnelshift_r(t[k], t[k + 1], 16u * (sh & 1u));
    return make_uint4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ uint4 load8(const uint4 *__restrict__ base, size_t first)
{
    const uint4 a = sste_ld(base + (first >> 3));
    const uint32_t sh = static_cast<uint32_t>(first) & 7u;
    return sh == 0 ? a : shift8(a, sste_ld(base + (first >> 3) + 1), sh);
}

// A [rows, cols] array of 2-byte elements whose rows may start anywhere, seen as the top-left corner of a larger one of zeros.
struct RaggedRows {
    const uint16_t *src;
    uint32_t rows, cols;
    // elements [c0, c0 + 8) of row r; c0 a multiple of 8
    __device__ __forceinline__ uint4 load(uint32_t r, uint32_t c0) const
    {
        if (r >= rows || c0 >= cols) return make_uint4(0u, 0u, 0u, 0u);
        const size_t lead = (reinterpret_cast<uintptr_t>(src) & 15u) / 2;       // src starts `lead` elements into its vector
        const size_t first = lead + static_cast<size_t>(r) * cols + c0, end = lead + static_cast<size_t>(rows) * cols;
        if (c0 + 8 <= cols && load8_fits(first, lead, end)) return load8(reinterpret_cast<const uint4 *>(src - lead), first);
        uint32_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = (c0 + i < cols) ? sste_ld(src + static_cast<size_t>(r) * cols + c0 + i) : 0u;
        return make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16), e[6] | (e[7] << 16));
    }
    // the same of four consecutive rows; all their loads are under way before the first is used
    __device__ __forceinline__ void load4(uint32_t r, uint32_t c0, uint4 (&out)[4]) const
    {
        const size_t lead = (reinterpret_cast<uintptr_t>(src) & 15u) / 2;
        const size_t first = lead + static_cast<size_t>(r) * cols + c0;
        if (r + 3 < rows && c0 + 8 <= cols && (first & ~static_cast<size_t>(7)) >= lead &&
            first + 3u * static_cast<size_t>(cols) + 16 <= lead + static_cast<size_t>(rows) * cols) {
            const uint4 *base = reinterpret_cast<const uint4 *>(src - lead);
            uint4 a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint4 *v = base + ((first + static_cast<size_t>(i) * cols) >> 3);
                a[i] = sste_ld(v);
                b[i] = sste_ld(v + 1);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] = shift8(a[i], b[i], static_cast<uint32_t>(first + static_cast<size_t>(i) * cols) & 7u);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] = load(r + i, c0);
        }
    }
};

// ---------------------------------------------------------------- MVUE + compress (transposing)

// One CTA: 4 G tokens x 64 output columns of dY.  A thread handles 4 tokens x 8 columns (8 groups, two Philox calls); results
// are transposed through shared memory so that every output row (= column of dY) receives whole lines (G = 32, 256 threads) or halves
// of them, the other half coming from the neighbouring CTA (G = 16, 128 threads).  Bound by instruction issue, not by HBM: dY[8192,
// 3072] takes 22.0 us in bf16 (25.9 with the rule by selections), of which the loads and stores alone take 15.6, and 26.2 in FP8 (31.6);
// five blocks per SM 23.4.
// ANY_COUNTER: counter_cols is not a multiple of 4 (a padded, odd column count), so a thread's eight
// consecutive group indices do not start on a Philox block and span three blocks instead of two.
// PADDED: dY is given as ragged rows; the kernel also writes the zero-padded copy that grad_X reads (a padding pass of its
// own took 35 us of reading and writing for 1000 rows of 50257).
template <bool FP8, bool ANY_COUNTER, bool PADDED, int G>
__global__ void __launch_bounds__(8 * G, G == 32 ? 4 : 8)
mvue_kernel(const uint4 *__restrict__ dY, int O, int T, uint32_t key0, uint32_t key1, uint32_t tensor_id,
            uint32_t step, uint64_t tg_offset, uint32_t counter_cols, const AmaxIn g_amax,
            void *__restrict__ gvals,
            uint8_t *__restrict__ gmeta, void *__restrict__ dense_q, const RaggedRows rag_in, uint4 *__restrict__ padded)
{
    // 64 rows of G words (bf16) or halfwords (fp8)
    __shared__ __align__(16) uint32_t vals_s[64 * G / (FP8 ? 2 : 1)];
    __shared__ __align__(16) uint8_t meta_s[1024];
    __shared__ uint2 lut[MVUE_ENTRIES];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // column block (64), token block (4 G)
    const int jb = G == 32 ? blockIdx.x : blockIdx.x >> 1, tb = G == 32 ? blockIdx.y : 2 * blockIdx.y + (blockIdx.x & 1);
    sste_pdl_trigger();
    if (tid < MVUE_ENTRIES) lut[tid] = FP8 ? mvue_table_fp8.e[tid] : mvue_table_bf16.e[tid];
    __syncthreads();                              // the table is in place
    RaggedRows rag = rag_in;
    sste_pdl_wait(dY, rag.src);
    const size_t row_chunks = static_cast<size_t>(O) / 8;
    bool plain = true;                                   // no infinity, NaN or sum that may overflow
    float gscale = 1.0f;
    {
        const int jc = lane & 7;                         // column chunk 0..7
        const int tgl = warp * 4 + (lane >> 3);          // token group 0..31 inside the tile
        const size_t tok0 = static_cast<size_t>(tb) * (4 * G) + 4 * tgl;
        uint4 in[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (!PADDED) in[i] = sste_ld_once(dY + (tok0 + i) * row_chunks + jb * 8 + jc);
        if (PADDED) {
            rag.load4(static_cast<uint32_t>(tok0), jb * 64u + jc * 8u, in);
#pragma unroll
            for (int i = 0; i < 4; ++i) padded[(tok0 + i) * row_chunks + jb * 8 + jc] = in[i];
        }
        // (behind the loads: nothing moves them in front of the store of the maximum)
        if (FP8) {
            gscale = sste_scale_from_amax(amax_take(g_amax, jb == 0 && tb == 0 && tid == 0), 57344.0f);
            plain = gscale < INFINITY;
        }

        const uint64_t g0 = (tg_offset + static_cast<uint64_t>(tb) * G + tgl) * static_cast<uint64_t>(counter_cols) +
                            static_cast<uint64_t>(jb) * 64 + jc * 8;
        const uint64_t q = g0 >> 2;
        uint32_t rnd[8];
        const int minus_one = -static_cast<int>(gridDim.z);
        if (!ANY_COUNTER && !FP8) {
            // drawn while the loads are on their way
#pragma unroll
            for (int c = 0; c < 4; c += 2)
                philox4x32_10(static_cast<uint32_t>(q + c / 2), static_cast<uint32_t>((q + c / 2) >> 32), tensor_id, step,
                              key0, key1, rnd + 2 * c);
#pragma unroll
            for (int i = 0; i < 8; ++i) asm volatile("" : "+r"(rnd[i]));
        }
        if (ANY_COUNTER) {
            uint32_t r12[12];
#pragma unroll
            for (int b = 0; b < 3; ++b)
                philox4x32_10(static_cast<uint32_t>(q + b), static_cast<uint32_t>((q + b) >> 32), tensor_id, step, key0,
                              key1, r12 + 4 * b);
            const uint32_t sh = static_cast<uint32_t>(g0) & 3u;     // group g0 + e uses word (g0 + e) & 3 of block (g0 + e) >> 2
#pragma unroll
            for (int e = 0; e < 8; ++e)
                rnd[e] = sh == 0 ? r12[e] : sh == 1 ? r12[e + 1] : sh == 2 ? r12[e + 2] : r12[e + 3];
        }

        const uint32_t raw[4][4] = {{in[0].x, in[0].y, in[0].z, in[0].w},
                                    {in[1].x, in[1].y, in[1].z, in[1].w},
                                    {in[2].x, in[2].y, in[2].z, in[2].w},
                                    {in[3].x, in[3].y, in[3].z, in[3].w}};
        uint32_t ex[8];                                 // first table word of every group: its nibble in byte 2
        uint32_t largest;
#pragma unroll
        for (int c = 0; c < 4; ++c) {                   // columns 2c, 2c + 1: one word of each token row
            if (!ANY_COUNTER && FP8 && c % 2 == 0)      // drawn when needed: fewer registers live
                philox4x32_10(static_cast<uint32_t>(q + c / 2), static_cast<uint32_t>((q + c / 2) >> 32), tensor_id, step,
                              key0, key1, rnd + 2 * c);
            const uint32_t w[4] = {raw[0][c], raw[1][c], raw[2][c], raw[3][c]};
            const MvuePair g = mvue_pair(w, rnd[2 * c], rnd[2 * c + 1], minus_one, reinterpret_cast<const uint8_t *>(lut));
            ex[2 * c] = g.e0.x;
            ex[2 * c + 1] = g.e1.x;
            largest = c == 0 ? g.mx : __vmaxu2(largest, g.mx);
            float h[2], mx[2];
            unpack2(FP8 ? mul2(g.h, both(gscale)) : g.h, h[0], h[1]);
            if (FP8) unpack2(mul2(pack2(mix_add<0>(g.mx, 0.0f), mix_add<1>(g.mx, 0.0f)), both(gscale)), mx[0], mx[1]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                // the group of column 2c + e: one bf16 from each of the four token rows, packed in pairs
                const uint32_t sel = e ? 0x7632u : 0x5410u;
                const uint32_t p01 = __byte_perm(w[0], w[1], sel), p23 = __byte_perm(w[2], w[3], sel);
                const uint2 t = e ? g.e1 : g.e0;
                const uint32_t kept = prmt(p01, p23, t.x);
                const int jl = jc * 8 + 2 * c + e;       // (mvue_slot, written out: through the call the kernel is 4 % slower)
                if (FP8) {
                    const uint32_t q = static_cast<uint32_t>(
                        __nv_cvt_float2_to_fp8x2(make_float2(h[e], mx[e]), __NV_SATFINITE, __NV_E5M2));
                    reinterpret_cast<uint16_t *>(vals_s)[G == 32 ? jl * 32 + (tgl ^ (8 * (jc & 3))) : jl * 16 + (tgl ^ (8 * (jc & 1)))] =
                        static_cast<uint16_t>((kept & (t.y >> 16)) | prmt(q, 0, t.y));
                } else {
                    const __nv_bfloat162 hb2 = __floats2bfloat162_rn(h[e], h[e]);
                    const uint32_t hb = *reinterpret_cast<const uint32_t *>(&hb2);
                    vals_s[G == 32 ? jl * 32 + (tgl ^ (4 * (jc & 7))) : mvue_slot<false, G>(jl, tgl)] = (kept & t.y) | (hb & ~t.y);
                }
            }
        }
        if (FP8 && dense_q) {
            // (x + -0 is x, of either sign)
            const f32x2 g2 = both(gscale);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t d[2];
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    uint32_t q[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t word = raw[i][2 * v + e];
                        float a, b;
                        unpack2(mul2(pack2(mix_add<0>(word, -0.0f), mix_add<1>(word, -0.0f)), g2), a, b);
                        q[e] = static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E5M2));
                    }
                    d[v] = __byte_perm(q[0], q[1], 0x5410);
                }
                reinterpret_cast<uint2 *>(dense_q)[(tok0 + i) * row_chunks + jb * 8 + jc] = make_uint2(d[0], d[1]);
            }
        }
        // nibbles of the even columns in the low halves of the bytes, of the odd ones in the high halves
        const uint32_t ev = __byte_perm(__byte_perm(ex[0], ex[2], 0x0062), __byte_perm(ex[4], ex[6], 0x0062), 0x5410);
        const uint32_t od = __byte_perm(__byte_perm(ex[1], ex[3], 0x0062), __byte_perm(ex[5], ex[7], 0x0062), 0x5410);
        mvue_put_meta<FP8>(ev | (od << 4), jc, tgl, meta_s);
        plain = plain && max(largest & 0xffffu, largest >> 16) < MVUE_HUGE;
    }
    // A group of this block with huge or other values (or, FP8, a scale that is not finite): all of them again, by the rule for any values.
    if (!__syncthreads_and(plain)) {
        const size_t at = (static_cast<size_t>(tb) * (4 * G) + warp * 16 + (lane >> 3) * 4) * row_chunks + jb * 8 + (lane & 7);
        mvue_any_values<FP8, G>((PADDED ? padded : dY) + at, row_chunks,
                             (tg_offset + static_cast<uint64_t>(tb) * G + warp * 4 + (lane >> 3)) * static_cast<uint64_t>(counter_cols) +
                                 static_cast<uint64_t>(jb) * 64 + (lane & 7) * 8,
                             tensor_id, step, key0, key1, gscale, vals_s, meta_s,
                             FP8 && dense_q ? reinterpret_cast<uint2 *>(dense_q) + at : nullptr);
        __syncthreads();
    }
    // rows of the transposed tile, in vectors of 16 bytes
    constexpr int VECS = G / (FP8 ? 8 : 4);
    const size_t out_row_vecs = static_cast<size_t>(T) / (FP8 ? 32 : 16);
#pragma unroll
    for (int it = 0; it < 64 * VECS / (8 * G); ++it) {
        const int v = it * 8 * G + tid, row = v / VECS, vec = v % VECS;
        const uint4 data = reinterpret_cast<const uint4 *>(vals_s)[mvue_slot<FP8, G>(row, vec * (FP8 ? 8 : 4)) / (FP8 ? 8 : 4)];
        reinterpret_cast<uint4 *>(gvals)[(static_cast<size_t>(jb) * 64 + row) * out_row_vecs + tb * VECS + vec] = data;
    }
    if (tid < 64) {
        const size_t atom = static_cast<size_t>(jb >> 1) * (T / 128) + (G == 32 ? tb : tb >> 1);
        uint8_t *to = gmeta + atom * 2048 + 1024 * (jb & 1);
        if (G == 32) reinterpret_cast<uint4 *>(to)[tid] = reinterpret_cast<const uint4 *>(meta_s)[tid];
        else reinterpret_cast<uint2 *>(to + 8 * (tb & 1))[2 * tid] = reinterpret_cast<const uint2 *>(meta_s)[2 * tid];      // half of the atom's tokens
    }
}

// ---------------------------------------------------------------- FP8 helpers

// *acc = max(*acc, every thread's `bits`), the bit patterns of non-negative fp32 values, which order like unsigned
// integers.  One atomic per block: with one per warp the 9472 of a full grid queued up at the one address for 9 us,
// whatever the tensor's size (amax of 12.6 MB: 10.3 -> 6.1 us).  True in the thread that did it, false in all others.
__device__ __forceinline__ bool grid_max_to(uint32_t bits, unsigned int *acc)
{
    __shared__ unsigned int best_s[EW_THREADS / 32];
    bits = __reduce_max_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31) == 0) best_s[threadIdx.x >> 5] = bits;
    __syncthreads();
    if (threadIdx.x != 0) return false;
#pragma unroll
    for (int w = 1; w < EW_THREADS / 32; ++w) bits = max(bits, best_s[w]);
    if (bits != 0) atomicMax(acc, bits);
    return true;
}

// running maximum of bf16 magnitude bits (they compare like unsigned integers) in both halves
__device__ __forceinline__ uint32_t max_magnitudes(uint32_t best2, const uint4 &v)
{
    best2 = __vmaxu2(best2, v.x & 0x7fff7fffu);
    best2 = __vmaxu2(best2, v.y & 0x7fff7fffu);
    best2 = __vmaxu2(best2, v.z & 0x7fff7fffu);
    return __vmaxu2(best2, v.w & 0x7fff7fffu);
}

__global__ void __launch_bounds__(EW_THREADS)
amax_kernel(const uint4 *__restrict__ x, size_t n_chunks, unsigned int *__restrict__ acc)
{
    uint32_t best2 = 0;   // magnitude bits of bf16 compare like unsigned integers: running maximum in both halves
    sste_pdl_trigger();
    sste_pdl_wait(x);
    // four independent 16-byte loads per thread and iteration: a pure read needs the bytes in flight
    const size_t stride = static_cast<size_t>(gridDim.x) * EW_THREADS;
    for (size_t c = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; c < n_chunks; c += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (c + j * stride < n_chunks) ? sste_ld_once(x + c + j * stride) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j) best2 = max_magnitudes(best2, v[j]);
    }
    grid_max_to(max(best2 & 0xffffu, best2 >> 16) << 16, acc);
}

// largest |w~| (before rounding) of eight features
__device__ __forceinline__ float max_projected(const uint4 &v, float beta)
{
    const uint32_t raw[4] = {v.x, v.y, v.z, v.w};
    float best = 0.0f;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        // the largest |w~| of a group belongs to its largest |w|: one product per group suffices
        const uint32_t m01 = raw[2 * g] & 0x7fff7fffu, m23 = raw[2 * g + 1] & 0x7fff7fffu;
        const uint32_t lo = __vminu2(m01, m23), hi = __vmaxu2(m01, m23);
        const uint32_t t2 = __vminu2(__vmaxu2(lo, __byte_perm(lo, 0, 0x1032)), __vminu2(hi, __byte_perm(hi, 0, 0x1032)));
        const uint32_t mx = __vmaxu2(hi, __byte_perm(hi, 0, 0x1032));
        const float d = __fsub_rn(__uint_as_float(mx << 16), __uint_as_float(t2 << 16));
        best = fmaxf(best, fabsf(__fmul_rn(d, beta)));
    }
    return best;
}

// amax of the bf16 projection w~ = bf16(beta * S_soft(W)) without writing it: rounding to bf16 is monotone,
// so the maximum of the rounded magnitudes is the rounded maximum of the fp32 ones.
__global__ void __launch_bounds__(EW_THREADS)
project_amax_kernel(const uint4 *__restrict__ W, size_t n_chunks, const float *__restrict__ beta_dev,
                    float *__restrict__ amax_dev, unsigned int *__restrict__ scratch)
{
    sste_pdl_trigger();
    sste_pdl_wait(W, beta_dev);
    const float beta = *beta_dev;
    float best = 0.0f;
    const size_t stride = static_cast<size_t>(gridDim.x) * EW_THREADS;
    for (size_t c = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; c < n_chunks; c += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (c + j * stride < n_chunks) ? sste_ld_once(W + c + j * stride) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j) best = fmaxf(best, max_projected(v[j], beta));
    }
    // scratch NULL: *amax_dev was zeroed by a memset.  Otherwise scratch[0] takes the maximum, scratch[1] counts the blocks,
    // and the last one stores the result and leaves both zero.
    unsigned int *acc = scratch ? scratch : reinterpret_cast<unsigned int *>(amax_dev);
    if (grid_max_to(sste_f32_to_bf16_bits(best) << 16, acc) && scratch) {
        __threadfence();
        if (atomicAdd(scratch + 1, 1u) == gridDim.x - 1) {
            __threadfence();
            *reinterpret_cast<unsigned int *>(amax_dev) = atomicExch(scratch, 0u);
            scratch[1] = 0u;
        }
    }
}

__global__ void fp8_scale_kernel(const float *amax_dev, float fp8_max, float *scale_dev, float *inv_scale_dev)
{
    sste_pdl_trigger();
    sste_pdl_wait(amax_dev);
    const float a = *amax_dev;
    const float s = sste_scale_from_amax(a, fp8_max);
    *scale_dev = s;
    if (inv_scale_dev) *inv_scale_dev = __fdiv_rn(1.0f, s);
}

// eight bf16 values to codes
template <bool E5M2>
__device__ __forceinline__ uint2 quantize8(const uint4 &v, float scale)
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t h[4];           // two codes per word: packed conversion of (low half, high half)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = make_float2(__fmul_rn(__uint_as_float(w[i] << 16), scale),
                                     __fmul_rn(__uint_as_float(w[i] & 0xffff0000u), scale));
        h[i] = static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(f, __NV_SATFINITE, E5M2 ? __NV_E5M2 : __NV_E4M3));
    }
    return make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
}

template <bool E5M2>
__global__ void __launch_bounds__(EW_THREADS)
quantize_kernel(const uint4 *__restrict__ x, size_t n_chunks, const AmaxIn amax,
                uint2 *__restrict__ q)
{
    sste_pdl_trigger();
    sste_pdl_wait(x);
    const float scale = sste_scale_from_amax(amax_take(amax, blockIdx.x == 0 && threadIdx.x == 0), E5M2 ? 57344.0f : 448.0f);
    const size_t stride = static_cast<size_t>(gridDim.x) * EW_THREADS;
    for (size_t c = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; c < n_chunks; c += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (c + j * stride < n_chunks) ? sste_ld_once(x + c + j * stride) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (c + j * stride >= n_chunks) break;
            q[c + j * stride] = quantize8<E5M2>(v[j], scale);
        }
    }
}

// ---------------------------------------------------------------- maximum of a tensor, then what is quantised with it, in one launch

// Block b keeps chunk b of the tensor in registers and leaves the chunk's maximum (its bits with the lowest set: bf16
// magnitudes end in zeros) in slot b of the layer's scratch.  Block 0 reads the slots until none is empty and leaves the tensor's maximum in
// one more word, which the others wait for; then each goes on with its chunk.  A word is both value and flag, so reading it needs
// no order: a store, and a load that finds it.  (Weight of 3072 x 768: two launches 8 us, all blocks reading all slots 13, atomics with
// a fence 7.5, this 6.)  A block that has waited for a while reads the slots itself and works out the missing
// chunks (a maximum may be left twice, a code written twice), so no block depends on another one running: the launch needs no
// guarantee that all its blocks run at the same time, which a collective beside it could hold up.  The last block empties the
// words.  That does need an order: a slot may hold somebody else's value by then while its owner's store is still on its way, so a
// block counts itself out behind a fence that follows its stores (put in front of the wait for the result, which takes longer than
// the fence), and the last block empties behind an acquiring load of the count (a fence there would wait for the block's own
// codes: 0.3 to 0.7 us).
constexpr int GM_SLOTS = SSTE_MAX_SLOTS - 2, GM_RESULT = GM_SLOTS, GM_LEFT = GM_SLOTS + 1;
constexpr unsigned long long GM_PATIENCE_NS = 20000ull, GM_LIMIT_NS = 2000000000ull;
__device__ __forceinline__ uint32_t ld_relaxed(const unsigned int *a)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(unsigned int *a, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const unsigned int *a)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
    return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ unsigned long long ns_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
struct GridMaximum {
    unsigned int *slots, *status;
    uint16_t *taken_s;             // chunks that this block worked out besides its own
    uint32_t *word_s;              // two shared words
    unsigned int n_taken;
    unsigned int left;             // (thread 0) blocks that were done before this one
    unsigned int *taken_test;      // test hook: null, or where the chunks are counted that blocks work out besides their own

    // The words are the layer's, so they are usually not in L2 any more: fetched while the previous kernel drains (a prefetch
    // into L2 needs no order with anybody's writes).
    __device__ __forceinline__ void fetch() const
    {
        if (blockIdx.x == 0 && threadIdx.x <= SSTE_MAX_SLOTS / 32)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(slots + min(threadIdx.x * 32u, SSTE_MAX_SLOTS - 1u)));
    }
    // thread 0 (test hook: every other block's own chunk is left to the others)
    __device__ __forceinline__ void put(uint32_t chunk, uint32_t bits)
    {
        if (taken_test && n_taken == 0 && (chunk & 1u)) return;
        st_relaxed(slots + chunk, bits | 1u);
    }
    // The maximum over all slots once they are filled, with the lowest bit set; another(chunk) works out a missing one, after
    // `patience`.
    template <int THREADS, typename F>
    __device__ __forceinline__ uint32_t gather(unsigned long long patience, F another)
    {
        const uint32_t chunks = gridDim.x;
        unsigned long long start = 0;
        uint32_t best;
        for (;;) {
            best = 0;
            uint32_t missing = chunks;
            for (uint32_t i = threadIdx.x; i < chunks; i += THREADS) {
                const uint32_t v = ld_relaxed(slots + i);
                best = max(best, v);
                if (v == 0) missing = min(missing, (i + chunks - blockIdx.x) % chunks);      // the blocks begin at different places
            }
            if (__syncthreads_and(missing == chunks)) break;
            if (threadIdx.x == 0) {
                const unsigned long long now = ns_now();
                if (start == 0) start = now;
                word_s[0] = chunks;
                word_s[1] = now - start > GM_LIMIT_NS ? 2u : now - start >= patience ? 1u : 0u;
            }
            __syncthreads();
            const uint32_t late = word_s[1];
            if (late == 2u) {
                if (threadIdx.x == 0) atomicMax(status, static_cast<unsigned int>(SSTE_ERR_TIMEOUT));
                break;
            }
            if (late == 1u) {
                atomicMin(word_s, missing);
                __syncthreads();
                const uint32_t first = word_s[0];
                if (first < chunks) {
                    const uint32_t chunk = (first + blockIdx.x) % chunks;
                    if (threadIdx.x == 0) taken_s[n_taken] = static_cast<uint16_t>(chunk);
                    ++n_taken;
                    another(chunk);
                }
                __syncthreads();
            }
        }
        best = __reduce_max_sync(0xffffffffu, best);
        if (threadIdx.x == 0) word_s[0] = 1u;
        __syncthreads();
        if ((threadIdx.x & 31) == 0) atomicMax(word_s, best);
        __syncthreads();
        const uint32_t result = word_s[0];
        if (threadIdx.x == 0) {
            st_relaxed(slots + GM_RESULT, result);
            fence_gpu();           // the result, and what was put in place of others, in front of the count
        }
        return result;
    }
    template <int THREADS, typename F>
    __device__ __forceinline__ float wait(F another)
    {
        uint32_t result = 0;
        if (blockIdx.x != 0) {
            if (threadIdx.x == 0) {
                fence_gpu();       // this block's slot, in front of the count
                const unsigned long long start = ns_now();
                do result = ld_relaxed(slots + GM_RESULT);
                while (result == 0 && ns_now() - start < GM_PATIENCE_NS);
                word_s[0] = result;
            }
            __syncthreads();
            result = word_s[0];
            __syncthreads();
        }
        if (result == 0) result = gather<THREADS>(blockIdx.x == 0 ? GM_PATIENCE_NS : 0ull, another);
        if (threadIdx.x == 0) left = atomicAdd(slots + GM_LEFT, 1u);
        return __uint_as_float(result & ~1u);
    }
    // after the block's own work (the count has had the time to come back)
    __device__ __forceinline__ void leave()
    {
        if (taken_test && threadIdx.x == 0) atomicAdd(taken_test, n_taken);
        if (threadIdx.x < 32 && __shfl_sync(0xffffffffu, left, 0) + 1 == gridDim.x) {
            if (threadIdx.x == 0) ld_acquire(slots + GM_LEFT);       // the other blocks' stores, in front of the empty words
            __syncwarp();
            for (uint32_t i = threadIdx.x; i < gridDim.x; i += 32) slots[i] = 0u;
            if (threadIdx.x == 0) slots[GM_RESULT] = slots[GM_LEFT] = 0u;
        }
    }
};

// maximum of `bits` over the block, valid in thread 0
template <int THREADS>
__device__ __forceinline__ uint32_t block_max(uint32_t bits)
{
    __shared__ uint32_t best_s[THREADS / 32];
    bits = __reduce_max_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31) == 0) best_s[threadIdx.x >> 5] = bits;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 1; w < THREADS / 32; ++w) bits = max(bits, best_s[w]);
    }
    return bits;
}

// sste_amax and sste_quantize_fp8 (E4M3): a chunk is AQ_THREADS * V vectors.
constexpr int AQ_THREADS = 512;
template <int V>
__global__ void __launch_bounds__(AQ_THREADS, 2)
amax_quantize_kernel(const uint4 *__restrict__ x, size_t n_vec, float *__restrict__ amax_dev, unsigned int *__restrict__ slots,
                     uint2 *__restrict__ q, unsigned int *__restrict__ status, unsigned int *__restrict__ taken_test)
{
    __shared__ uint16_t taken_s[GM_SLOTS];
    __shared__ uint32_t word_s[2];
    const int tid = threadIdx.x;
    sste_pdl_trigger();
    GridMaximum gm{slots, status, taken_s, word_s, 0, 0, taken_test};
    gm.fetch();
    sste_pdl_wait(x);
    uint4 v[V];
    auto load = [&](uint32_t chunk) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const size_t c = (static_cast<size_t>(chunk) * V + i) * AQ_THREADS + tid;
            v[i] = c < n_vec ? sste_ld_once(x + c) : make_uint4(0, 0, 0, 0);
        }
    };
    auto put_max = [&](uint32_t chunk) {
        uint32_t best2 = 0;
#pragma unroll
        for (int i = 0; i < V; ++i) best2 = max_magnitudes(best2, v[i]);
        const uint32_t best = block_max<AQ_THREADS>(max(best2 & 0xffffu, best2 >> 16) << 16);
        if (tid == 0) gm.put(chunk, best);
    };
    load(blockIdx.x);
    put_max(blockIdx.x);
    const float amax = gm.wait<AQ_THREADS>([&](uint32_t chunk) {
        load(chunk);
        put_max(chunk);
    });
    const float scale = sste_scale_from_amax(amax, 448.0f);
    if (blockIdx.x == 0 && tid == 0) *amax_dev = amax;
    auto quantize = [&](uint32_t chunk) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const size_t c = (static_cast<size_t>(chunk) * V + i) * AQ_THREADS + tid;
            if (c < n_vec) q[c] = quantize8<false>(v[i], scale);
        }
    };
    if (gm.n_taken > 0) load(blockIdx.x);
    quantize(blockIdx.x);
    for (unsigned int k = 0; k < gm.n_taken; ++k) {
        load(taken_s[k]);
        quantize(taken_s[k]);
    }
    gm.leave();
}

// sste_project_amax and sste_project_compress (E4M3): a chunk is R tiles, numbered along the rows of tiles.
template <int R>
__global__ void __launch_bounds__(EW_THREADS, R == 4 ? 3 : 4)
project_fp8_kernel(const uint4 *__restrict__ W, int I, uint32_t tiles, const float *__restrict__ beta_dev,
                   float *__restrict__ amax_dev, unsigned int *__restrict__ slots, void *__restrict__ vals,
                   uint8_t *__restrict__ meta, void *__restrict__ dense, unsigned int *__restrict__ status,
                   unsigned int *__restrict__ taken_test)
{
    __shared__ __align__(16) uint8_t meta_s[512];
    __shared__ uint2 lut[PROJECT_ENTRIES];
    __shared__ uint16_t taken_s[GM_SLOTS];
    __shared__ uint32_t word_s[2];
    const int tid = threadIdx.x;
    const uint32_t across = static_cast<uint32_t>(I) / 128;
    if (tid < PROJECT_ENTRIES) lut[tid] = project_table_dev.e[tid];
    sste_pdl_trigger();
    GridMaximum gm{slots, status, taken_s, word_s, 0, 0, taken_test};
    gm.fetch();
    sste_pdl_wait(W, beta_dev);
    const float beta = *beta_dev;
    const size_t row_chunks = static_cast<size_t>(I) / 8;
    uint4 v[R][PC_CHUNKS];
    auto load = [&](uint32_t chunk) {
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const uint32_t tile = chunk * R + t, rb = tile / across;
#pragma unroll
            for (int i = 0; i < PC_CHUNKS; ++i)
                v[t][i] = tile < tiles ? sste_ld_once(project_src(W, row_chunks, tile - rb * across, rb, i * EW_THREADS + tid)) : make_uint4(0, 0, 0, 0);
        }
    };
    auto put_max = [&](uint32_t chunk) {
        float best = 0.0f;
#pragma unroll
        for (int t = 0; t < R; ++t)
#pragma unroll
            for (int i = 0; i < PC_CHUNKS; ++i) best = fmaxf(best, max_projected(v[t][i], beta));
        const uint32_t bits = block_max<EW_THREADS>(sste_f32_to_bf16_bits(best) << 16);
        if (tid == 0) gm.put(chunk, bits);
    };
    load(blockIdx.x);
    put_max(blockIdx.x);
    const float amax = gm.wait<EW_THREADS>([&](uint32_t chunk) {
        load(chunk);
        put_max(chunk);
    });
    if (blockIdx.x == 0 && tid == 0) *amax_dev = amax;
    const ProjectOut p{W, row_chunks, beta, sste_scale_from_amax(amax, 448.0f), 0.0f, vals, meta, dense};
    auto project = [&](uint32_t chunk) {
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const uint32_t tile = chunk * R + t, rb = tile / across;
            if (tile < tiles) project_tile<true, 0>(v[t], static_cast<int>(tile - rb * across), static_cast<int>(rb), p, meta_s, lut);
            if (t + 1 < R) __syncthreads();      // the metadata has left shared memory
        }
    };
    if (gm.n_taken > 0) load(blockIdx.x);
    project(blockIdx.x);
    for (unsigned int k = 0; k < gm.n_taken; ++k) {
        load(taken_s[k]);
        __syncthreads();
        project(taken_s[k]);
    }
    gm.leave();
}

// ---------------------------------------------------------------- metadata image -> canonical

template <bool EIGHT_BIT>
__global__ void __launch_bounds__(EW_THREADS)
meta_to_canonical_kernel(const uint8_t *__restrict__ meta, int rows, int k, uint16_t *__restrict__ out)
{
    sste_pdl_trigger();
    sste_pdl_wait(meta);
    const size_t words = static_cast<size_t>(rows) * (k / 16);
    for (size_t w = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; w < words;
         w += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        const uint32_t r = static_cast<uint32_t>(w / (k / 16));
        const uint32_t kk = static_cast<uint32_t>(w % (k / 16)) * 16;   // first K index of this word
        const size_t atom = static_cast<size_t>(r >> 7) * (k / 128) + (kk >> 7);
        const uint8_t *base = meta + atom * 2048;
        const uint32_t m = r & 127u, ko = kk & 127u;
        const uint32_t b0 = EIGHT_BIT ? sste_meta_atom_byte8(m, ko) : sste_meta_atom_byte16(m, ko);
        const uint32_t b1 = EIGHT_BIT ? sste_meta_atom_byte8(m, ko + 8) : sste_meta_atom_byte16(m, ko + 8);
        out[w] = static_cast<uint16_t>(base[b0] | (base[b1] << 8));
    }
}

// ---------------------------------------------------------------- compressed operand -> dense (grad_X of a layer without a dense copy)

// One thread per 16 bytes of values: bf16 4 groups (16 dense elements), fp8 8 groups (32 dense elements).
template <bool EIGHT_BIT>
__global__ void __launch_bounds__(EW_THREADS)
decompress_kernel(const uint4 *__restrict__ vals, const uint8_t *__restrict__ meta, int k, size_t n_units,
                  uint4 *__restrict__ dense)
{
    sste_pdl_trigger();
    sste_pdl_wait(vals, meta);
    const uint32_t units_per_row = static_cast<uint32_t>(k) / (EIGHT_BIT ? 32 : 16);
    for (size_t un = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; un < n_units;
         un += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        // (a 64-bit division costs more than the copy; larger weights still take it)
        const uint32_t row = (un >> 32) ? static_cast<uint32_t>(un / units_per_row) : static_cast<uint32_t>(un) / units_per_row;
        const uint32_t kk = static_cast<uint32_t>(un - static_cast<size_t>(row) * units_per_row) * (EIGHT_BIT ? 32u : 16u);
        const uint8_t *atom = meta + (static_cast<size_t>(row >> 7) * (k / 128) + (kk >> 7)) * 2048;
        const uint4 v = sste_ld_once(vals + un);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t o[8];
        if (EIGHT_BIT) {
            const uint32_t codes = *reinterpret_cast<const uint32_t *>(atom + sste_meta_atom_byte8(row & 127u, kk & 127u));
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const uint32_t nib = (codes >> (4 * g)) & 0xfu, p0 = nib & 3u, p1 = nib >> 2;
                const uint32_t pr = (g & 1) ? (w[g >> 1] >> 16) : (w[g >> 1] & 0xffffu);
                o[g] = ((pr & 0xffu) << (8 * p0)) | ((pr >> 8) << (8 * p1));
            }
        } else {
            const uint32_t codes = *reinterpret_cast<const uint16_t *>(atom + sste_meta_atom_byte16(row & 127u, kk & 127u));
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t nib = (codes >> (4 * g)) & 0xfu, p0 = nib & 3u, p1 = nib >> 2;
                const uint64_t d = (static_cast<uint64_t>(w[g] & 0xffffu) << (16 * p0)) |
                                   (static_cast<uint64_t>(w[g] >> 16) << (16 * p1));
                o[2 * g] = static_cast<uint32_t>(d);
                o[2 * g + 1] = static_cast<uint32_t>(d >> 32);
            }
        }
        dense[2 * un] = make_uint4(o[0], o[1], o[2], o[3]);
        dense[2 * un + 1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// ---------------------------------------------------------------- zero padding to multiples of 128 and back

// Rows of an odd number of 2-byte elements start anywhere: both kernels work in 16-byte vectors of the destination and
// assemble each from the two aligned source vectors that hold its eight elements (the second one hits L1), with element
// accesses only where a vector is cut by a row end or an array end.  Element by element, with a 64-bit division for each,
// 1000 rows of 50257 took 50 us to pad and 119 us to crop; now 35 us each (about 6 TB/s).

// dst [rows_p, cols_p] <- src [rows, cols] in the top-left corner, zeros elsewhere; one thread per 8 destination elements.
// INDEX: unsigned type that holds the number of destination vectors (a 64-bit division costs more than the copy).
template <typename INDEX>
__global__ void __launch_bounds__(EW_THREADS)
pad_2d_kernel(const RaggedRows src_in, uint4 *__restrict__ dst, uint32_t vec_per_row, INDEX n_vec)
{
    RaggedRows src = src_in;
    sste_pdl_trigger();
    sste_pdl_wait(src.src);
    for (INDEX v = static_cast<INDEX>(blockIdx.x) * EW_THREADS + threadIdx.x; v < n_vec;
         v += static_cast<INDEX>(gridDim.x) * EW_THREADS) {
        const uint32_t r = static_cast<uint32_t>(v / vec_per_row);
        dst[v] = src.load(r, static_cast<uint32_t>(v - static_cast<INDEX>(r) * vec_per_row) * 8u);
    }
}

// dst [rows, cols] <- top-left corner of src [rows_p, cols_p] (16-byte aligned rows or not); one thread per aligned vector
// of dst, n = rows * cols elements.  Up to two tensors per launch: the blocks from `blocks` on work on the second.
struct CropJob {
    const uint16_t *src;
    size_t src_elements;
    uint16_t *dst;
    uint32_t cols_p, cols;
    size_t n, n_vec;
    uint32_t blocks;
};
template <typename INDEX>
__global__ void __launch_bounds__(EW_THREADS)
crop_2d_kernel(const CropJob job0, const CropJob job1)
{
    sste_pdl_trigger();
    sste_pdl_wait();
    const bool second = blockIdx.x >= job0.blocks;
    const CropJob &job = second ? job1 : job0;
    const uint16_t *src = job.src;
    sste_fresh(src);
    uint16_t *__restrict__ dst = job.dst;
    const uint32_t cols = job.cols, cols_p = job.cols_p, block = blockIdx.x - (second ? job0.blocks : 0u);
    const INDEX n = static_cast<INDEX>(job.n), n_vec = static_cast<INDEX>(job.n_vec);
    const size_t lead = (reinterpret_cast<uintptr_t>(src) & 15u) / 2;
    const uint4 *base = reinterpret_cast<const uint4 *>(src - lead);
    const INDEX dlead = static_cast<INDEX>((reinterpret_cast<uintptr_t>(dst) & 15u) / 2);
    for (INDEX v = static_cast<INDEX>(block) * EW_THREADS + threadIdx.x; v < n_vec;
         v += static_cast<INDEX>(job.blocks) * EW_THREADS) {
        // elements [e0, e1) of dst
        const INDEX e0 = v == 0 ? 0 : v * 8 - dlead, e1 = (v + 1) * 8 - dlead < n ? (v + 1) * 8 - dlead : n;
        INDEX r = e0 / cols;
        uint32_t c = static_cast<uint32_t>(e0 - r * cols);
        const size_t first = lead + static_cast<size_t>(r) * cols_p + c;
        if (e1 - e0 == 8 && c + 8 <= cols && load8_fits(first, lead, lead + job.src_elements)) {
            *reinterpret_cast<uint4 *>(dst + e0) = load8(base, first);
        } else {
            for (INDEX e = e0; e < e1; ++e) {
                dst[e] = sste_ld(src + static_cast<size_t>(r) * cols_p + c);
                if (++c == cols) { c = 0; ++r; }
            }
        }
    }
}

int grid_for(size_t work_items, int sm_count)
{
    size_t blocks = (work_items + EW_THREADS - 1) / EW_THREADS;
    size_t cap = static_cast<size_t>(sm_count) * 8;
    if (cap > SSTE_MAX_REDUCE_BLOCKS) cap = SSTE_MAX_REDUCE_BLOCKS;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

// every entry point of this file launches exactly one kernel
sste_status launch_result()
{
    if (cudaGetLastError() != cudaSuccess) return SSTE_ERR_CUDA;
    sste_count_launches(1);
    return SSTE_OK;
}

// ---------------------------------------------------------------- SR-STE decay term (Sec. 3.2)

// grad_W += lambda * w on the entries the 2:4 mask prunes: the gradient of (lambda / 2) ||w (1 - m_h(w))||^2.
// A thread handles 8 consecutive features of a row (two groups: one metadata byte of the operand image).
template <bool EIGHT_BIT>
__global__ void __launch_bounds__(EW_THREADS)
srste_decay_kernel(const uint4 *__restrict__ W, const uint8_t *__restrict__ meta, int I, size_t n_chunks, float lambda,
                   uint4 *__restrict__ dW)
{
    sste_pdl_trigger();
    sste_pdl_wait(W, meta);
    const size_t row_chunks = static_cast<size_t>(I) / 8;
    for (size_t c = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; c < n_chunks;
         c += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        const uint32_t row = static_cast<uint32_t>(c / row_chunks), k = static_cast<uint32_t>(c % row_chunks) * 8u;
        const size_t atom = static_cast<size_t>(row >> 7) * (I / 128) + (k >> 7);
        const uint32_t byte = sste_ld(meta + atom * 2048 + (EIGHT_BIT ? sste_meta_atom_byte8(row & 127u, k & 127u)
                                                                     : sste_meta_atom_byte16(row & 127u, k & 127u)));
        const uint4 w = sste_ld_once(W + c);
        uint4 g = dW[c];
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
        uint32_t gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int grp = 0; grp < 2; ++grp) {
            const uint32_t nib = (byte >> (4 * grp)) & 0xfu;
            const uint32_t keep = (1u << (nib & 3u)) | (1u << (nib >> 2));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (keep & (1u << e)) continue;
                const int word = 2 * grp + (e >> 1), sh = 16 * (e & 1);
                const float wv = sste_bf16_bits_to_f32((ww[word] >> sh) & 0xffffu);
                const float gv = sste_bf16_bits_to_f32((gw[word] >> sh) & 0xffffu);
                const uint32_t out = sste_f32_to_bf16_bits(__fadd_rn(gv, __fmul_rn(lambda, wv)));
                gw[word] = (gw[word] & ~(0xffffu << sh)) | (out << sh);
            }
        }
        dW[c] = make_uint4(gw[0], gw[1], gw[2], gw[3]);
    }
}

// ---------------------------------------------------------------- flip count (Sec. 3.1, "Flip rate")

// Number of entries in which the 2:4 masks of two operand images differ.  Both images have the same layout,
// so nibbles are compared in place: a nibble p0 | p1 << 2 stands for the mask (1 << p0) | (1 << p1).
__global__ void __launch_bounds__(EW_THREADS)
flip_count_kernel(const uint4 *__restrict__ a, const uint4 *__restrict__ b, size_t n_vec,
                  unsigned long long *__restrict__ count)
{
    sste_pdl_trigger();
    sste_pdl_wait(a, b);
    unsigned int local = 0;
    for (size_t v = static_cast<size_t>(blockIdx.x) * EW_THREADS + threadIdx.x; v < n_vec;
         v += static_cast<size_t>(gridDim.x) * EW_THREADS) {
        const uint4 x = sste_ld_once(a + v), y = sste_ld_once(b + v);
        const uint32_t wx[4] = {x.x, x.y, x.z, x.w}, wy[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (wx[w] == wy[w]) continue;
#pragma unroll
            for (int n = 0; n < 8; ++n) {
                const uint32_t nx = (wx[w] >> (4 * n)) & 0xfu, ny = (wy[w] >> (4 * n)) & 0xfu;
                const uint32_t mx = (1u << (nx & 3u)) | (1u << (nx >> 2)), my = (1u << (ny & 3u)) | (1u << (ny >> 2));
                local += __popc(mx ^ my);
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(count, static_cast<unsigned long long>(local));
}

}  // namespace

// ---------------------------------------------------------------- entry points

namespace {

sste_status beta_launch(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt, float *beta_dev, void *stream, bool l1)
{
    if (!ctx || !W || !beta_dev) return SSTE_ERR_INVALID_ARG;
    if (wdt != SSTE_BF16) return SSTE_ERR_DTYPE;
    if (!sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(W, 128) || !sste_aligned(beta_dev, 4)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_chunks = static_cast<size_t>(O) * I / 8;
    const int grid = grid_for(n_chunks, ctx->sm_count);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (l1)
        sste_launch(beta_kernel<true>, dim3(grid), dim3(EW_THREADS), 0, s, static_cast<const uint4 *>(W), n_chunks,
                    ctx->partials_dev, ctx->counter_dev, beta_dev, ctx->status_dev);
    else
        sste_launch(beta_kernel<false>, dim3(grid), dim3(EW_THREADS), 0, s, static_cast<const uint4 *>(W), n_chunks,
                    ctx->partials_dev, ctx->counter_dev, beta_dev, ctx->status_dev);
    return launch_result();
}

// mode: 0 = the method's projection, 1 = interpolated threshold, 2 = hard thresholding
sste_status project_launch(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt, const float *beta_dev,
                           const float *w_amax_dev, sste_dtype odt, int mode, float gamma, void *vals, void *meta,
                           void *dense_out, void *stream)
{
    if (!ctx || !W || !beta_dev || !vals || !meta) return SSTE_ERR_INVALID_ARG;
    if (wdt != SSTE_BF16 || (odt != SSTE_BF16 && odt != SSTE_E4M3)) return SSTE_ERR_DTYPE;
    if (odt == SSTE_E4M3 && !w_amax_dev) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(W, 128) || !sste_aligned(vals, 128) || !sste_aligned(meta, 128) ||
        !sste_aligned(dense_out, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const dim3 grid(I / 128, O / PC_ROWS);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint4 *w = static_cast<const uint4 *>(W);
    uint8_t *m = static_cast<uint8_t *>(meta);
    const bool f8 = (odt == SSTE_E4M3);
#define SSTE_PC_LAUNCH(F8, MODE)                                                                                   \
    sste_launch(project_compress_kernel<F8, MODE>, dim3(grid), dim3(EW_THREADS), 0, s, w, I, beta_dev,           \
                F8 ? w_amax_dev : nullptr, gamma, vals, m, dense_out)
    if (mode == 0) { if (f8) SSTE_PC_LAUNCH(true, 0); else SSTE_PC_LAUNCH(false, 0); }
    else if (mode == 1) { if (f8) SSTE_PC_LAUNCH(true, 1); else SSTE_PC_LAUNCH(false, 1); }
    else { if (f8) SSTE_PC_LAUNCH(true, 2); else SSTE_PC_LAUNCH(false, 2); }
#undef SSTE_PC_LAUNCH
    return launch_result();
}

}  // namespace

extern "C" sste_status sste_beta_init(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt, float *beta_dev,
                                      void *stream)
{
    return beta_launch(ctx, W, O, I, wdt, beta_dev, stream, false);
}

extern "C" sste_status sste_beta_init_l1(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt, float *beta_dev,
                                         void *stream)
{
    return beta_launch(ctx, W, O, I, wdt, beta_dev, stream, true);
}

extern "C" sste_status sste_project_compress(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt,
                                             const float *beta_dev, const float *w_amax_dev, sste_dtype odt,
                                             void *vals, void *meta, void *dense_out, void *stream)
{
    return project_launch(ctx, W, O, I, wdt, beta_dev, w_amax_dev, odt, 0, 0.0f, vals, meta, dense_out, stream);
}

extern "C" sste_status sste_project_compress_variant(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt,
                                                     const float *beta_dev, const float *w_amax_dev, sste_dtype odt,
                                                     sste_pruning pruning, float gamma, void *vals, void *meta,
                                                     void *dense_out, void *stream)
{
    if (pruning != SSTE_PRUNE_SOFT && pruning != SSTE_PRUNE_HARD) return SSTE_ERR_INVALID_ARG;
    if (!(gamma >= 0.0f && gamma <= 1.0f)) return SSTE_ERR_INVALID_ARG;
    const int mode = (pruning == SSTE_PRUNE_HARD) ? 2 : (gamma == 0.0f ? 0 : 1);
    return project_launch(ctx, W, O, I, wdt, beta_dev, w_amax_dev, odt, mode, gamma, vals, meta, dense_out, stream);
}

extern "C" sste_status sste_srste_decay(sste_ctx *ctx, const void *W, const void *meta, int O, int I,
                                        sste_dtype meta_dt, float lambda, void *dW, void *stream)
{
    if (!ctx || !W || !meta || !dW) return SSTE_ERR_INVALID_ARG;
    if (meta_dt != SSTE_BF16 && meta_dt != SSTE_E4M3 && meta_dt != SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (!sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(W, 16) || !sste_aligned(meta, 16) || !sste_aligned(dW, 16)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_chunks = static_cast<size_t>(O) * I / 8;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (meta_dt == SSTE_BF16)
        sste_launch(srste_decay_kernel<false>, dim3(grid_for(n_chunks, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                    static_cast<const uint4 *>(W), static_cast<const uint8_t *>(meta), I, n_chunks, lambda,
                    static_cast<uint4 *>(dW));
    else
        sste_launch(srste_decay_kernel<true>, dim3(grid_for(n_chunks, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                    static_cast<const uint4 *>(W), static_cast<const uint8_t *>(meta), I, n_chunks, lambda,
                    static_cast<uint4 *>(dW));
    return launch_result();
}

namespace {

sste_status mvue_launch(sste_ctx *ctx, const void *dY, int T, int O, sste_dtype gdt, uint64_t seed, uint32_t tensor_id,
                        uint32_t step, uint64_t token_offset, int counter_cols, const float *g_amax_dev, void *scratch,
                        sste_dtype odt, void *gvals, void *gmeta, void *dense_q_out, void *stream)
{
    if (!ctx || !dY || !gvals || !gmeta) return SSTE_ERR_INVALID_ARG;
    if (gdt != SSTE_BF16 || (odt != SSTE_BF16 && odt != SSTE_E5M2)) return SSTE_ERR_DTYPE;
    if (odt == SSTE_E5M2 && !g_amax_dev) return SSTE_ERR_INVALID_ARG;
    if (counter_cols < 0 || counter_cols > O) return SSTE_ERR_INVALID_ARG;
    const uint32_t ccols = static_cast<uint32_t>(counter_cols == 0 ? O : counter_cols);
    if (odt == SSTE_BF16 && dense_q_out) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(O) || !sste_mult128(T) || (token_offset % 4) != 0) return SSTE_ERR_SHAPE;
    if (!sste_aligned(dY, 128) || !sste_aligned(gvals, 128) || !sste_aligned(gmeta, 128) ||
        !sste_aligned(dense_q_out, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint32_t key0 = static_cast<uint32_t>(seed), key1 = static_cast<uint32_t>(seed >> 32);
    const uint4 *g = static_cast<const uint4 *>(dY);
    uint8_t *gm = static_cast<uint8_t *>(gmeta);
    const uint64_t tg0 = token_offset / 4;
    const bool f8 = (odt == SSTE_E5M2), any = (ccols % 4) != 0;
    const AmaxIn g_amax{const_cast<float *>(g_amax_dev), static_cast<unsigned int *>(scratch)};
    // Small blocks where the large ones would be less than one round of the SMs (512 x 256: 2.6 us with large ones, 2.2 with small
    // ones) and in FP8 (8192 x 3072: 27.7 and 26.9 us; bf16, of which rows are twice as long: 22.7 and 23.5).
    const bool small = static_cast<long long>(O / 64) * (T / 128) <= 4ll * ctx->sm_count;
#define SSTE_MVUE_LAUNCH(F8, ANY, G)                                                                                 \
    sste_launch(mvue_kernel<F8, ANY, false, G>, dim3(O / (G == 32 ? 64 : 32), T / 128), dim3(8 * G), 0, s, g, O, T, key0, key1,         \
                tensor_id, step, tg0, ccols, F8 ? g_amax : AmaxIn{}, gvals, gm, F8 ? dense_q_out : nullptr, RaggedRows{}, nullptr)
    if (f8) { if (any) SSTE_MVUE_LAUNCH(true, true, 16); else SSTE_MVUE_LAUNCH(true, false, 16); }
    else if (small) { if (any) SSTE_MVUE_LAUNCH(false, true, 16); else SSTE_MVUE_LAUNCH(false, false, 16); }
    else { if (any) SSTE_MVUE_LAUNCH(false, true, 32); else SSTE_MVUE_LAUNCH(false, false, 32); }
#undef SSTE_MVUE_LAUNCH
    return launch_result();
}

}  // namespace

extern "C" sste_status sste_mvue_sparsify(sste_ctx *ctx, const void *dY, int T, int O, sste_dtype gdt, uint64_t seed,
                                          uint32_t tensor_id, uint32_t step, uint64_t token_offset, int counter_cols,
                                          const float *g_amax_dev, sste_dtype odt, void *gvals, void *gmeta,
                                          void *dense_q_out, void *stream)
{
    return mvue_launch(ctx, dY, T, O, gdt, seed, tensor_id, step, token_offset, counter_cols, g_amax_dev, nullptr, odt, gvals,
                       gmeta, dense_q_out, stream);
}

sste_status sste_mvue_scratch(sste_ctx *ctx, const void *dY, int T, int O, uint64_t seed, uint32_t tensor_id, uint32_t step,
                              uint64_t token_offset, int counter_cols, float *g_amax_dev, void *scratch, void *gvals,
                              void *gmeta, void *dense_q_out, void *stream)
{
    return mvue_launch(ctx, dY, T, O, SSTE_BF16, seed, tensor_id, step, token_offset, counter_cols, g_amax_dev, scratch, SSTE_E5M2,
                       gvals, gmeta, dense_q_out, stream);
}

sste_status sste_mvue_padded(sste_ctx *ctx, const void *dY, int rows, int cols, void *dYp, int T, int O, uint64_t seed,
                             uint32_t tensor_id, uint32_t step, uint64_t token_offset, int counter_cols, void *gvals,
                             void *gmeta, void *stream)
{
    if (!ctx || !dY || !dYp || !gvals || !gmeta || counter_cols < 0 || counter_cols > O) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(O) || !sste_mult128(T) || rows <= 0 || cols <= 0 || rows > T || cols > O || token_offset % 4 != 0)
        return SSTE_ERR_SHAPE;
    if (!sste_aligned(dY, 2) || !sste_aligned(dYp, 128) || !sste_aligned(gvals, 128) || !sste_aligned(gmeta, 128))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const uint32_t ccols = static_cast<uint32_t>(counter_cols == 0 ? O : counter_cols);
    const RaggedRows rag{static_cast<const uint16_t *>(dY), static_cast<uint32_t>(rows), static_cast<uint32_t>(cols)};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    auto kern = ccols % 4 ? mvue_kernel<false, true, true, 32> : mvue_kernel<false, false, true, 32>;
    sste_launch(kern, dim3(O / 64, T / 128), dim3(256), 0, s, nullptr, O, T, static_cast<uint32_t>(seed),
                static_cast<uint32_t>(seed >> 32), tensor_id, step, token_offset / 4, ccols, AmaxIn{}, gvals,
                static_cast<uint8_t *>(gmeta), nullptr, rag, static_cast<uint4 *>(dYp));
    return launch_result();
}

namespace {

// Blocks of an amax pass: as few as four loads per thread allow, because each ends with atomics at one address (the E4M3
// prune of 1.6 M weights: 8.9 us with 800 blocks, 7.2 with 200), and eight per SM where the tensor is large (with four, 12 MB
// take 1 us longer).
int amax_grid(size_t n_chunks, int sm_count)
{
    const size_t blocks = (n_chunks + 4 * EW_THREADS - 1) / (4 * EW_THREADS), cap = static_cast<size_t>(sm_count) * 8;
    return static_cast<int>(blocks < cap ? blocks : cap);
}

sste_status amax_launch(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, void *scratch, void *stream)
{
    if (!ctx || !x || !amax_dev) return SSTE_ERR_INVALID_ARG;
    if (n == 0 || n % 8 != 0) return SSTE_ERR_SHAPE;
    if (!sste_aligned(x, 16) || !sste_aligned(amax_dev, 4) || !sste_aligned(scratch, 8)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_chunks = n / 8;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!scratch) SSTE_CUDA_TRY(cudaMemsetAsync(amax_dev, 0, sizeof(float), s));
    sste_launch(amax_kernel, dim3(amax_grid(n_chunks, ctx->sm_count)), dim3(EW_THREADS), 0, s, static_cast<const uint4 *>(x),
                n_chunks, static_cast<unsigned int *>(scratch ? scratch : amax_dev));
    return launch_result();
}

sste_status project_amax_launch(sste_ctx *ctx, const void *W, int O, int I, const float *beta_dev, float *amax_dev,
                                void *scratch, void *stream)
{
    if (!ctx || !W || !beta_dev || !amax_dev) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(O) || !sste_mult128(I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(W, 16) || !sste_aligned(amax_dev, 4) || !sste_aligned(scratch, 8)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_chunks = static_cast<size_t>(O) * I / 8;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!scratch) SSTE_CUDA_TRY(cudaMemsetAsync(amax_dev, 0, sizeof(float), s));
    sste_launch(project_amax_kernel, dim3(amax_grid(n_chunks, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                static_cast<const uint4 *>(W), n_chunks, beta_dev, amax_dev, static_cast<unsigned int *>(scratch));
    return launch_result();
}

}  // namespace

extern "C" sste_status sste_amax(sste_ctx *ctx, const void *x, size_t n, sste_dtype dt, float *amax_dev, void *stream)
{
    if (!ctx || !x || !amax_dev) return SSTE_ERR_INVALID_ARG;
    if (dt != SSTE_BF16) return SSTE_ERR_DTYPE;
    return amax_launch(ctx, x, n, amax_dev, nullptr, stream);
}

sste_status sste_amax_scratch(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, void *scratch, void *stream)
{
    return amax_launch(ctx, x, n, amax_dev, scratch, stream);
}

extern "C" sste_status sste_project_amax(sste_ctx *ctx, const void *W, int O, int I, sste_dtype wdt,
                                         const float *beta_dev, float *amax_dev, void *stream)
{
    if (!ctx || !W || !beta_dev || !amax_dev) return SSTE_ERR_INVALID_ARG;
    if (wdt != SSTE_BF16) return SSTE_ERR_DTYPE;
    return project_amax_launch(ctx, W, O, I, beta_dev, amax_dev, nullptr, stream);
}

sste_status sste_project_amax_scratch(sste_ctx *ctx, const void *W, int O, int I, const float *beta_dev, float *amax_dev,
                                      void *scratch, void *stream)
{
    return project_amax_launch(ctx, W, O, I, beta_dev, amax_dev, scratch, stream);
}

extern "C" sste_status sste_fp8_scale(sste_ctx *ctx, const float *amax_dev, sste_dtype odt, float *scale_dev,
                                      float *inv_scale_dev, void *stream)
{
    if (!ctx || !amax_dev || !scale_dev) return SSTE_ERR_INVALID_ARG;
    if (odt != SSTE_E4M3 && odt != SSTE_E5M2) return SSTE_ERR_DTYPE;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    sste_launch(fp8_scale_kernel, dim3(1), dim3(1), 0, static_cast<cudaStream_t>(stream), amax_dev,
                odt == SSTE_E4M3 ? 448.0f : 57344.0f, scale_dev, inv_scale_dev);
    return launch_result();
}

namespace {

sste_status quantize_launch(sste_ctx *ctx, const void *x, size_t n, const float *amax_dev, void *scratch, sste_dtype odt, void *q,
                            void *stream)
{
    if (!ctx || !x || !amax_dev || !q) return SSTE_ERR_INVALID_ARG;
    if (odt != SSTE_E4M3 && odt != SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (n == 0 || n % 16 != 0) return SSTE_ERR_SHAPE;
    if (!sste_aligned(x, 16) || !sste_aligned(q, 16)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_chunks = n / 8;
    const AmaxIn amax{const_cast<float *>(amax_dev), static_cast<unsigned int *>(scratch)};
    const int grid = grid_for(n_chunks, ctx->sm_count);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (odt == SSTE_E5M2)
        sste_launch(quantize_kernel<true>, dim3(grid), dim3(EW_THREADS), 0, s, static_cast<const uint4 *>(x),
                    n_chunks, amax, static_cast<uint2 *>(q));
    else
        sste_launch(quantize_kernel<false>, dim3(grid), dim3(EW_THREADS), 0, s, static_cast<const uint4 *>(x),
                    n_chunks, amax, static_cast<uint2 *>(q));
    return launch_result();
}

}  // namespace

extern "C" sste_status sste_quantize_fp8(sste_ctx *ctx, const void *x, size_t n, const float *amax_dev,
                                         sste_dtype odt, void *q, void *stream)
{
    return quantize_launch(ctx, x, n, amax_dev, nullptr, odt, q, stream);
}

sste_status sste_quantize_scratch(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, void *scratch, void *q, void *stream)
{
    return quantize_launch(ctx, x, n, amax_dev, scratch, SSTE_E4M3, q, stream);
}

namespace { unsigned int *g_taken_test = nullptr; }     // see sste_debug_withhold_maxima

extern "C" sste_status sste_debug_withhold_maxima(void *taken_dev)
{
    if (!sste_aligned(taken_dev, 4)) return SSTE_ERR_ALIGN;
    g_taken_test = static_cast<unsigned int *>(taken_dev);
    return SSTE_OK;
}

// One launch up to the size at which all blocks run at once with their values in registers (two passes' loads are plain streams), and
// from a million elements on: a product of 256 features behind it takes 8.7 us instead of 8.4 with 64 K of them, 8.8 and 8.9 with
// 256 K, 9.0 and 9.7 with 1 M, 9.4 and 10.9 with 2 M, 14.0 and 15.9 with 9.4 M.
bool sste_amax_quantize_fits(const sste_ctx *ctx, size_t n)
{
    const size_t blocks = static_cast<size_t>(ctx->sm_count) * 2;
    return blocks <= GM_SLOTS && n >= (size_t(1) << 20) && n / 8 <= blocks * AQ_THREADS * 8;
}

sste_status sste_amax_quantize(sste_ctx *ctx, const void *x, size_t n, float *amax_dev, unsigned int *slots, void *q, void *stream)
{
    if (!ctx || !x || !amax_dev || !slots || !q) return SSTE_ERR_INVALID_ARG;
    if (n == 0 || n % 16 != 0 || !sste_amax_quantize_fits(ctx, n)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(x, 16) || !sste_aligned(amax_dev, 4) || !sste_aligned(slots, 4) || !sste_aligned(q, 16)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_vec = n / 8;
    // few vectors per thread where that fills the SMs
    int v = 1;
    auto chunks = [&] { return (n_vec + AQ_THREADS * v - 1) / (AQ_THREADS * v); };
    while (chunks() > static_cast<size_t>(ctx->sm_count) * 2) v *= 2;
    auto kern = v == 1 ? amax_quantize_kernel<1> : v == 2 ? amax_quantize_kernel<2> : v == 4 ? amax_quantize_kernel<4> : amax_quantize_kernel<8>;
    sste_launch(kern, dim3(static_cast<unsigned int>(chunks())), dim3(AQ_THREADS), 0, static_cast<cudaStream_t>(stream),
                static_cast<const uint4 *>(x), n_vec, amax_dev, slots, static_cast<uint2 *>(q), ctx->status_dev, g_taken_test);
    return launch_result();
}

namespace {

// tiles per block of project_fp8_kernel: as few as keep all blocks running at once, 0 if there are too many tiles
int project_fp8_tiles(const sste_ctx *ctx, int O, int I)
{
    const long long tiles = static_cast<long long>(I / 128) * (O / PC_ROWS), sms = ctx->sm_count;
    if (sms * 4 > GM_SLOTS) return 0;
    return tiles <= sms * 4 ? 1 : tiles <= sms * 8 ? 2 : tiles <= sms * 12 ? 4 : 0;
}

}  // namespace

bool sste_project_fp8_fits(const sste_ctx *ctx, int O, int I) { return project_fp8_tiles(ctx, O, I) != 0; }

sste_status sste_project_fp8(sste_ctx *ctx, const void *W, int O, int I, const float *beta_dev, float *amax_dev, unsigned int *slots,
                             void *vals, void *meta, void *dense_out, void *stream)
{
    if (!ctx || !W || !beta_dev || !amax_dev || !slots || !vals || !meta) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(O) || !sste_mult128(I) || !sste_project_fp8_fits(ctx, O, I)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(W, 128) || !sste_aligned(vals, 128) || !sste_aligned(meta, 128) || !sste_aligned(dense_out, 128) ||
        !sste_aligned(amax_dev, 4) || !sste_aligned(slots, 4))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const int r = project_fp8_tiles(ctx, O, I);
    const uint32_t tiles = static_cast<uint32_t>(I / 128) * static_cast<uint32_t>(O / PC_ROWS), chunks = (tiles + r - 1) / r;
    auto kern = r == 1 ? project_fp8_kernel<1> : r == 2 ? project_fp8_kernel<2> : project_fp8_kernel<4>;
    sste_launch(kern, dim3(chunks), dim3(EW_THREADS), 0, static_cast<cudaStream_t>(stream), static_cast<const uint4 *>(W), I, tiles, beta_dev,
                amax_dev, slots, vals, static_cast<uint8_t *>(meta), dense_out, ctx->status_dev, g_taken_test);
    return launch_result();
}

extern "C" sste_status sste_meta_to_canonical(sste_ctx *ctx, const void *meta, int rows, int k, sste_dtype dt,
                                              void *canonical_out, void *stream)
{
    if (!ctx || !meta || !canonical_out) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(rows) || !sste_mult128(k)) return SSTE_ERR_SHAPE;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t words = static_cast<size_t>(rows) * (k / 16);
    const int grid = grid_for(words, ctx->sm_count);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (dt == SSTE_BF16)
        sste_launch(meta_to_canonical_kernel<false>, dim3(grid), dim3(EW_THREADS), 0, s,
                    static_cast<const uint8_t *>(meta), rows, k, static_cast<uint16_t *>(canonical_out));
    else
        sste_launch(meta_to_canonical_kernel<true>, dim3(grid), dim3(EW_THREADS), 0, s,
                    static_cast<const uint8_t *>(meta), rows, k, static_cast<uint16_t *>(canonical_out));
    return launch_result();
}

extern "C" sste_status sste_flip_count(sste_ctx *ctx, const void *meta_prev, const void *meta_cur, int rows, int k,
                                       unsigned long long *count_dev, void *stream)
{
    if (!ctx || !meta_prev || !meta_cur || !count_dev) return SSTE_ERR_INVALID_ARG;
    if (!sste_mult128(rows) || !sste_mult128(k)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(meta_prev, 16) || !sste_aligned(meta_cur, 16) || !sste_aligned(count_dev, 8)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_vec = sste_meta_bytes(rows, k) / 16;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    SSTE_CUDA_TRY(cudaMemsetAsync(count_dev, 0, sizeof(unsigned long long), s));
    sste_launch(flip_count_kernel, dim3(grid_for(n_vec, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                static_cast<const uint4 *>(meta_prev), static_cast<const uint4 *>(meta_cur), n_vec, count_dev);
    return launch_result();
}

extern "C" sste_status sste_decompress(sste_ctx *ctx, const void *vals, const void *meta, int rows, int k, sste_dtype dt,
                                       void *dense_out, void *stream)
{
    if (!ctx || !vals || !meta || !dense_out) return SSTE_ERR_INVALID_ARG;
    if (dt != SSTE_BF16 && dt != SSTE_E4M3 && dt != SSTE_E5M2) return SSTE_ERR_DTYPE;
    if (!sste_mult128(rows) || !sste_mult128(k)) return SSTE_ERR_SHAPE;
    if (!sste_aligned(vals, 16) || !sste_aligned(meta, 16) || !sste_aligned(dense_out, 16)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const bool eight = (dt != SSTE_BF16);
    const size_t n_units = static_cast<size_t>(rows) * k / (eight ? 32 : 16);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (eight)
        sste_launch(decompress_kernel<true>, dim3(grid_for(n_units, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                    static_cast<const uint4 *>(vals), static_cast<const uint8_t *>(meta), k, n_units,
                    static_cast<uint4 *>(dense_out));
    else
        sste_launch(decompress_kernel<false>, dim3(grid_for(n_units, ctx->sm_count)), dim3(EW_THREADS), 0, s,
                    static_cast<const uint4 *>(vals), static_cast<const uint8_t *>(meta), k, n_units,
                    static_cast<uint4 *>(dense_out));
    return launch_result();
}

extern "C" int sste_padded_dim(int n) { return n <= 0 ? 0 : (n + 127) / 128 * 128; }

extern "C" sste_status sste_pad_2d(sste_ctx *ctx, const void *src, int rows, int cols, void *dst, int rows_p, int cols_p,
                                   void *stream)
{
    if (!ctx || !src || !dst) return SSTE_ERR_INVALID_ARG;
    if (rows <= 0 || cols <= 0 || rows_p < rows || cols_p < cols || cols_p % 8 != 0) return SSTE_ERR_SHAPE;
    if (!sste_aligned(src, 2) || !sste_aligned(dst, 16)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    const size_t n_vec = static_cast<size_t>(rows_p) * cols_p / 8;
    const dim3 grid(grid_for(n_vec, ctx->sm_count));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const RaggedRows rag{static_cast<const uint16_t *>(src), static_cast<uint32_t>(rows), static_cast<uint32_t>(cols)};
    // 32-bit indices with room for one grid stride beyond the end
    if (n_vec < (size_t(1) << 31))
        sste_launch(pad_2d_kernel<uint32_t>, grid, dim3(EW_THREADS), 0, s, rag, static_cast<uint4 *>(dst), cols_p / 8, n_vec);
    else
        sste_launch(pad_2d_kernel<uint64_t>, grid, dim3(EW_THREADS), 0, s, rag, static_cast<uint4 *>(dst), cols_p / 8, n_vec);
    return launch_result();
}

namespace {

CropJob crop_job(const sste_ctx *ctx, const void *src, int rows_p, int cols_p, void *dst, int rows, int cols)
{
    CropJob j{};
    j.src = static_cast<const uint16_t *>(src);
    j.src_elements = static_cast<size_t>(rows_p) * cols_p;
    j.dst = static_cast<uint16_t *>(dst);
    j.cols_p = static_cast<uint32_t>(cols_p);
    j.cols = static_cast<uint32_t>(cols);
    j.n = static_cast<size_t>(rows) * cols;
    j.n_vec = (j.n + (reinterpret_cast<uintptr_t>(dst) & 15u) / 2 + 7) / 8;
    j.blocks = static_cast<uint32_t>(grid_for(j.n_vec, ctx->sm_count));
    return j;
}

sste_status crop_launch(const sste_ctx *, const CropJob &a, const CropJob &b, void *stream)
{
    const dim3 grid(a.blocks + b.blocks);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (a.n < (size_t(1) << 31) && b.n < (size_t(1) << 31))
        sste_launch(crop_2d_kernel<uint32_t>, grid, dim3(EW_THREADS), 0, s, a, b);
    else
        sste_launch(crop_2d_kernel<uint64_t>, grid, dim3(EW_THREADS), 0, s, a, b);
    return launch_result();
}

}  // namespace

extern "C" sste_status sste_crop_2d(sste_ctx *ctx, const void *src, int rows_p, int cols_p, void *dst, int rows, int cols,
                                    void *stream)
{
    if (!ctx || !src || !dst) return SSTE_ERR_INVALID_ARG;
    if (rows <= 0 || cols <= 0 || rows_p < rows || cols_p < cols) return SSTE_ERR_SHAPE;
    if (!sste_aligned(src, 2) || !sste_aligned(dst, 2)) return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    return crop_launch(ctx, crop_job(ctx, src, rows_p, cols_p, dst, rows, cols), CropJob{}, stream);
}

sste_status sste_crop_two(sste_ctx *ctx, const void *src0, int rows_p0, int cols_p0, void *dst0, int rows0, int cols0,
                          const void *src1, int rows_p1, int cols_p1, void *dst1, int rows1, int cols1, void *stream)
{
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    return crop_launch(ctx, crop_job(ctx, src0, rows_p0, cols_p0, dst0, rows0, cols0),
                       crop_job(ctx, src1, rows_p1, cols_p1, dst1, rows1, cols1), stream);
}

extern "C" sste_status sste_debug_mvue_groups(sste_ctx *ctx, const void *a, const void *k24, size_t n, void *pos_out,
                                              void *val_out, void *stream)
{
    if (!ctx || !a || !k24 || !pos_out || !val_out || n == 0) return SSTE_ERR_INVALID_ARG;
    if (!sste_aligned(a, 8) || !sste_aligned(k24, 4) || !sste_aligned(pos_out, 4) || !sste_aligned(val_out, 8))
        return SSTE_ERR_ALIGN;
    sste_device_guard guard(ctx->device);
    if (!guard.ok) return SSTE_ERR_CUDA;
    sste_launch(mvue_groups_kernel, dim3(grid_for(n, ctx->sm_count)), dim3(EW_THREADS), 0, static_cast<cudaStream_t>(stream),
                static_cast<const uint2 *>(a), static_cast<const uint32_t *>(k24), n, static_cast<uint32_t *>(pos_out),
                static_cast<float2 *>(val_out));
    return launch_result();
}
