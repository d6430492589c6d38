// The FP64 Hodgkin-Huxley map in 64-bit fixed point.
//
// This part issues one FP64 warp instruction per scheduler in about 64 cycles (76 with every scheduler busy), whatever
// the number of active lanes, but a 32-bit integer one in 2 and a 32x32+64 multiply-add in about 4; a 64-bit high
// product costs 16-20 cycles.  So a fixed-point evaluation of the RK4 map with 46 fractional bits of the currents, 51 to
// 66 of the increments and 55 or 62 of the state runs several times faster than the FP64 one.
//
// A value a in "format f" is the integer a 2^f.  Every intermediate has a range that the checks below guarantee: a
// state, parameter, drive or step outside it makes hh_map_fixed return false, and the caller evaluates the FP64 map
// instead (per lane).  In range, the map is as exact as the same formulas in FP64: its rms error against extended
// precision was 0.5 to 1.01 times FP64's in V, and in every binade of a gate's result from 1 down to 2^-13 at most 1.12
// times it (h deep in a spike), mostly less than it; the last addition of a gate is FP64's own, so that small gates keep
// their bits.  The stages' Jacobians keep a relative precision of FP64's, whatever their size: below threshold d/dgNa is
// off by 1.2e-16 of its rms, d/dm by 1.2e-16, d/dC (net currents of 0.1 out of 10) by 2e-14, as with FP64 instructions;
// in absolute formats of 50 to 60 bits they were off by 4.7e-14, 1.5e-15 and 4.1e-13.
//
// Measured: the FP64 map is some 650 FP64 instructions, 49 000 scheduler cycles a warp; this one 6 460 with two warps a
// scheduler (6.2e9 maps/s; 6 200 with absolute formats of 59 and 60 bits) and some 9 000 alone: integer ALU and
// multiply-add pipes together, or latency alone.  FP64 sweeps: M = 1000, 3 free parameters, 120 -> 43 us; a pass of 20
// sweeps at M = 32768, 7 free, 7.7 -> 2.06 ms.  Of these the formats that follow a gate's range and the FP64 additions
// cost 2 %, and the Jacobians' normalised products 5 % of an FP64 leapfrog step (M = 16384: 2437 -> 2570 us for four
// trajectories of 20 steps).  Normals by the FP64 functions: some 90 FP64 instructions each; here 350 cycles, of which
// the relative precision next to zeros costs 1 % of a sweep at M = 1000 (absolute formats: 5e-16 of a normal's size, rms,
// where FP64 has 9e-17).
//
// Integer arithmetic gives the same bits in every kernel and on the host, so the file also compiles as plain C++.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define PIMC_HD __host__ __device__ __forceinline__
#else
#define PIMC_HD inline
#endif

namespace pimc {

constexpr int64_t kFxOne62 = 0x4000000000000000ll;  // 1 in format 62

// ---- 64-bit products -----------------------------------------------------------------------------------------------

// floor(a b / 2^64)
PIMC_HD uint64_t fx_umul(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// a b / 2^64 for signed operands, at most 3 below it: three 32x32 + 64 multiply-adds; the low halves enter with 31
// bits so that every partial product is a signed one, and their own product is left out.  kCentred adds what that leaves
// out on average, 1.25 (sums over a path would collect it); it takes a constant's registers, so only the products that
// carry a result's last bits use it.  On the device as PTX: compiled from the C++ below it takes 25 cycles a warp
// instead of 16.
template <bool kCentred = false> PIMC_HD int64_t fx_smul(int64_t a, int64_t b)
{
#ifdef __CUDA_ARCH__
    int64_t r;
    if (kCentred) {
        asm("{\n\t.reg .s32 a0, a1, b0, b1;\n\t.reg .s64 t;\n\t"
            "mov.b64 {a0, a1}, %1;\n\tmov.b64 {b0, b1}, %2;\n\tshr.u32 a0, a0, 1;\n\tshr.u32 b0, b0, 1;\n\t"
            "mad.wide.s32 t, a1, b0, 2684354560;\n\tmad.wide.s32 t, a0, b1, t;\n\tshr.s64 t, t, 31;\n\t"
            "mad.wide.s32 %0, a1, b1, t;\n\t}"
            : "=l"(r)
            : "l"(a), "l"(b));
    } else {
        asm("{\n\t.reg .s32 a0, a1, b0, b1;\n\t.reg .s64 t;\n\t"
            "mov.b64 {a0, a1}, %1;\n\tmov.b64 {b0, b1}, %2;\n\tshr.u32 a0, a0, 1;\n\tshr.u32 b0, b0, 1;\n\t"
            "mul.wide.s32 t, a1, b0;\n\tmad.wide.s32 t, a0, b1, t;\n\tshr.s64 t, t, 31;\n\t"
            "mad.wide.s32 %0, a1, b1, t;\n\t}"
            : "=l"(r)
            : "l"(a), "l"(b));
    }
    return r;
#else
    const int32_t a1 = (int32_t)(a >> 32), b1 = (int32_t)(b >> 32);
    const int32_t a0 = (int32_t)((uint32_t)a >> 1), b0 = (int32_t)((uint32_t)b >> 1);
    const int64_t t = (int64_t)a1 * b0 + (int64_t)a0 * b1 + (kCentred ? 2684354560ll : 0ll);  // 1.25 2^31
    return (int64_t)a1 * b1 + (t >> 31);
#endif
}

// a b / 2^(64 - kMore) to the nearest: kMore more result bits, where the product leaves room for them, and the low halves'
// product counted.  Left out is the lowest bit of each operand times the other's high half: below half a unit of fx_smul,
// nothing for even operands and little for small ones.
template <int kMore> PIMC_HD int64_t fx_smul_more(int64_t a, int64_t b)
{
    const int32_t a1 = (int32_t)(a >> 32), b1 = (int32_t)(b >> 32);
    const int32_t a0 = (int32_t)((uint32_t)a >> 1), b0 = (int32_t)((uint32_t)b >> 1);
    constexpr int64_t half = 1ll << (30 - kMore);
#ifdef __CUDA_ARCH__
    int64_t t = (int64_t)(__umulhi((uint32_t)a, (uint32_t)b) >> 1) + half, r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(t) : "r"(a1), "r"(b0), "l"(t));
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(t) : "r"(a0), "r"(b1), "l"(t));
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a1), "r"(b1));
    return (int64_t)((uint64_t)r << kMore) + (t >> (31 - kMore));
#else
    const int64_t t = (int64_t)a1 * b0 + (int64_t)a0 * b1 + (int64_t)(((uint64_t)(uint32_t)a * (uint32_t)b) >> 33) + half;
    return (int64_t)((uint64_t)((int64_t)a1 * b1) << kMore) + (t >> (31 - kMore));
#endif
}

// Shifts by 0..31 bits: two funnel shifts, without the general 64-bit shift's selects.
PIMC_HD int64_t fx_sar(int64_t a, int s)
{
#ifdef __CUDA_ARCH__
    const uint32_t lo = (uint32_t)a;
    const int32_t hi = (int32_t)(a >> 32);
    return (int64_t)(((uint64_t)(uint32_t)(hi >> s) << 32) | __funnelshift_r(lo, (uint32_t)hi, s));
#else
    return a >> s;
#endif
}
PIMC_HD uint64_t fx_shl(uint64_t a, int s)
{
#ifdef __CUDA_ARCH__
    const uint32_t lo = (uint32_t)a, hi = (uint32_t)(a >> 32);
    return ((uint64_t)__funnelshift_l(lo, hi, s) << 32) | (lo << s);
#else
    return a << s;
#endif
}

// |v| < lim for |v| lim < 2^63, both to the precision of the high words (lim's low word zero).
PIMC_HD bool fx_inside(int64_t v, int64_t lim)
{
    const uint32_t h = (uint32_t)((uint64_t)v >> 32), l = (uint32_t)((uint64_t)lim >> 32);
    return h + l < 2u * l;
}

// floor(a b / 2^32)
PIMC_HD int32_t fx_mulhi32(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

PIMC_HD int fx_clz32(uint32_t v)
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

// ---- FP64 <-> fixed point by integer operations (an FP64 conversion instruction would queue for the FP64 pipe) ------

PIMC_HD uint64_t fx_bits(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    memcpy(&b, &v, 8);
    return b;
#endif
}

PIMC_HD double fx_from_bits(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, 8);
    return v;
#endif
}

// The double equal to v: normal values by integer operations (the conversion instruction queues for the FP64 pipe).
PIMC_HD double fx_widen(float v)
{
#ifdef __CUDA_ARCH__
    const uint32_t b = __float_as_uint(v), e = b & 0x7f800000u;
    if (__builtin_expect(e == 0u || e == 0x7f800000u, 0)) return (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
#else
    return (double)v;
#endif
}

// The float nearest v (ties to even): results in the normal range by integer operations.
PIMC_HD float fx_narrow(double v)
{
#ifdef __CUDA_ARCH__
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;
    if (__builtin_expect(e - 897u >= 253u, 0)) return (float)v;  // below 2^-126, near overflow, or not finite
    const uint64_t t = (b & 0x7fffffffffffffffull) + 0xfffffffull + ((b >> 29) & 1ull);
    return __uint_as_float(((uint32_t)(t >> 29) - (896u << 23)) | ((uint32_t)(b >> 32) & 0x80000000u));
#else
    return (float)v;
#endif
}

// |v| < lim for a lim whose low word is zero (false for NaN): a comparison of high words.
PIMC_HD bool fx_below(double v, double lim)
{
    return ((uint32_t)(fx_bits(v) >> 32) & 0x7fffffffu) < (uint32_t)(fx_bits(lim) >> 32);
}

// v in format f, truncated toward zero; |v| 2^f < 2^63 is the caller's.
PIMC_HD int64_t fx_of(double v, int f)
{
    const uint64_t b = fx_bits(v);
    const int sh = (int)((b >> 52) & 0x7ffu) - 1075 + f;
    const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const uint64_t r = sh >= 0 ? m << (sh & 63) : (sh > -64 ? m >> (-sh & 63) : 0ull);
    return (b >> 63) ? -(int64_t)r : (int64_t)r;
}

// The double nearest a 2^-f.
PIMC_HD double fx_double(int64_t a, int f)
{
    if (a == 0) return 0.0;
    uint64_t m = a < 0 ? 0ull - (uint64_t)a : (uint64_t)a;
    const uint32_t mh = (uint32_t)(m >> 32);
    const int lz = mh ? fx_clz32(mh) : 32 + fx_clz32((uint32_t)m);
    m <<= lz;  // bit 63 set
    // 53 bits, rounded by adding the half; a carry moves on into the exponent
    const uint64_t r = ((uint64_t)(1085 - lz - f) << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return fx_from_bits(r | ((uint64_t)a & 0x8000000000000000ull));
}

// ---- normalised values ----------------------------------------------------------------------------------------------

// A signed value with its exponent taken out, m 2^-f, for products that keep their relative precision however small the
// factors are: 2^62 <= |m| < 2^63 from fx_norm and fx_norm_of, a bit less with every product.
struct Fxn {
    int64_t m;
    int f;
};
// v in format f (values below 2^31 keep leading zeros).
PIMC_HD Fxn fx_norm(int64_t v, int f)
{
    const uint32_t h = (uint32_t)((uint64_t)(v < 0 ? -v : v) >> 32);
    const int lz = fx_clz32(h | 1u) - 1;
    return {(int64_t)fx_shl((uint64_t)v, lz), f + lz};
}
// From a double (zero below 2^-200: products of a few factors stay far from FP64's smallest exponent).
PIMC_HD Fxn fx_norm_of(double v)
{
    const uint64_t b = fx_bits(v);
    const int ex = (int)((b >> 52) & 0x7ffu);
    const int64_t m = ex >= 823 ? (int64_t)(((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) : 0;
    return {(b >> 63) ? -m : m, 1085 - ex};
}
// (Not centred: a factor of zero gives zero.)
PIMC_HD Fxn fx_fmul(const Fxn& a, const Fxn& b) { return {fx_smul(a.m, b.m) * 2, a.f + b.f - 63}; }
PIMC_HD double fx_double(const Fxn& a) { return fx_double(a.m, a.f); }
// m 2^-f as a double by the conversion instruction (its pipe is idle where this is used: 2596 -> 2570 us for the above).
PIMC_HD double fx_double_conv(int64_t m, int f)
{
    const uint64_t b = fx_bits((double)m);
    return fx_from_bits(m == 0 ? 0ull : b - ((uint64_t)(int64_t)f << 52));
}
// a b as a double.
PIMC_HD double fx_dmul(const Fxn& a, const Fxn& b) { return fx_double_conv(fx_smul(a.m, b.m), a.f + b.f - 64); }

// ---- 2^-y, 1/d -------------------------------------------------------------------------------------------------------

// 2^((j + 1/2)/256), j = 0..255, in format 62, rounded down.
#ifdef __CUDACC__
__device__
#endif
static const uint64_t kFxExp2[256] = {
    0x4016321b687027a7ull, 0x4042ad6cb2f445c0ull, 0x406f479dc5c2d056ull, 0x409c00c40ec437bcull, 0x40c8d8f50ac09dfdull,
    0x40f5d046456a29b6ull, 0x4122e6cd59676023ull, 0x41501c9ff05d8653ull, 0x417d71d3c2fb0998ull, 0x41aae67e9901ef2cull,
    0x41d87ab649524b12ull, 0x42062e90b9f4be44ull, 0x42340223e024fc1cull, 0x4261f585c05c5716ull, 0x429008cc6e5c54dfull,
    0x42be3c0e0d3949baull, 0x42ec8f60cf64fb49ull, 0x431b02daf6b94ab0ull, 0x43499692d482e623ull, 0x43784a9ec98c01e0ull,
    0x43a71f1546271897ull, 0x43d6140cca39b34eull, 0x4405299be54738bcull, 0x44345fd9367bc427ull, 0x4463b6db6cb703c5ull,
    0x44932eb946971eadull, 0x44c2c7899283a257ull, 0x44f281632eb877aeull, 0x45225c5d0950dfbeull, 0x4552588e2052780bull,
    0x4582760d81b8467dull, 0x45b2b4f24b7dcd0bull, 0x45e31553abaa24ffull, 0x46139748e05b2208ull, 0x46443ae937d07cf3ull,
    0x4675004c1077062eull, 0x46a5e788d8f3e011ull, 0x46d6f0b7102fc0ebull, 0x47081bee45623ce8ull, 0x47396946181d17c9ull,
    0x476ad8d638579e73ull, 0x479c6ab6667a0868ull, 0x47ce1efe7368e11dull, 0x47fff5c640907941ull, 0x4831ef25bff05ff6ull,
    0x48640b34f426e3fbull, 0x48964a0bf07c9cd8ull, 0x48c8abc2d8effc09ull, 0x48fb3071e240e631ull, 0x492dd83151fc5459ull,
    0x4960a3197e87fd43ull, 0x49939142cf2e06d4ull, 0x49c6a2c5bc28bf9cull, 0x49f9d7baceae6081ull, 0x4a2d303aa0fcd692ull,
    0x4a60ac5dde65950eull, 0x4a944c3d43596f95ull, 0x4ac80ff19d747c9eull, 0x4afbf793cb8a0028ull, 0x4b30033cbdb05eadull,
    0x4b643305754d1864ull, 0x4b9887070520ccd8ull, 0x4bccff5a915346cbull, 0x4c019c194f7f9080ull, 0x4c365d5c86c01061ull,
    0x4c6b433d8fbaae11ull, 0x4ca04dd5d4acffe6ull, 0x4cd57d3ed17880e0ull, 0x4d0ad19213aecf12ull, 0x4d404ae93a9df28bull,
    0x4d75e95df75cacccull, 0x4dabad0a0cd6d0beull, 0x4de196074fd9a342ull, 0x4e17a46fa7204459ull, 0x4e4dd85d0b6020ddull,
    0x4e8431e987556cf0ull, 0x4ebab12f37cfa700ull, 0x4ef156484bbe238eull, 0x4f28214f043ca19aull, 0x4f5f125db49fe7d1ull,
    0x4f96298ec2826a80ull, 0x4fcd66fca5d0fa48ull, 0x5004cac1e8d77ba1ull, 0x503c54f9284da733ull, 0x507405bd1363d308ull,
    0x50abdd286bcfc49bull, 0x50e3db5605d98bd3ull, 0x511c0060c86866e1ull, 0x51544c63ad0faf1bull, 0x518cbf79c01bcec9ull,
    0x51c559be209f3fefull, 0x51fe1b4c007f9425ull, 0x5237043ea4828570ull, 0x527014b1645b1036ull, 0x52a94cbfaab69640ull,
    0x52e2ac84f54a0ae4ull, 0x531c341cd4df284cull, 0x5355e3a2ed61adeeull, 0x538fbb32f5eca830ull, 0x53c9bae8b8d7c146ull,
    0x5403e2e013c49b4full, 0x543e3334f7ac33b7ull, 0x5478ac0368ec4fddull, 0x54b34d677f54f317ull, 0x54ee177d6635de00ull,
    0x55290a615c6c172eull, 0x5564262fb46f7d4aull, 0x559f6b04d4606292ull, 0x55dad8fd361531ccull, 0x5616703567281cb7ull,
    0x565230ca0904d3f5ull, 0x568e1ad7d0f6487cull, 0x56ca2e7b88347696ull, 0x57066bd20bf23a70ull, 0x5742d2f84d6b2e46ull,
    0x577f640b51f1922aull, 0x57bc1f2832fc3d7aull, 0x57f9046c1e3499fbull, 0x583613f45584a8acull, 0x58734dde2f251057ull,
    0x58b0b24715ab35ddull, 0x58ee414c88175e4eull, 0x592bfb0c19e2dad4ull, 0x5969dfa3730e3e6dull, 0x59a7ef30502f9d86ull,
    0x59e629d08280d778ull, 0x5a248fa1efede9f5ull, 0x5a6320c293234e5cull, 0x5aa1dd507b9c6110ull, 0x5ae0c569cdb1d2c9ull,
    0x5b1fd92cc2a823e8ull, 0x5b5f18b7a8be29e5ull, 0x5b9e8428e33b9ebeull, 0x5bde1b9eea7fba96ull, 0x5c1ddf384c0fd763ull,
    0x5c5dcf13aaa61ed4ull, 0x5c9deb4fbe40425full, 0x5cde340b542e3d8aull, 0x5d1ea9654f21226full, 0x5d5f4b7ca739f08bull,
    0x5da01a706a1875d5ull, 0x5de1165fbaea3a28ull, 0x5e223f69d2797510ull, 0x5e6395adff3c0dedull, 0x5ea5194ba562a68bull,
    0x5ee6ca623ee7b023ull, 0x5f28a9115b9e8ad9ull, 0x5f6ab578a142afb2ull, 0x5facefb7cb86e519ull, 0x5fef57eeac247deeull,
    0x6031ee3d2aeaa327ull, 0x6074b2c345cda813ull, 0x60b7a5a110f6693aull, 0x60fac6f6b6d1b5f3ull, 0x613e16e4781fc49full,
    0x6181958aac03b1a7ull, 0x61c54309c013093bull, 0x62091f8238655bd7ull, 0x624d2b14afa3dd97ull, 0x629165e1d7191068ull,
    0x62d5d00a76c07916ull, 0x631a69af6d565f3eull, 0x635f32f1b0679834ull, 0x63a42bf24c615cdcull, 0x63e954d264a12a7dull,
    0x642eadb33384aea4ull, 0x647436b60a79be09ull, 0x64b9effc520e568cull, 0x64ffd9a78a00ac53ull, 0x6545f3d9494f4209ull,
    0x658c3eb33e490c41ull, 0x65d2ba572e9da01full, 0x661966e6f76d6d26ull, 0x666044848d5a025dull, 0x66a75351fc965eb1ull,
    0x66ee937168f74cb2ull, 0x673605050e03c9a5ull, 0x677da82f3f0577ffull, 0x67c57d1267191d42ull, 0x680d83d1093f2b54ull,
    0x6855bc8dc06c554eull, 0x689e276b3f9a2fcbull, 0x68e6c48c51d7dcc0ull, 0x692f9413da5ac2f0ull, 0x69789624d48f50edull,
    0x69c1cae25429cbc6ull, 0x6a0b326f85372956ull, 0x6a54ccefac2df651ull, 0x6a9e9a8625ff4801ull, 0x6ae89b566827b9ccull,
    0x6b32cf8400c0767full, 0x6b7d373296904d78ull, 0x6bc7d285e91cd39aull, 0x6c12a1a1d0bb9037ull, 0x6c5da4aa3ea335d5ull,
    0x6ca8dbc33cfce6f4ull, 0x6cf44710eef586caull, 0x6d3fe6b790cf1604ull, 0x6d8bbadb77f21b97ull, 0x6dd7c3a112ff19a0ull,
    0x6e24012ce9e00e6eull, 0x6e7073a39dda01a2ull, 0x6ebd1b29e99e9d8cull, 0x6f09f7e4a15dd4b6ull, 0x6f5709f8b2d793b5ull,
    0x6fa4518b256d7f3bull, 0x6ff1cec11a34be7full, 0x703f81bfcc07d1feull, 0x708d6aac8f98769aull, 0x70db89acd3819528ull,
    0x7129dee620593e6dull, 0x71786a7e18c2b397ull, 0x71c72c9a79807b3full, 0x72162561198682efull, 0x726554f7ea0c4d4aull,
    0x72b4bb84f69f2cc2ull, 0x7304592e65348b0aull, 0x73542e1a763c3d1full, 0x73a43a6f84b2e424ull, 0x73f47e5406345ae8ull,
    0x7444f9ee8b0e3048ull, 0x7495ad65be522e5bull, 0x74e698e065e8ee79ull, 0x7537bc8562a47a31ull, 0x7589187bb052f921ull,
    0x75daacea65d16bceull, 0x762c79f8b51e7377ull, 0x767e7fcdeb6d26f3ull, 0x76d0be917137f4a2ull, 0x7723366aca539174ull,
    0x7775e7819601f51dull, 0x77c8d1fd8f056370ull, 0x781bf6068bb382f1ull, 0x786f53c47e0880a8ull, 0x78c2eb5f73ba413full,
    0x7916bcff964b9f6bull, 0x796ac8cd2b1fb7bdull, 0x79bf0ef0938d41c7ull, 0x7a138f924cf1f6bdull, 0x7a684adaf0c6058aull,
    0x7abd40f334af945dull, 0x7b127203ea964fccull, 0x7b67de3600b70784ull, 0x7bbd85b281b75895ull, 0x7c1368a294b96568ull,
    0x7c69872f7d6f9b61ull, 0x7cbfe1829c30863full, 0x7d1677c56e0ab137ull, 0x7d6d4a218cd895e3ull, 0x7dc458c0af549907ull,
    0x7e1ba3cca92d152aull, 0x7e732b6f6b187329ull, 0x7ecaefd302e950aeull, 0x7f22f1219ba2b4adull, 0x7f7b2f857d8c51e4ull,
    0x7fd3ab290e46d767ull,
};

PIMC_HD uint64_t fx_exp2_table(uint32_t j)
{
#ifdef __CUDA_ARCH__
    return __ldg((const unsigned long long*)kFxExp2 + j);
#else
    return kFxExp2[j];
#endif
}

// 2^frac for the fraction frac 2^-64 as a mantissa in [1, 2) of format 63: the table entry of its top 8 bits times
// e^{r ln 2}, |r| <= 2^-9, by its Taylor polynomial of degree 5 (error 2^-66); the coefficients that r^3 and higher
// powers scale down are 32-bit products.
PIMC_HD uint64_t fx_exp2_mant(uint64_t frac)
{
    const uint32_t j = (uint32_t)(frac >> 56);
    const int64_t r71 = (int64_t)((frac & 0xffffffffffffffull) - 0x80000000000000ull) * 128;
    const int32_t r39 = (int32_t)(r71 >> 32);
    const int32_t a = 1321905599 + (fx_mulhi32(r39, 733020111) >> 9);               // ln2^4/24 + r ln2^5/120, format 37
    const int32_t b = 1907106652 + (fx_mulhi32(r39, a) >> 9);                       // ln2^3/6 + ..., format 35
    const int64_t c = 0x3d7f7bff058b1d51ll + (((int64_t)r39 * b) >> 10);            // ln2^2/2 + ..., format 64
    const int64_t d = 0x58b90bfbe8e7bcd6ll + (fx_smul(r71, c) >> 8);                // ln2 + ..., format 63
    const int64_t u = fx_smul(r71, d);                                              // 2^r - 1, format 70
    const int64_t t = (int64_t)fx_exp2_table(j);
    return (uint64_t)(t + (fx_smul(t, u) >> 6)) << 1;
}

// Square of a mantissa in [1, 2) (format 63); the exponent e doubles with it.
PIMC_HD uint64_t fx_square(uint64_t m, int& e)
{
    const uint64_t s = fx_umul(m, m);  // [1, 4), format 62
    const int big = (int)(s >> 63);
    e = 2 * e + big;
    return big ? s : s << 1;
}

PIMC_HD float fx_rcp_seed(float d)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    return y;
#else
    return 1.0f / d;
#endif
}

// x = 1/d in format 61 for d = mag 2^lz 2^-64 in [1/2, 1) (mag's high word nonzero; lz is returned): an FP32 seed
// (error below 2^-22) and one third-order Newton step x0 (1 + e + e^2), e = 1 - d x0.
PIMC_HD int64_t fx_recip(uint64_t mag, int& lz)
{
    lz = fx_clz32((uint32_t)(mag >> 32) | 1u);
    const uint64_t N = fx_shl(mag, lz & 31);
    const uint32_t nh = (uint32_t)(N >> 32);
    const uint32_t fb = 0x3f000000u | ((nh << 1) >> 9);
    float fd, r;
#ifdef __CUDA_ARCH__
    fd = __uint_as_float(fb);
#else
    memcpy(&fd, &fb, 4);
#endif
    r = fx_rcp_seed(fd);
    r = r < 1.99999988f ? r : 1.99999988f;
    uint32_t rb;
#ifdef __CUDA_ARCH__
    rb = __float_as_uint(r);
#else
    memcpy(&rb, &r, 4);
#endif
    const uint32_t x0 = ((rb & 0x7fffffu) | 0x800000u) << 7;                               // format 30
    const uint64_t p = (uint64_t)nh * x0 + (((uint64_t)(uint32_t)N * x0) >> 32);           // d x0, format 62
    const int64_t e = (int64_t)(0x4000000000000000ull - p);
    const int32_t e43 = (int32_t)(e >> 19);
    const int64_t w = e + (((int64_t)e43 * e43) >> 24);
    const int64_t x1 = (int64_t)x0 << 31;  // format 61
    return x1 + (fx_smul(x1, (int64_t)((uint64_t)w << 20)) >> 18);
}

// ---- the HH map ------------------------------------------------------------------------------------------------------

// Constants of the step dt (host-made, passed to the kernels by value).  ok: dt lies in the range of the formats.
struct HhFixed {
    int64_t c_bn, c_ah, c_bm;  // dt beta_n (format 67), dt alpha_h (68), dt beta_m (62) at V = -101
    int64_t dt67, dt10, dt100; // dt (67), dt/10 (70), dt/100 (73)
    int ok;
};

inline HhFixed hh_fixed_of(double dt)
{
    HhFixed c{};
    c.ok = dt >= 0.01 && dt <= 0.04;
    if (!c.ok) return c;
    c.c_bn = fx_of(dt * 0.1960390231862711014, 67);  // 0.125 e^{36/80}
    c.c_ah = fx_of(dt * 0.42347532250890622586, 68); // 0.07 e^{36/20}
    c.c_bm = fx_of(dt * 29.556224395722600909, 62);  // 4 e^{36/18}
    c.dt67 = fx_of(dt, 67);
    c.dt10 = fx_of(dt / 10.0, 70);
    c.dt100 = fx_of(dt / 100.0, 73);
    return c;
}

// Model parameters in fixed point: conductances, reversal potentials, kappa = dt/C.
struct HhFixedParams {
    int64_t gNa, gK, gL, ENa, EK, EL, kappa;  // formats 55, 57, 60, 55, 55, 55, 66
    Fxn kap;                                  // kappa without the rounding of dt (1/C)
    bool ok;
};

// q = (gNa, gK, gL, ENa, EK, EL, C, 1/C)
PIMC_HD HhFixedParams hh_fixed_params(const HhFixed& c, const double* q, double dt)
{
    HhFixedParams p;
    const double kappa = dt * q[7];
    p.ok = c.ok && fx_below(q[0], 256.0) && fx_below(q[1], 64.0) && fx_below(q[2], 8.0) && fx_below(q[3], 150.0) &&
           fx_below(q[4], 150.0) && fx_below(q[5], 150.0) && fx_below(kappa, 0.125);
    p.gNa = fx_of(q[0], 55);
    p.gK = fx_of(q[1], 57);
    p.gL = fx_of(q[2], 60);
    p.ENa = fx_of(q[3], 55);
    p.EK = fx_of(q[4], 55);
    p.EL = fx_of(q[5], 55);
    p.kappa = fx_of(kappa, 66);
    p.kap = fx_fmul(fx_norm_of(dt), fx_norm_of(q[7]));
    return p;
}

// psi(u) = u/(1 - e^{-u}) for |u| < 1/16 in format 62, v = 10 u in format 55:
// 1 + u/2 + u^2/12 (1 - u^2/60 (1 - u^2/42 (1 - u^2/40))).
PIMC_HD int64_t fx_psi_series(int64_t v)
{
    const int64_t u = fx_smul(v * 256, 0x6666666666666666ll);  // format 65
    const int64_t u2 = fx_smul(u, u);                          // format 66
    const int64_t s1 = kFxOne62 - (fx_smul(u2, 0x19999999999999all) >> 2);
    const int64_t s2 = kFxOne62 - fx_smul(fx_smul(u2, 0x186186186186186ll), s1);
    const int64_t s3 = kFxOne62 - fx_smul(fx_smul(u2, 0x111111111111111ll), s2);
    return kFxOne62 + (u >> 4) + fx_smul(fx_smul(u2, 0x555555555555555ll), s3);
}

// psi'(u) for |u| < 1/16 in format 62: 1/2 + u/6 (1 - u^2/30 (1 - u^2/28 (1 - u^2/30))).
PIMC_HD int64_t fx_dpsi_series(int64_t v)
{
    const int64_t u = fx_smul(v * 256, 0x6666666666666666ll);  // format 65
    const int64_t u2 = fx_smul(u, u);                          // format 66
    const int64_t s1 = kFxOne62 - (fx_smul(u2, 0x222222222222222ll) >> 2);
    const int64_t s2 = kFxOne62 - fx_smul(fx_smul(u2, 0x249249249249249ll), s1);
    const int64_t s3 = kFxOne62 - fx_smul(fx_smul(u2, 0x222222222222222ll), s2);
    return (kFxOne62 >> 1) + (fx_smul(fx_smul(u, s3), 0xaaaaaaaaaaaaaabll) * 2);  // u s3: format 63; /6 (1/6, 62): 61
}

// psi'(u) for |u| >= 1/16 in format 62, from v = 10 u (55), p = 10 psi (55), x and s with 1/|1 - e^{-u}| = x 2^s.
PIMC_HD int64_t fx_dpsi(int64_t v, int64_t p, int64_t x, int s)
{
    const int64_t u = fx_smul(v, 0x6666666666666666ll);                              // format 57
    const int64_t psi = fx_smul(p, 0x6666666666666666ll);  // format 57
    int64_t n = ((int64_t)1 << 57) + u - psi;  // the sign of 1 - e^{-u}
    n = n < 0 ? -n : n;
    const int64_t q = fx_smul((int64_t)fx_shl((uint64_t)n << 3, s > 0 ? s & 15 : 0), x);  // format 57
    return fx_sar(q, s < 0 ? -s & 31 : 0) * 32;
}

// Gate rates at V (format 55, |V| < 100), each gate's in a format of its own, as fine as its range allows (the small
// values of a gate are rounded finely in FP64, too): a[g] = dt alpha in formats 62 (m), 67 (h), 64 (n), l[g] =
// dt (alpha + beta) in 62, 67, 66.  With t = V + 101 in (1, 201): e^{-t/80} and e^{-t/18} from the table, e^{-t/20} and
// B = e^{-t/10} by squaring mantissas; 1 - e^{-u} of alpha_m and alpha_n and 1 + e^{-(V+35)/10} of beta_h from B scaled
// by 2^-k, which keeps all three below 1 at every V.
// With kAdj also da[g] = dt d(alpha)/dV and db[g] = dt d(beta)/dV in formats fd[g]: 66 (m), 70 to 78 (h, whose
// derivatives fall with V), 71 (n); alpha' from psi'(u) = (1 + u - psi)/(1 - e^{-u}), or its series.
template <bool kAdj>
PIMC_HD void hh_fixed_rates(const HhFixed& c, int64_t V, int64_t a[3], int64_t l[3], int64_t* da, int64_t* db, int* fd)
{
    const uint64_t U = ((uint64_t)V + (101ull << 55)) << 1;                   // t, format 56
    const uint64_t z80 = 0ull - fx_umul(U, 0x93bb62877cdff3c9ull);           // -t log2(e)/80, format 61, modulo 8
    const uint64_t z18 = 0ull - fx_umul(U, 0xa42589ebe01547c3ull);           // -t log2(e)/18, format 59, modulo 32
    const uint64_t m1 = fx_exp2_mant(z80 << 3), m18 = fx_exp2_mant(z18 << 5);
    const int e1 = (int)(z80 >> 61) - 8, e18 = (int)(z18 >> 59) - 32;         // both negative
    int e4 = e1;
    const uint64_t m4 = fx_square(fx_square(m1, e4), e4);
    int e8 = e4;
    const uint64_t m8 = fx_square(m4, e8);                                    // B = m8 2^e8, -30 < e8 <= 0

    const int64_t bn = fx_sar((int64_t)fx_umul(m1, (uint64_t)c.c_bn), -e1);        // dt beta_n, format 66
    const int64_t ah4 = (int64_t)fx_umul(m4, (uint64_t)c.c_ah), ah = fx_sar(ah4, -e4);  // dt alpha_h, format 67
    const int64_t bm = fx_sar((int64_t)fx_umul(m18, (uint64_t)c.c_bm), -e18 - 1);  // dt beta_m, format 62

    // e^{6.1} = 1.7416 2^8, e^{4.6} = 1.5544 2^6, e^{6.6} = 1.4357 2^9: e^{-u_m}, e^{-u_n}, e^{-(V+35)/10} over B
    const int k = 11 + e8 > 0 ? 11 + e8 : 0, b = -e8 - 11 + k;  // b = max(0, -e8 - 11)
    const int64_t one = (int64_t)((uint64_t)((uint32_t)(kFxOne62 >> 32) >> k) << 32);
    const int64_t Dm = one - fx_sar((int64_t)(fx_umul(m8, 0xdeedcb68f9f2df6dull) >> 1), 2 + b);
    const int64_t Dn = one - fx_sar((int64_t)(fx_umul(m8, 0xc6f7f83846180a73ull) >> 1), 4 + b);
    const int64_t Eh = (int64_t)(fx_umul(m8, 0xb7c617949e4d1866ull) >> 1), Dh = one + fx_sar(Eh, 1 + b);
    int zm, zn, zh;
    const int64_t xm = fx_recip((uint64_t)(Dm < 0 ? -Dm : Dm), zm);
    const int64_t xn = fx_recip((uint64_t)(Dn < 0 ? -Dn : Dn), zn);
    const int64_t xh = fx_recip((uint64_t)Dh, zh);
    // 10 u/(1 - e^{-u}) = (V + V0) x 2^s, s = z - 2 - k: a left shift goes before the product (it comes with a small
    // V + V0), a right shift after it.  u and 1 - e^{-u} have the same sign.  beta_h = x 2^-s with s >= 1.
    const int64_t vm = V + (40ll << 55), vn = V + (55ll << 55);
    const int sm = zm - 2 - k, sn = zn - 2 - k, shh = k + 2 - zh;
    const int64_t pm = fx_sar(fx_smul_more<3>((int64_t)fx_shl((uint64_t)(vm < 0 ? -vm : vm), sm > 0 ? sm & 15 : 0), xm),
                              sm < 0 ? -sm & 31 : 0);  // below 160: format 55
    const int64_t pn = fx_sar(fx_smul<true>((int64_t)fx_shl((uint64_t)(vn < 0 ? -vn : vn), sn > 0 ? sn & 15 : 0), xn),
                              sn < 0 ? -sn & 31 : 0) * 8;  // its 2^-52 is 2^-64 in dt alpha_n
    int64_t am = fx_smul_more<1>(pm, c.dt10), an = fx_smul<true>(pn, c.dt100);
    const int64_t bx = fx_smul(c.dt67, xh) << 2, bh = fx_sar(bx, shh - 1);
    // |u| < 1/16: the series (the quotient above is not used there)
    constexpr int64_t kCut = 5ll << 52;  // 10/16, format 55
    const bool cut_m = fx_inside(vm, kCut), cut_n = fx_inside(vn, kCut);
    if (cut_m) am = fx_smul(c.dt67, fx_psi_series(vm)) >> 3;
    if (cut_n) an = fx_smul(c.dt10, fx_psi_series(vn)) >> 4;
    if (kAdj) {
        const int64_t dm = cut_m ? fx_dpsi_series(vm) : fx_dpsi(vm, pm, xm, sm);
        const int64_t dn = cut_n ? fx_dpsi_series(vn) : fx_dpsi(vn, pn, xn, sn);
        da[0] = fx_smul(c.dt10, dm) >> 2;
        db[0] = fx_smul(bm, -0x71c71c71c71c71c7ll) * 2;                        // -beta_m/18 (8/18 of 2^64)
        // -alpha_h/20 (8/20 of 2^64) and beta_h (1 - beta_h)/10 = beta_h^2 e^{-(V+35)/10}/10 (4/10 of 2^64)
        const int x = -e4 - 4 < 0 ? 0 : (-e4 - 4 > 8 ? 8 : -e4 - 4);
        da[1] = fx_sar(fx_smul(ah4, -0x6666666666666666ll), -e4 - x);
        const int64_t bb = fx_smul(fx_smul(bx, fx_smul(Eh, xh) << 2), 0x6666666666666666ll);
        const int r = b + 2 * shh - k - x, r1 = r > 0 ? 1 : 0;                 // 0 to 12; bb below 2^59.6, below 2^59 at r = 0
        db[1] = fx_sar(bb << (4 - r1), r - r1);
        da[2] = fx_smul(c.dt100, dn);
        db[2] = fx_smul(bn, -0x6666666666666666ll);                            // -beta_n/80 (32/80 of 2^64)
        fd[0] = 66;
        fd[1] = 70 + x;
        fd[2] = 71;
    }
    a[0] = am;
    a[1] = ah;
    a[2] = an;
    l[0] = am + bm;
    l[1] = ah + bh;
    l[2] = (an << 2) + bn;
}

// The increments dt F of the gates at state s (format 62) from the rates: formats 62 (m), 66 (h), 64 (n).  The products'
// errors are a quarter of a unit of 2^-60 (m), 2^-65 (h), 2^-64 (n).
PIMC_HD void hh_fixed_increments(const int64_t a[3], const int64_t l[3], const int64_t* s, int64_t* k)
{
    k[0] = a[0] - fx_smul_more<2>(l[0], s[0]);
    k[1] = (a[1] >> 1) - fx_smul_more<1>(l[1], s[1]);
    k[2] = a[2] - fx_smul<true>(l[2], s[2]);
}

// The part of a stage that no parameter enters: the gates' increments in k[0..2], m^3 h and n^4 (format
// 60) in k[3], k[4].  A site's parameter moves share the first stage's (the path stands still during them).
PIMC_HD void hh_fixed_gates(const HhFixed& c, int64_t V, const int64_t* s, int64_t* k)
{
    int64_t a[3], l[3];
    hh_fixed_rates<false>(c, V, a, l, nullptr, nullptr, nullptr);
    hh_fixed_increments(a, l, s, k);
    const int64_t m2 = fx_smul(s[0], s[0]) * 4, mh = fx_smul(s[0], s[1]) * 4, n2 = fx_smul(s[2], s[2]) * 4;  // format 62
    k[3] = fx_smul<true>(m2, mh);
    k[4] = fx_smul<true>(n2, n2);
}

// The increment of V, K[0] (format 51), from m^3 h and n^4; false when a term or a gate's increment K[1..3] leaves its
// format.
PIMC_HD bool hh_fixed_current(const HhFixedParams& p, int64_t I46, int64_t V, int64_t m3h, int64_t n4, int64_t* K)
{
    const int64_t tNa = fx_smul<true>(V - p.ENa, (int64_t)((uint64_t)m3h << 2));    // format 53
    const int64_t tK = fx_smul<true>(V - p.EK, (int64_t)((uint64_t)n4 << 2));
    constexpr int64_t kTwo = 1ll << 61, kT = 1ll << 61, kS = 1ll << 60;       // 2, 256, 2^14
    constexpr int64_t kM = 0x27ae147a00000000ll, kH = 0x2aaaaaaa00000000ll;  // 0.62 (62), 1/24 (66)
    const bool ok = fx_inside(m3h, kTwo) && fx_inside(n4, kTwo) && fx_inside(tNa, kT) && fx_inside(tK, kT) &&
                    fx_inside(K[1], kM) && fx_inside(K[2], kH);
    const int64_t tKL = fx_smul<true>(p.gK, (int64_t)((uint64_t)tK << 2)) + (fx_smul<true>(p.gL, V - p.EL) >> 3);  // 48
    const int64_t S = I46 - fx_smul<true>(p.gNa, (int64_t)((uint64_t)tNa << 2)) - ((tKL + 2) >> 2);
    K[0] = fx_smul_more<1>((int64_t)((uint64_t)S << 2), p.kappa);
    constexpr int64_t kK = 100ll << 51;
    return ok && fx_inside(S, kS) && fx_inside(K[0], kK);
}

// What the reverse pass of one stage takes: the Jacobian of its increments K = dt F, as doubles of FP64's own relative
// precision (the small entries below threshold -- m^3 h is 1e-4 there -- are what data without spikes have):
//   kJlam: -dK_g/ds_g (3), kJgam: dK_g/dV (3), kJV: dK_0/dV, kJg: -dK_0/ds_g (3), and -dK_0/dgNa, -dK_0/dgK, -dK_0/dgL,
//   dK_0/dENa, dK_0/dEK, K_0 (dK_0/dEL = kappa gL and dK_0/dC = -K_0/C are the caller's).
enum { kJlam = 0, kJgam = 3, kJV = 6, kJg = 7, kJp = 10, kJlen = 16 };

// A stage's increments -- K[0] of V (format 51), K[1..3] of the gates (as hh_fixed_increments) -- and its Jacobian:
// element j goes to J[j * stride].  sn: the gates s normalised; kNa, kK: kappa gNa, kappa gK; kq: kappa I, gNa, gK, gL
// and kappa gL as doubles.  dK_0/dV and K_0 are sums of entries formed in FP64, whose pipe is idle here (five operations).
PIMC_HD bool hh_fixed_stage_adj(const HhFixed& c, const HhFixedParams& p, int64_t I46, int64_t V, const int64_t* s,
                                const Fxn* sn, const Fxn& kNa, const Fxn& kK, const double* kq, int64_t* K, double* J,
                                int stride)
{
    int64_t a[3], l[3], da[3], db[3];
    int fd[3];
    hh_fixed_rates<true>(c, V, a, l, da, db, fd);
    hh_fixed_increments(a, l, s, K + 1);
    constexpr int kFl[3] = {62, 67, 66};
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        J[(kJlam + g) * stride] = fx_double(l[g], kFl[g]);
        J[(kJgam + g) * stride] = fx_double(da[g] - fx_smul_more<2>(da[g] + db[g], s[g]), fd[g]);
    }
    const int64_t m2 = fx_smul(s[0], s[0]) * 4, mh = fx_smul(s[0], s[1]) * 4, n2 = fx_smul(s[2], s[2]) * 4;  // format 62
    const bool ok = hh_fixed_current(p, I46, V, fx_smul<true>(m2, mh), fx_smul<true>(n2, n2), K);
    const Fxn vNa = fx_norm(V - p.ENa, 55), vK = fx_norm(V - p.EK, 55), vL = {V - p.EL, 55};
    const Fxn mm = fx_fmul(sn[0], sn[0]), m3 = fx_fmul(mm, sn[0]), m3h = fx_fmul(m3, sn[1]);
    const Fxn nn = fx_fmul(sn[2], sn[2]), n3 = fx_fmul(nn, sn[2]), n4 = fx_fmul(n3, sn[2]);
    const Fxn kvNa = fx_fmul(kNa, vNa), kvK = fx_fmul(kK, vK);
    const Fxn gm = fx_fmul(kvNa, fx_fmul(mm, sn[1]));
    const double dNa = fx_dmul(fx_fmul(p.kap, vNa), m3h), dK = fx_dmul(fx_fmul(p.kap, vK), n4), dL = fx_dmul(p.kap, vL);
    const double eNa = fx_dmul(kNa, m3h), eK = fx_dmul(kK, n4);
    J[(kJg + 0) * stride] = fx_double_conv((gm.m >> 2) * 3, gm.f - 2);
    J[(kJg + 1) * stride] = fx_dmul(kvNa, m3);
    J[(kJg + 2) * stride] = fx_dmul({kvK.m, kvK.f - 2}, n3);
    J[(kJp + 0) * stride] = dNa;
    J[(kJp + 1) * stride] = dK;
    J[(kJp + 2) * stride] = dL;
    J[(kJp + 3) * stride] = eNa;
    J[(kJp + 4) * stride] = eK;
    J[(kJp + 5) * stride] = fma(-kq[3], dL, fma(-kq[2], dK, fma(-kq[1], dNa, kq[0])));
    J[kJV * stride] = -(eNa + eK + kq[4]);
    return ok;
}

// Whether a state in fixed point is inside the range of the stage: |V| < 100, |gate| < 1.41 (their products of two stay
// below 2; sampled gates scatter past 1 at the spikes).
PIMC_HD bool hh_fixed_inside(int64_t V, const int64_t* s)
{
    constexpr int64_t kV = 100ll << 55, kS = 0x5a3d70a300000000ll;  // 1.41, format 62
    return fx_inside(V, kV) && fx_inside(s[0], kS) && fx_inside(s[1], kS) && fx_inside(s[2], kS);
}

// The next stage's state and the weighted sums of the increments after stage st (weights 1, 2, 2, 1): aV in format 51,
// as[g] in formats 61 (m), 65 (h), 63 (n): room for six increments, below 0.62, 1/24 (both checked) and 0.153.
PIMC_HD void hh_fixed_step(int st, int64_t V0, const int64_t* s0, const int64_t* K, int64_t& V, int64_t* s, int64_t& aV,
                           int64_t* as)
{
    const int w = (st == 1 || st == 2) ? 1 : 0, d = st < 2 ? 0 : 1;  // weight 2^w; next stage at x + K 2^(d - 1)
    constexpr int kTo62[3] = {1, 5, 3};                              // K[1 + g] / 2 to format 62
    aV += K[0] << w;
    V = V0 + (K[0] << (3 + d));
#pragma unroll
    for (int g = 0; g < 3; ++g) {
        as[g] += w ? K[1 + g] : (K[1 + g] + (st >> 1)) >> 1;  // one rounding down, one up
        s[g] = s0[g] + (K[1 + g] >> (kTo62[g] - d));
    }
}

// f from the sums.  The gates' increment is added to x in FP64: rounded once, with every bit of a small x in it.
PIMC_HD void hh_fixed_result(const double* x, int64_t V0, int64_t aV, const int64_t* as, double* f)
{
    constexpr int64_t kSixth = 0x5555555555555555ll;  // 1/6, format 65
    f[0] = fx_double(V0 + fx_smul<true>(aV * 4, kSixth) * 2, 55);
    f[1] = x[1] + fx_double(fx_smul<true>(as[0], kSixth), 62);
    f[2] = x[2] + fx_double(fx_smul_more<1>(as[1], kSixth), 67);
    f[3] = x[3] + fx_double(fx_smul<true>(as[2], kSixth), 64);
}

// One RK4 step of the HH field, f = x + (K1 + 2 K2 + 2 K3 + K4)/6, drive held at I.  False (f untouched) when a value
// leaves the range of the formats.  s1: the first stage's parameter-free part (hh_fixed_gates), element g at
// s1[g * stride], taken from there (kStage1Load; written for this very x) or left there (kStage1Store) -- the same bits.
enum { kStage1None, kStage1Store, kStage1Load };
PIMC_HD bool hh_map_fixed(const HhFixed& c, const HhFixedParams& p, const double* x, double I, double* f,
                          int first = kStage1None, int64_t* s1 = nullptr, int64_t stride = 0)
{
    if (!p.ok || !fx_below(x[0], 100.0) || !fx_below(x[1], 1.375) || !fx_below(x[2], 1.375) ||
        !fx_below(x[3], 1.375) || !fx_below(I, 16384.0))
        return false;
    const int64_t V0 = fx_of(x[0], 55), I46 = (fx_of(I, 47) + 1) >> 1;
    int64_t s0[3], V = V0, s[3], aV = 0, as[3] = {0, 0, 0}, K[4];
    for (int g = 0; g < 3; ++g) s[g] = s0[g] = fx_of(x[1 + g], 62);
    // one copy of the stage's code: four would not fit the instruction cache
#pragma unroll 1
    for (int st = 0; st < 4; ++st) {
        if (first == kStage1Load && st == 0) {
#pragma unroll
            for (int g = 0; g < 3; ++g) K[1 + g] = s1[g * stride];
            if (!hh_fixed_current(p, I46, V, s1[3 * stride], s1[4 * stride], K)) return false;
        } else {
            int64_t k[5];
            hh_fixed_gates(c, V, s, k);
            if (first == kStage1Store && st == 0) {
#pragma unroll
                for (int g = 0; g < 5; ++g) s1[g * stride] = k[g];
            }
#pragma unroll
            for (int g = 0; g < 3; ++g) K[1 + g] = k[g];
            if (!hh_fixed_current(p, I46, V, k[3], k[4], K)) return false;
        }
        hh_fixed_step(st, V0, s0, K, V, s, aV, as);
        if (st < 3 && !hh_fixed_inside(V, s)) return false;
    }
    hh_fixed_result(x, V0, aV, as, f);
    return true;
}

// The forward half of the adjoint: f as hh_map_fixed (the same bits), and the four stages' Jacobians, element j of stage
// st at J[(st * kJlen + j) * stride].  False when a value leaves the range (f untouched, J undefined).
PIMC_HD bool hh_map_fixed_adj(const HhFixed& c, const HhFixedParams& p, const double* x, double I, double* f, double* J,
                              int stride)
{
    if (!p.ok || !fx_below(x[0], 100.0) || !fx_below(x[1], 1.375) || !fx_below(x[2], 1.375) ||
        !fx_below(x[3], 1.375) || !fx_below(I, 16384.0))
        return false;
    const int64_t V0 = fx_of(x[0], 55), I46 = (fx_of(I, 47) + 1) >> 1;
    int64_t s0[3], V = V0, s[3], aV = 0, as[3] = {0, 0, 0}, K[4];
    Fxn sn[3];
    for (int g = 0; g < 3; ++g) {
        s[g] = s0[g] = fx_of(x[1 + g], 62);
        sn[g] = fx_norm_of(x[1 + g]);
    }
    const Fxn kNa = fx_fmul(p.kap, fx_norm(p.gNa, 55)), kK = fx_fmul(p.kap, fx_norm(p.gK, 57));
    const double kq[5] = {fx_double(fx_fmul(p.kap, fx_norm_of(I))), fx_double(p.gNa, 55), fx_double(p.gK, 57),
                          fx_double(p.gL, 60), fx_double(fx_fmul(p.kap, fx_norm(p.gL, 60)))};
#pragma unroll 1
    for (int st = 0; st < 4; ++st) {
        if (!hh_fixed_stage_adj(c, p, I46, V, s, sn, kNa, kK, kq, K, J + (int64_t)st * kJlen * stride, stride)) return false;
        hh_fixed_step(st, V0, s0, K, V, s, aV, as);
        if (st < 3 && !hh_fixed_inside(V, s)) return false;
#pragma unroll
        for (int g = 0; g < 3; ++g) sn[g] = fx_norm(s[g], 62);
    }
    hh_fixed_result(x, V0, aV, as, f);
    return true;
}

// The reverse half, in FP64: w is the cotangent of f; gx = J_x f^T w, gp += J_p f^T w (7 entries).  kgL = kappa gL,
// iC = 1/C.  With the increments' Jacobians: u = JK^T b stage by stage from b_4 = w/6, b_3 = w/3 + u_4,
// b_2 = w/3 + u_3/2, b_1 = w/6 + u_2/2, and gx = w + u_1 + ... + u_4.
PIMC_HD void hh_reverse(const double* J, int stride, double kgL, double iC, const double* w, double* gx, double* gp)
{
    double u[4], gq[6] = {0, 0, 0, 0, 0, 0}, sb = 0.0;
    const double sixth = 1.0 / 6.0, third = 1.0 / 3.0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        gx[a] = w[a];
        u[a] = 0.0;
    }
#pragma unroll 1
    for (int st = 3; st >= 0; --st) {
        const double* j = J + (int64_t)st * kJlen * stride;
        const double cw = (st == 0 || st == 3) ? sixth : third, cu = st == 2 ? 1.0 : 0.5;
        double b[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) b[a] = fma(cu, u[a], cw * w[a]);
        u[0] = b[0] * j[kJV * stride];
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            u[0] = fma(b[1 + g], j[(kJgam + g) * stride], u[0]);
            u[1 + g] = fma(-b[1 + g], j[(kJlam + g) * stride], -b[0] * j[(kJg + g) * stride]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) gx[a] += u[a];
#pragma unroll
        for (int l = 0; l < 6; ++l) gq[l] = fma(b[0], j[(kJp + l) * stride], gq[l]);
        sb += b[0];
    }
    gp[0] -= gq[0];
    gp[1] -= gq[1];
    gp[2] -= gq[2];
    gp[3] += gq[3];
    gp[4] += gq[4];
    gp[5] = fma(kgL, sb, gp[5]);
    gp[6] = fma(-iC, gq[5], gp[6]);
}

// ---- draws -----------------------------------------------------------------------------------------------------------
// The FP64 draws -- Box-Muller normals and -log u -- from their integers: the uniform (k + 1/2) 2^-52, k < 2^52, is
// N 2^-53 with N = 2 k + 1.  Relative errors below 2^-53 beside the rounding, for small values as well: -log u near
// u = 1, the radius made of it, and the sine and cosine next to their zeros are formed from normalised mantissas.

// log(C_j/256), format 63, and C_j, about 256 over the middle of [1/2 + j/256, 1/2 + (j + 1)/256); C_127 = 256.
#ifdef __CUDACC__
__device__
#endif
static const uint64_t kFxLog[128] = {
    0x5838cbd11e23632aull, 0x5736c771b05d9234ull, 0x5632b6d735e624c2ull, 0x552c919e66525ea4ull, 0x54669302e8d1199bull,
    0x535cb4e8e7f4011dull, 0x5250aa0e8bf01dedull, 0x51862f08717b09f4ull, 0x50763fa119cab992ull, 0x4fa8ce4dacbd6e0full,
    0x4e94dcf9faf7e632ull, 0x4dc45ed51d1ed717ull, 0x4cac4ce44875c4c8ull, 0x4bd8aa65425518b6ull, 0x4b03a7b5123a2ee6ull,
    0x4a2d4037d81e0abcull, 0x49556f3a63df2cf0ull, 0x483373464aadb64dull, 0x475843f99dc00c21ull, 0x467b9ad19f25bb31ull,
    0x459d72aeae98380eull, 0x44bdc6564fbef14cull, 0x43dc90726d25f53bull, 0x43458f32e75adf82ull, 0x4261bd3d5cd482e4ull,
    0x417c52f49916702aull, 0x40954a969743fb1aull, 0x3fac9e41ec2ae395ull, 0x3f10946dfd3d8459ull, 0x3e251ebf5e0dd967ull,
    0x3d37f4cb30c3eac9ull, 0x3c98e350d0ee085aull, 0x3ba8d4098389417eull, 0x3b07ce4b145e7ca1ull, 0x3a14c75ce43cc84bull,
    0x3971c0e89af593fbull, 0x387baf4f9b5a9ae7ull, 0x37d69b3b4e36f7efull, 0x3730b12d2621f6b3ull, 0x36363c1d7bf8b6d2ull,
    0x358e3184b161c818ull, 0x34e5492cd7b3d42dull, 0x33e647d97f3097e5ull, 0x333b2b022fc11597ull, 0x328f2838422df575ull,
    0x31e23d0e6cc58efcull, 0x3134670d8284b56bull, 0x302de83b41a92b6bull, 0x2f7dbc146f5f7f3cull, 0x2ecc9c2473b79d82ull,
    0x2e1a85c4f1246babull, 0x2d6776446b287b13ull, 0x2cb36ae607c3e504ull, 0x2bfe60e14f27a791ull, 0x2b485561e99fc339ull,
    0x2a9145875ba4c5a0ull, 0x29d92e64c004d35full, 0x29200d008013a198ull, 0x2865de5409d0276bull, 0x2808610d0d4fc77aull,
    0x274c98aad28bd38eull, 0x268fbb3530faa9adull, 0x25d1c575c23a6138ull, 0x2512b427bd0d46bdull, 0x245283f79ef2cb45ull,
    0x23f1ff3c9145e51bull, 0x23301a5ba846decfull, 0x226d0e05275160beull, 0x220b17f35c95aa31ull, 0x214649c4e721c6bfull,
    0x20804b2969a081b6ull, 0x201cd88b5aa0398dull, 0x1f550a564b7b3707ull, 0x1e8c0252aa5a5fe9ull, 0x1e27076e2af2e5eaull,
    0x1d5c216b4fbb915cull, 0x1c8ff7c79a9a21acull, 0x1c2968558c18c0a3ull, 0x1b5b519e8fb5a46full, 0x1af3c94e80bff2d9ull,
    0x1a23bc1fe2b56319ull, 0x19bb362e7dfb8356ull, 0x18e928de886d40aaull, 0x187fa06520c91090ull, 0x17ab890210d9091cull,
    0x1740f8f54037a4caull, 0x16d60fe719d21c8dull, 0x15ff3070a793d3c8ull, 0x159338d9982085d3ull, 0x14ba36f39a55e55aull,
    0x144d2b6ccb7d1e68ull, 0x13dfc2b0ecc629cbull, 0x1303d718e47fd2ffull, 0x129552f81ff5234cull, 0x12266f190a5acb7dull,
    0x114785846742ac69ull, 0x10d77e7cd08e5967ull, 0x10671512ca596e2aull, 0xf85186008b15331ull, 0xf1383b7157972f5ull,
    0xea189eb3659aeafull, 0xe2f2a47ade3a18bull, 0xd49369d256ab1b3ull, 0xcd5a1231019d66eull, 0xc61a2eb18cd907bull,
    0xbed3b36bd896642ull, 0xb032c549ba861d9ull, 0xa8d839f830c1fb5ull, 0xa176e5f5323781eull, 0x9a0ebcb0de8e849ull,
    0x929fb17850a0b7cull, 0x8b29b7751bd7074ull, 0x7c28c300458a998ull, 0x749dae2b6c2d484ull, 0x6d0b75c465c6fb1ull,
    0x65720c3b238fadfull, 0x5dd163d8cb73f12ull, 0x56296ebf2393523ull, 0x4e7a1ee7faf57eaull, 0x46c366248f65ff1ull,
    0x3f05361cf06600aull, 0x373f804f5f232ffull, 0x2f72360fab62355ull, 0x279d48868d4ae9eull, 0x1fc0a8b0fc03e3dull,
    0x17dc475f810a76eull, 0xff015358833c48ull, 0x0ull,
};
#ifdef __CUDACC__
__device__
#endif
static const uint16_t kFxLogC[128] = {
    510, 506, 502, 498, 495, 491, 487, 484, 480, 477, 473, 470, 466, 463, 460, 457, 454, 450, 447, 444,
    441, 438, 435, 433, 430, 427, 424, 421, 419, 416, 413, 411, 408, 406, 403, 401, 398, 396, 394, 391,
    389, 387, 384, 382, 380, 378, 376, 373, 371, 369, 367, 365, 363, 361, 359, 357, 355, 353, 351, 350,
    348, 346, 344, 342, 340, 339, 337, 335, 334, 332, 330, 329, 327, 325, 324, 322, 320, 319, 317, 316,
    314, 313, 311, 310, 308, 307, 306, 304, 303, 301, 300, 299, 297, 296, 295, 293, 292, 291, 289, 288,
    287, 286, 284, 283, 282, 281, 279, 278, 277, 276, 275, 274, 272, 271, 270, 269, 268, 267, 266, 265,
    264, 263, 262, 261, 260, 259, 258, 256,
};
// sin(pi/2 (j + 1/2)/64), format 63.
#ifdef __CUDACC__
__device__
#endif
static const uint64_t kFxSin[64] = {
    0x1921d1fcdec7846ull, 0x4b6195d65157345ull, 0x7d95b9e7e0837fbull, 0xafb68054d520c60ull, 0xe1bc2e3cf616a7aull,
    0x1139f0cedaf576abull, 0x145576b1293e59daull, 0x176dd9de50bf3147ull, 0x1a82a025b004509eull, 0x1d934fe54543115dull,
    0x209f701c6ffb5bfeull, 0x23a6887e99b67ba3ull, 0x26a82185c302a361ull, 0x29a3c484f1ced449ull, 0x2c98fbba7e4f8c22ull,
    0x2f8752623b99ce03ull, 0x326e54c77927ae5aull, 0x354d9056da7f9315ull, 0x382493b0023dcd3full, 0x3af2eeb70dc712aaull,
    0x3db832a5def1ab11ull, 0x4073f21d30fadb65ull, 0x4325c13576263a72ull, 0x45cd358f7b6d2281ull, 0x4869e664cfad62c5ull,
    0x4afb6c97ebcfa7ddull, 0x4d8162c41967cae0ull, 0x4ffb654d155b5136ull, 0x5269126e6c24e2d8ull, 0x54ca0a4a8d56572full,
    0x571deef994063106ull, 0x59646497c1e0f5c3ull, 0x5b9d1153aaa2ba24ull, 0x5dc79d7c0dc984aeull, 0x5fe3b38d5c5dc263ull,
    0x61f1003ee8bafad2ull, 0x63ef328fbe5033a4ull, 0x65ddfbd31f5d06eaull, 0x67bd0fbca6be50d8ull, 0x698c246c0beb870bull,
    0x6b4af278875442b8ull, 0x6cf934fbd55c4614ull, 0x6e96a99cd643497eull, 0x70231099c9552436ull, 0x719e2cd221ce6c76ull,
    0x7307c3cff3f170f2ull, 0x745f9dd0f8d76fddull, 0x75a585cf279a2b0bull, 0x76d94988e2826b29ull, 0x77fab988b6f8aaaeull,
    0x7909a92caf05f9a8ull, 0x7a05eead33443317ull, 0x7aef63237c2dd0e3ull, 0x7bc5e28f91cf0963ull, 0x7c894bddd8eb66dfull,
    0x7d3980ec2cbcb338ull, 0x7dd6668e8481dd84ull, 0x7e5fe49324266a1dull, 0x7ed5e5c6575d048dull, 0x7f3857f5b699eb51ull,
    0x7f872bf2f56c2468ull, 0x7fc2559639c6b501ull, 0x7fe9cbbffbdd7274ull, 0x7ffd885a6e4b6d5dull,
};

PIMC_HD int64_t fx_log_table(uint32_t j)
{
#ifdef __CUDA_ARCH__
    return (int64_t)__ldg((const unsigned long long*)kFxLog + j);
#else
    return (int64_t)kFxLog[j];
#endif
}
PIMC_HD uint32_t fx_logc_table(uint32_t j)
{
#ifdef __CUDA_ARCH__
    return __ldg((const unsigned short*)kFxLogC + j);
#else
    return kFxLogC[j];
#endif
}
PIMC_HD int64_t fx_sin_table(uint32_t j)
{
#ifdef __CUDA_ARCH__
    return (int64_t)__ldg((const unsigned long long*)kFxSin + j);
#else
    return (int64_t)kFxSin[j];
#endif
}

// -log(N 2^-53) for odd N < 2^53, in format F (returned): 57 for u < 1/2, 63 for u in [1/2, 255/256); above, where the
// logarithm goes to 0, 70 + s with the result in [2^61, 2^62.1).
// u = m 2^-E, m in [1/2, 1): E log 2 + log c_j - log(m c_j), with r = 1 - m c_j exact (|r| < 2^-7) and
// -log(1 - r) = r + r^2/2 + ... + r^8/8 (error 2^-66).
PIMC_HD int64_t fx_neglog(uint64_t N, int& F)
{
    const uint32_t nh = (uint32_t)(N >> 32);
    const int lz = nh ? fx_clz32(nh) : 32 + fx_clz32((uint32_t)N);
    const uint64_t m = N << lz;  // format 64; its low 11 bits are zero
    const uint32_t j = (uint32_t)(m >> 56) & 0x7fu;
    const int64_t r70 = (int64_t)(0ull - (m >> 8) * fx_logc_table(j)) * 64;
    const int32_t r38 = (int32_t)(r70 >> 32);
    const int32_t t7 = 306783378 + (fx_mulhi32(r38, 268435456) >> 6);  // 1/7 + r/8, format 31
    const int32_t t6 = 357913941 + (fx_mulhi32(r38, t7) >> 6);
    const int32_t t5 = 429496730 + (fx_mulhi32(r38, t6) >> 6);
    const int64_t t4 = (kFxOne62 >> 2) + (((int64_t)r38 * t5) >> 7);       // 1/4 + ..., format 62
    const int64_t t3 = 0x1555555555555555ll + (fx_smul(r70, t4) >> 6);
    const int64_t t2 = (kFxOne62 >> 1) + (fx_smul(r70, t3) >> 6);
    const int64_t q = fx_smul(r70, t2);                                    // r/2 + r^2/3 + ..., format 68
    const int E = lz - 11;
    if (E == 0 && j == 127u) {  // r > 0: r (1 + q) from r's mantissa
        const uint32_t rh = (uint32_t)((uint64_t)r70 >> 32);
        const int s = (rh ? fx_clz32(rh) : 32 + fx_clz32((uint32_t)r70)) - 2;  // to [2^61, 2^62): 1 + q < 1 + 2^-8
        const int64_t rm = (int64_t)((uint64_t)r70 << s);
        F = 70 + s;
        return rm + (fx_smul(rm, q << 3) >> 7);
    }
    const int64_t w = r70 + (fx_smul(r70, q) >> 4);                        // format 70
    const int64_t lc = fx_log_table(j);
    F = E > 0 ? 57 : 63;
    if (E == 0) return lc + (w >> 7);
    // log 2 in format 57 and its rest in format 68
    return (int64_t)E * 0x162e42fefa39ef3ll + ((E * (701)) >> 11) + (lc >> 6) + (w >> 13);
}

PIMC_HD float fx_rsqrt_seed(float d)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    return y;
#else
    return 1.0f / __builtin_sqrtf(d);
#endif
}

// sqrt(2 a 2^-F) for a > 0 as a mantissa in [2^61, 2^62] of format f (returned).  With 2 a 2^-F = d 4^h, d in [1/4, 1):
// an FP32 seed y of 1/sqrt(d) and sqrt(d) = d y (1 + e/2 + 3 e^2/8), e = 1 - d y^2 (|e| < 2^-21).
PIMC_HD int64_t fx_sqrt2(int64_t a, int F, int& f)
{
    const uint32_t ah = (uint32_t)((uint64_t)a >> 32);
    int lz = ah ? fx_clz32(ah) : 32 + fx_clz32((uint32_t)a);
    // 2 a 2^-F = (a << lz) 2^-64 2^(65 - F - lz): an even exponent 2 h
    int ex = 65 - F - lz;
    const int odd = ex & 1;
    const uint64_t d = ((uint64_t)a << lz) >> odd;
    f = 62 - ((ex + odd) >> 1);
    const uint32_t dh = (uint32_t)(d >> 32);
    float y = fx_rsqrt_seed((float)(dh >> 8) * 0x1p-24f);
    y = y < 1.99999988f ? y : 1.99999988f;
    const uint32_t y0 = (uint32_t)(int32_t)(y * 0x1p30f);                          // format 30, in [2^30, 2^31)
    const uint64_t g = (uint64_t)dh * y0 + (((uint64_t)(uint32_t)d * y0) >> 32);   // d y, format 62
    const int64_t e = (int64_t)((1ull << 60) - fx_umul(d, (uint64_t)y0 * y0));     // format 60
    const int32_t e41 = (int32_t)(e >> 19);
    const int64_t c = (e >> 1) + ((3 * (((int64_t)e41 * e41) >> 22)) >> 3);        // format 60
    return (int64_t)g + (fx_smul((int64_t)g, c * (1 << 20)) >> 16);                // format 62
}

// sin(theta) for theta = pi/2 d 2^-64 > 0, d < 2^56 (theta < 2^-7.3), as theta (1 - theta^2/6 + theta^4/120) from the mantissa
// of d (the rest is below 2^-56 of it), in format f (returned).
PIMC_HD int64_t fx_sin_small(uint64_t d, int& f)
{
    constexpr int64_t kHalfPi = 0x6487ed5110b4611all;                                       // pi/2, format 62
    const uint32_t h = (uint32_t)(d >> 32);
    const int s = (h ? fx_clz32(h) : 32 + fx_clz32((uint32_t)d)) - 1;
    const int64_t t = fx_smul((int64_t)(d << 7), kHalfPi), t2 = fx_smul(t, t);              // theta (69), theta^2 (74)
    const int64_t q = fx_smul(t2, 0xaaaaaaaaaaaaaabll - (fx_smul(t2, 0x4444444444444444ll) >> 17));  // format 72
    const int64_t tm = fx_smul<true>((int64_t)(d << s), kHalfPi);                           // theta, format 62 + s
    f = 62 + s;
    return tm - (fx_smul(tm, q) >> 8);
}

// (cos, sin)(2 pi N 2^-53) in formats fc, fs (62 but next to a zero): quadrant, 64 table angles a in it, and the angle
// difference delta (|delta| <= pi/256) by its Taylor polynomials of degree 7 and 6 (errors below 2^-66 and 2^-60).
PIMC_HD void fx_sincos(uint64_t N, int64_t& cs, int64_t& sn, int& fc, int& fs)
{
    const uint32_t q = (uint32_t)(N >> 51);
    const uint64_t fr = N << 13;  // fraction of the quadrant, format 64
    const uint32_t j = (uint32_t)(fr >> 58);
    const int64_t r70 = (int64_t)((fr & 0x3ffffffffffffffull) - 0x200000000000000ull) * 64;
    const int64_t dl = fx_smul(r70, 0x6487ed5110b4611all) * 2;  // delta, format 69
    const int64_t d2 = fx_smul(dl, dl);                         // format 74
    const int32_t d42 = (int32_t)(d2 >> 32);
    const int32_t ts = 1145324612 - (fx_mulhi32(d42, 218157069) >> 13);                    // 1/120 - d2/5040, format 37
    const int64_t us = -0xaaaaaaaaaaaaaabll + (((int64_t)d42 * ts) >> 17);                 // format 62
    const int64_t sd = dl + (fx_smul(dl, fx_smul(d2, us)) >> 8);                           // sin delta, format 69
    const int32_t tc = 1431655765 - (fx_mulhi32(d42, 763549742) >> 14);                    // 1/24 - d2/720, format 35
    const int64_t c1 = fx_smul(d2, -(kFxOne62 >> 1) + (((int64_t)d42 * tc) >> 15));        // cos delta - 1, format 72
    const int64_t S = fx_sin_table(j), C = fx_sin_table(63u - j);
    int64_t s0 = (S >> 1) + (fx_smul(S, c1) >> 9) + (fx_smul(C, sd) >> 6);
    int64_t c0 = (C >> 1) + (fx_smul(C, c1) >> 9) - (fx_smul(S, sd) >> 6);
    // within 2^-8 of a quadrant of a zero (one pair in 128)
    const uint64_t near_end = fr >> 63 ? 0ull - fr : fr;
    int f0 = 62;
    if (near_end < (1ull << 56)) {
        const int64_t z = fx_sin_small(near_end, f0);
        if (fr >> 63) c0 = z;
        else s0 = z;
    }
    const int f1 = fr >> 63 ? f0 : 62, f2 = fr >> 63 ? 62 : f0;  // of c0, s0
    const int64_t a = (q & 1u) ? -s0 : c0, b = (q & 1u) ? c0 : s0;
    cs = (q & 2u) ? -a : a;
    sn = (q & 2u) ? -b : b;
    fc = (q & 1u) ? f2 : f1;
    fs = (q & 1u) ? f1 : f2;
}

// N of the open-interval uniform that two Philox words give: k from the top 26 bits of each.
PIMC_HD uint64_t fx_uniform(uint32_t hi, uint32_t lo)
{
    return ((((uint64_t)(hi >> 6) << 26) | (uint64_t)(lo >> 6)) << 1) | 1ull;
}

// Box-Muller from four words: sqrt(-2 log u1) (cos, sin)(2 pi u2).
PIMC_HD void fx_box_muller(uint32_t x, uint32_t y, uint32_t z, uint32_t w, double& z0, double& z1)
{
    int F, f, fc, fs;
    const int64_t L = fx_neglog(fx_uniform(x, y), F);
    const int64_t r = fx_sqrt2(L, F, f);
    int64_t c, s;
    fx_sincos(fx_uniform(z, w), c, s, fc, fs);
    z0 = fx_double(fx_smul<true>(r, c), f + fc - 64);
    z1 = fx_double(fx_smul<true>(r, s), f + fs - 64);
}

// -log u from two words.
PIMC_HD double fx_neglog_uniform(uint32_t hi, uint32_t lo)
{
    int F;
    const int64_t L = fx_neglog(fx_uniform(hi, lo), F);
    return fx_double(L, F);
}

}  // namespace pimc
