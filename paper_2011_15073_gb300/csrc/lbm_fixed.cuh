// lbm_fixed.cuh -- 64-bit fixed-point logarithm and exponential, and FP64
// reciprocal and square root, for a GPU whose FP64 pipe is slow.
//
// On this part one FP64 instruction of a warp holds a quarter SM's FP64 pipe
// for 64 cycles, however many of its lanes are active (measured), while the
// integer pipes take a warp instruction every cycle or two.  The library's
// pow() costs 96 FP64 instructions, an IEEE division 5 and a square root 9
// (measured).  Here the logarithm and the exponential run in fixed point,
// without FP64 instructions, and the reciprocal (3) and the square root (5)
// start from the special-function unit's approximation.
//
// Method (table-driven as in Tang, "Table-driven implementation of the
// logarithm function in IEEE floating-point arithmetic", ACM TOMS 16, 1990,
// carried out in fixed point):
//   x = 2^E m, 1 <= m < 2; an 11-bit c from the top seven bits of m
//   makes m c = 1 + z with 0 <= z < 2^-6.8, and the product is exact in 64 bits;
//   log2 x = E - log2 c + log2(1 + z), the last by its Taylor series;
//   2^y = 2^floor(y) 2^(j/64) 2^r with 0 <= r < 1/64, the last by its Taylor
//   series.
// Qn below means an integer holding the value times 2^n.  The logarithm is
// within 2^-56, the exponential within 0.53 units in the last place (against
// 80-bit arithmetic).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace lbm {

// High 64 bits of a 64 x 64-bit product, without the carry out of the low
// half: at most 2 below it.  Three wide multiplies instead of
// four, and no carry chain.
__host__ __device__ __forceinline__ uint64_t mulhi(uint64_t a, uint64_t b)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    return (uint64_t)ah * bh + ((uint64_t)ah * bl >> 32) + ((uint64_t)al * bh >> 32);
}
__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b)
{
    return (uint32_t)(((uint64_t)a * b) >> 32);
}

// {-log2(c / 2048) in Q57, c}, c = ceil(2048 / (1 + i / 128)).
struct LogEntry {
    unsigned long long t;
    unsigned c;
};
#define LBM_LOG_TABLE \
    {0x0000000000000000ull, 2048u}, {0x00056e1588a63197ull, 2033u}, {0x000b4430e855f27aull, 2017u}, {0x0010c7b844ef1795ull, 2002u}, \
    {0x0016b50e297afcceull, 1986u}, {0x001beec9151aac2eull, 1972u}, {0x002192a5da15c4ecull, 1957u}, {0x0027419ead40d895ull, 1942u}, \
    {0x002c99c4d80ce2adull, 1928u}, {0x0031fbe3951dd4d4ull, 1914u}, {0x003768205f24a728ull, 1900u}, {0x003cdea185b3eea8ull, 1886u}, \
    {0x0041fa91b28ff78aull, 1873u}, {0x00471f9df778cf6eull, 1860u}, {0x004c4de70b2f8870ull, 1847u}, {0x0051858e55ebc0b7ull, 1834u}, \
    {0x0056c6b5f668599bull, 1821u}, {0x005c1180c71e7e13ull, 1808u}, {0x0060fcc133716a9bull, 1796u}, {0x0065f072c4f1fb02ull, 1784u}, \
    {0x006aecb2a7b1d1caull, 1772u}, {0x006ff19e9fffd330ull, 1760u}, {0x0074ff550e92b572ull, 1748u}, {0x0079a90fb95cb380ull, 1737u}, \
    {0x007ec7f6c1d2efdbull, 1725u}, {0x008381a9149eb923ull, 1714u}, {0x0088432546743f30ull, 1703u}, {0x008d0c852eb3a503ull, 1692u}, \
    {0x0091dde3262f321bull, 1681u}, {0x0096b75a0a91927bull, 1670u}, {0x009b271288e64106ull, 1660u}, {0x00a0104b5f240f66ull, 1649u}, \
    {0x00a48e85c70377cfull, 1639u}, {0x00a913ca43f0a90cull, 1629u}, {0x00ada02f076a607cull, 1619u}, {0x00b233caac8a52d9ull, 1609u}, \
    {0x00b6ceb43aa75f41ull, 1599u}, {0x00bb7103280ce84eull, 1589u}, {0x00bfa3172c70b441ull, 1580u}, {0x00c453b5bf2a4e2dull, 1570u}, \
    {0x00c892d2eff0efccull, 1561u}, {0x00ccd83954b63593ull, 1552u}, {0x00d123fba540439aull, 1543u}, {0x00d5762ced6d6df0ull, 1534u}, \
    {0x00d9cee08f2ef08aull, 1525u}, {0x00de2e2a4492a65dull, 1516u}, {0x00e2941e21dc48d3ull, 1507u}, {0x00e700d097aec689ull, 1498u}, \
    {0x00eaf5626a31ebefull, 1490u}, {0x00eeef67c386260bull, 1482u}, {0x00f36f44b111098eull, 1473u}, {0x00f7751200c275f9ull, 1465u}, \
    {0x00fb8082e07c57f7ull, 1457u}, {0x00ff91a735abf046ull, 1449u}, {0x0103a88f29557b75ull, 1441u}, {0x0107c54b2995836cull, 1433u}, \
    {0x010be7ebeb2cfa18ull, 1425u}, {0x011010826b187a8full, 1417u}, {0x0113b8f7444275bbull, 1410u}, {0x0117ece9555fd721ull, 1402u}, \
    {0x011b9f698381225full, 1395u}, {0x011f56ac9ed9a8d2ull, 1388u}, {0x01239bb9203bcc33ull, 1380u}, {0x01275d59f70079abull, 1373u}, \
    {0x012b23e51b39c7b0ull, 1366u}, {0x012eef677ad6fcaeull, 1359u}, {0x0132bfee370ee686ull, 1352u}, {0x01369586a5706f2full, 1345u}, \
    {0x013a703e50fa4df3ull, 1338u}, {0x013e5022fb3a0e98ull, 1331u}, {0x014235429d72a9ddull, 1324u}, {0x014590247acce3c2ull, 1318u}, \
    {0x01497f209a9b0863ull, 1311u}, {0x014ce28bc4549be5ull, 1305u}, {0x0150db96d04eaa35ull, 1298u}, {0x015447b7266439aaull, 1292u}, \
    {0x0157b7eb8038faf3ull, 1286u}, {0x015bc007cc076f22ull, 1279u}, {0x015f3933dcb120a2ull, 1273u}, {0x0162b69356def7f4ull, 1267u}, \
    {0x01663830703da8d7ull, 1261u}, {0x0169be1583dfc0a4ull, 1255u}, {0x016d484d12f52cfaull, 1249u}, {0x0170d6e1c5872d9bull, 1243u}, \
    {0x017469de6b38d25dull, 1237u}, {0x0178014dfc0c271full, 1231u}, {0x017b9d3b992c30e3ull, 1225u}, {0x017ea2a2ed97cce2ull, 1220u}, \
    {0x018246ea6a6006abull, 1214u}, {0x0185535771691f09ull, 1209u}, {0x0189001fcdbed999ull, 1203u}, {0x018c13b3791cefffull, 1198u}, \
    {0x018fc924c89ac847ull, 1192u}, {0x0192e400f3ff2f96ull, 1187u}, {0x0196a244683409e2ull, 1181u}, {0x0199c48be2063c84ull, 1176u}, \
    {0x019cea3e7366be59ull, 1171u}, {0x01a0136399883a4cull, 1166u}, {0x01a3e2f4ac43f603ull, 1160u}, {0x01a713ca57071aeaull, 1155u}, \
    {0x01aa482b35ca9cebull, 1150u}, {0x01ad801f307aa07bull, 1145u}, {0x01b0bbae4995d670ull, 1140u}, {0x01b3fae09ea5172cull, 1135u}, \
    {0x01b73dbe68b5a1bbull, 1130u}, {0x01b9dc4d0b8ba507ull, 1126u}, {0x01bd25daeddc5a84ull, 1121u}, {0x01c0732be1e9feb7ull, 1116u}, \
    {0x01c3c4488dde1ffaull, 1111u}, {0x01c66e54373091e0ull, 1107u}, {0x01c9c65c26a33233ull, 1102u}, {0x01cd2248a6c7353bull, 1097u}, \
    {0x01cfd50cb182f873ull, 1093u}, {0x01d338120a6dd9d3ull, 1088u}, {0x01d5f08f93f98892ull, 1084u}, {0x01d95acc02d690a2ull, 1079u}, \
    {0x01dc191b896a324bull, 1075u}, {0x01df8aae0e46f567ull, 1070u}, {0x01e24ee8ae9f0c50ull, 1066u}, {0x01e515cce9f6a08eull, 1062u}, \
    {0x01e7df5fe538ab35ull, 1058u}, {0x01eb5f254ba8bf06ull, 1053u}, {0x01ee2ed49397813aull, 1049u}, {0x01f10143bbf63308ull, 1045u}, \
    {0x01f3d6782ae1fbc3ull, 1041u}, {0x01f6ae77566e830dull, 1037u}, {0x01f98946c4e51d34ull, 1033u}, {0x01fc66ec0d05314eull, 1029u}
// 2^(j / 64) in Q63.
#define LBM_EXP_TABLE \
    0x8000000000000000ull, 0x8164d1f3bc030773ull, 0x82cd8698ac2ba1d7ull, 0x843a28c3acde4046ull, \
    0x85aac367cc487b15ull, 0x871f61969e8d1010ull, 0x88980e8092da8527ull, 0x8a14d575496efd9aull, \
    0x8b95c1e3ea8bd6e7ull, 0x8d1adf5b7e5ba9e6ull, 0x8ea4398b45cd53c0ull, 0x9031dc431466b1dcull, \
    0x91c3d373ab11c336ull, 0x935a2b2f13e6e92cull, 0x94f4efa8fef70961ull, 0x96942d3720185a00ull, \
    0x9837f0518db8a96full, 0x99e0459320b7fa65ull, 0x9b8d39b9d54e5539ull, 0x9d3ed9a72cffb751ull, \
    0x9ef5326091a111aeull, 0xa0b0510fb9714fc2ull, 0xa27043030c496819ull, 0xa43515ae09e6809eull, \
    0xa5fed6a9b15138eaull, 0xa7cd93b4e965356aull, 0xa9a15ab4ea7c0ef8ull, 0xab7a39b5a93ed337ull, \
    0xad583eea42a14ac6ull, 0xaf3b78ad690a4375ull, 0xb123f581d2ac2590ull, 0xb311c412a9112489ull, \
    0xb504f333f9de6484ull, 0xb6fd91e328d17791ull, 0xb8fbaf4762fb9ee9ull, 0xbaff5ab2133e45fbull, \
    0xbd08a39f580c36bfull, 0xbf1799b67a731083ull, 0xc12c4cca66709456ull, 0xc346ccda24976407ull, \
    0xc5672a115506daddull, 0xc78d74c8abb9b15dull, 0xc9b9bd866e2f27a3ull, 0xcbec14fef2727c5dull, \
    0xce248c151f8480e4ull, 0xd06333daef2b2595ull, 0xd2a81d91f12ae45aull, 0xd4f35aabcfedfa1full, \
    0xd744fccad69d6af4ull, 0xd99d15c278afd7b6ull, 0xdbfbb797daf23755ull, 0xde60f4825e0e9124ull, \
    0xe0ccdeec2a94e111ull, 0xe33f8972be8a5a51ull, 0xe5b906e77c8348a8ull, 0xe8396a503c4bdc68ull, \
    0xeac0c6e7dd24392full, 0xed4f301ed9942b84ull, 0xefe4b99bdcdaf5cbull, 0xf281773c59ffb13aull, \
    0xf5257d152486cc2cull, 0xf7d0df730ad13bb9ull, 0xfa83b2db722a033aull, 0xfd3e0c0cf486c175ull

#ifdef __CUDA_ARCH__
static __device__ const LogEntry kLog2Table[128] = {LBM_LOG_TABLE};
static __device__ const unsigned long long kExp2Table[64] = {LBM_EXP_TABLE};
#else
static const LogEntry kLog2Table[128] = {LBM_LOG_TABLE};
static const unsigned long long kExp2Table[64] = {LBM_EXP_TABLE};
#endif

// log2 of the mantissa of x (normal, positive) in Q57.
__host__ __device__ __forceinline__ int64_t log2_mantissa_q57(uint64_t bits)
{
    const LogEntry t = kLog2Table[(bits >> 45) & 127];
    const uint64_t m = (bits & 0xfffffffffffffull) | (1ull << 52);
    // z in Q63 exactly; z' = 32 z in Q64 (below 0.28)
    const uint64_t z = (m * t.c - (1ull << 63)) << 6;
    const uint32_t z32 = (uint32_t)(z >> 32);
    // sum over k of (-1)^(k-1) C_k z'^(k-1), C_k = 1 / (k ln 2 32^k): the
    // terms from k = 4 in Q53 on 32 bits, the first three in Q64
    uint32_t v = 2017034u - mulhi32(54028u, z32);
    v = 77454100u - mulhi32(v, z32);
    v = 3098164009u - mulhi32(v, z32);
    uint64_t u = 0x0000f6384ee1d020ull - mulhi(z, (uint64_t)v << 11);
    u = 0x002e2a8eca5705fcull - mulhi(z, u);
    u = 0x0b8aa3b295c17f0cull - mulhi(z, u);
    return (int64_t)t.t + (int64_t)(mulhi(z, u) >> 7);
}
// log2 sqrt(x) in Q57, 2^-126 <= x < 2^126.
__host__ __device__ __forceinline__ int64_t log2_sqrt_q57(uint64_t bits)
{
    return ((int64_t)((int)(bits >> 52) - 1023) << 56) + (log2_mantissa_q57(bits) >> 1);
}

// 2^(p / 2^56) as a double.
__host__ __device__ __forceinline__ double exp2_q56(int64_t p)
{
    const int k = (int)(p >> 56);
    const uint64_t f = (uint64_t)p << 8;
    const uint64_t s = kExp2Table[f >> 58];
    // r' = 64 r in Q64; sum over k of D_k r'^k, D_k = ln2^k / (k! 64^k): the
    // terms from k = 4 in Q60 on 32 bits, the first three in Q64
    const uint64_t r = f << 6;
    const uint32_t r32 = (uint32_t)(r >> 32);
    uint32_t v = 1431680u + mulhi32(2584u + mulhi32(4u, r32), r32);
    v = 660952799u + mulhi32(v, r32);
    uint64_t u = 0x0000038d611ae094ull + mulhi(r, (uint64_t)v << 4);
    u = 0x0003d7f7bff058b2ull + mulhi(r, u);
    u = 0x02c5c85fdf473de7ull + mulhi(r, u);
    uint64_t w = s + mulhi(s, mulhi(r, u));   // Q63, 1 <= w < 2
    if (w < s) w = ~0ull;                     // just below 2, rounded over it
    const uint64_t bits = ((uint64_t)(int64_t)(k + 1022) << 52) + (w >> 11) + (w >> 10 & 1);
    double d;
    memcpy(&d, &bits, 8);
    return d;
}

#ifdef __CUDACC__
// 1 / x, x normal with a normal reciprocal: two orders beyond the 2^-23 of
// the approximation in one step (y (1 + e + e^2), e = 1 - x y).  0 and the
// infinities give NaN.
__device__ __forceinline__ double rcp_f64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// sqrt(x), x >= 0; 0 below the normal range.  Two Newton steps on the root
// s = x y with the approximate 1 / (2 sqrt x) as their slope.
__device__ __forceinline__ double sqrt_f64(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double s = x * y;
    // y / 2 by its exponent
    const double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
    const double s1 = fma(fma(-s, s, x), h, s);
    const double r = fma(fma(-s1, s1, x), h, s1);
    return __double2hiint(x) < 0x00100000 && __double2hiint(x) >= 0 ? 0.0 : r;
}
#endif

}  // namespace lbm
