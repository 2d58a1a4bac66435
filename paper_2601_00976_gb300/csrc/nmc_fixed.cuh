// Logarithm, exponential and linear interpolation in 64-bit fixed point, for the FP64 table
// interpolation (nmc_interp.cu).
//
// An FP64 instruction holds an SMSP's pipe ~64 cycles here, a 32-bit integer multiply-add a few, so a
// logarithm built from ~40 integer instructions is several times cheaper than one built from ~35 FP64
// ones.  The method is the table-driven reduction of Tang (ACM TOMS 15, 1989, exp; 16, 1990, log) with
// the polynomials evaluated in integers:
//   log2 m = -log2 c_i + log2(1 + r),  c_i ~ 1/m from the top 7 mantissa bits, r = m c_i - 1 < 2^-7 exact
//            in 64 bits, log2(1 + r) by the Taylor series to r^7 (coefficients 2^(-7 (n-1)) / (n ln 2));
//   2^f    = 2^(j/64) 2^(z/64),  z in [0, 1), 2^(z/64) by the Taylor series to z^6
//            (coefficients (ln 2 / 64)^n / n!).
// High-order terms take 32-bit products, whose rounding lies below the result's.  Qk: a fixed-point
// value with k fraction bits.  Errors, measured against 60-digit decimals over 2 x 10^4 arguments each:
// log2_q52 at most 2^-52.2 absolute (its last bit is 2^-52), exp_q53 at most 2^-52.3 relative.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace nmc {

// round-up 15-bit reciprocals of (128 + i) / 128 and -log2 of them (Q60); 2^(j/64) rounded down (Q63)
#define NMC_LOG_C \
    32768, 32514, 32264, 32018, 31776, 31537, 31301, 31069, 30841, 30616, 30394, 30175, 29960, 29747, 29538, 29331, \
    29128, 28927, 28729, 28533, 28340, 28150, 27963, 27777, 27595, 27414, 27236, 27061, 26887, 26716, 26547, 26380, \
    26215, 26052, 25891, 25732, 25576, 25421, 25267, 25116, 24967, 24819, 24673, 24529, 24386, 24245, 24106, 23968, \
    23832, 23697, 23564, 23432, 23302, 23173, 23046, 22920, 22796, 22672, 22551, 22430, 22311, 22193, 22076, 21960, \
    21846, 21733, 21621, 21510, 21400, 21291, 21184, 21077, 20972, 20868, 20764, 20662, 20561, 20461, 20361, 20263, \
    20165, 20069, 19973, 19879, 19785, 19692, 19600, 19509, 19419, 19329, 19240, 19153, 19066, 18979, 18894, 18809, \
    18725, 18642, 18559, 18478, 18397, 18316, 18237, 18158, 18079, 18002, 17925, 17849, 17773, 17698, 17624, 17550, \
    17477, 17404, 17332, 17261, 17190, 17120, 17051, 16981, 16913, 16845, 16778, 16711, 16645, 16579, 16514, 16449
#define NMC_LOG_L \
    0x0ull, 0x2dfbe8c3a5c9f0ull, 0x5b9894c5eaa7e2ull, 0x88d314bc93b24cull, 0xb5a8714bd7e670ull, 0xe245a30862bf1full, \
    0x10ea8b8033bc2f3ull, 0x13a9f062a91011full, 0x1662577cadaccaeull, 0x1916a59b80a2354ull, 0x1bc6b9d7c06b6fdull, 0x1e7272e1dcb45d5ull, \
    0x2116871ca2f5188ull, 0x23b91e7467aab32ull, 0x2653c0dd04dba21ull, 0x28ecac98e83b874ull, 0x2b7d51cdedacb2bull, 0x2e0c051d8c46953ull, \
    0x3095696fc797b6bull, 0x331caad559941c9ull, 0x359e600657cf1baull, 0x381a64275cf62b8ull, 0x3a90921377c45c4ull, 0x3d0793145a2855full, \
    0x3f751ca1cb3c62cull, 0x41e35024db98f1full, 0x444b3896ca5c852ull, 0x46acaf6b048763dull, 0x490e96434adc9b7ull, 0x4b69d4b4bc9999dull, \
    0x4dc1d33430af450ull, 0x50167b85b43f975ull, 0x5267b732226f7d5ull, 0x54b56f88451a836ull, 0x56ff8d9e0a32eacull, 0x5945fa51ce3d145ull, \
    0x5b84ebe7ce851b2ull, 0x5dc3a9d612ddf97ull, 0x60022daca5c5817ull, 0x6238e96295884c0ull, 0x646b7cfff4f171eull, 0x669d9f6d46e3849ull, \
    0x68cb747814170aeull, 0x6af4e371a90bf55ull, 0x6d1db40a1c795d2ull, 0x6f41f839e04b456ull, 0x716196cf5639f39ull, 0x7380684bd763448ull, \
    0x759a6cdac1a7df6ull, 0x77b38837ff27c4eull, 0x79c7aeb4d7c222cull, 0x7bdacf4d112166bull, 0x7de8d279d1f4dceull, 0x7ff5b27a3301a67ull, \
    0x81fd4bf3cf8baf1ull, 0x8403a46aa15b8c4ull, 0x86048cb80c26d48ull, 0x880841358c3d479ull, 0x8a023592b402770ull, 0x8bfee2c9ab511aeull, \
    0x8df5d690fbda2e3ull, 0x8feb3845697b749ull, 0x91defdd0ffaa8ebull, 0x93d11d02d43961dull, 0x95bd3793f1d62b1ull, 0x97a78b86644eab1ull, \
    0x99900e52617f91cull, 0x9b76b5567f9c8ebull, 0x9d5b75d7ef0c87cull, 0x9f3e4502b8d46fbull, 0xa11aa14eb954eeaull, 0xa2f967200d5fb41ull, \
    0xa4d1986156dda95ull, 0xa6a7a075ebcfe16ull, 0xa88001b8b2e0abbull, 0xaa519b3221a6e24ull, 0xac20e94f75b637bull, 0xadede07f8269898ull, \
    0xafbd19d7cafaa57ull, 0xb18545e52a6403full, 0xb34fa81d2a3c522ull, 0xb512d9c6d14e92cull, 0xb6d835497f32c40ull, 0xb8963cafb5b959aull, \
    0xba56614bb8690fbull, 0xbc13db1700b229bull, 0xbdce9dcc961871aull, 0xbf869d1639f3f55ull, 0xc13bcc8d0d10d42ull, 0xc2f303ed8469906ull, \
    0xc4a75e0325724dcull, 0xc653de69b4605dcull, 0xc802523b281fc7aull, 0xc9b2be08f80b48dull, 0xcb5b2431b3096e9ull, 0xcd05743b76dfc74ull, \
    0xceaca5ed6e86ec9ull, 0xd050ac4d739ae3eull, 0xd1f6927d01dd8b0ull, 0xd39420d6131fddcull, 0xd533804c22e7027ull, 0xd6d4b4fa01a1427ull, \
    0xd86d6475828abc1ull, 0xda07da23e21665cull, 0xdba419fb172fb72ull, 0xdd37a6c3c5f2a74ull, 0xdeccee614704ea6ull, 0xe05ea88943f6771ull, \
    0xe1f219861cf5ed7ull, 0xe381ed6e2c85ccaull, 0xe50e169a67816a0ull, 0xe69bea816759b2cull, 0xe82603c65f5e984ull, 0xe9b1c3556cee553ull, \
    0xeb39b82d157f25eull, 0xecbdd46b5d9bc97ull, 0xee438a30a58504aull, 0xefc55707237ab3bull, 0xf1432cf360d7297ull, 0xf2c820944bf271dull, \
    0xf443811f3eabc87ull, 0xf5c068eed572deeull, 0xf7393881b6d3f4cull, 0xf8b38a1000af685ull, 0xfa29b280d2cc451ull, 0xfba1577fe0f0fa6ull, \
    0xfd14c25a5b15c9full, 0xfe89a43254e3cdcull
#define NMC_EXP_T \
    0x8000000000000000ull, 0x8164d1f3bc030773ull, 0x82cd8698ac2ba1d7ull, 0x843a28c3acde4046ull, 0x85aac367cc487b14ull, 0x871f61969e8d1010ull, \
    0x88980e8092da8527ull, 0x8a14d575496efd9aull, 0x8b95c1e3ea8bd6e6ull, 0x8d1adf5b7e5ba9e5ull, 0x8ea4398b45cd53c0ull, 0x9031dc431466b1dcull, \
    0x91c3d373ab11c336ull, 0x935a2b2f13e6e92bull, 0x94f4efa8fef70961ull, 0x96942d3720185a00ull, 0x9837f0518db8a96full, 0x99e0459320b7fa64ull, \
    0x9b8d39b9d54e5538ull, 0x9d3ed9a72cffb750ull, 0x9ef5326091a111adull, 0xa0b0510fb9714fc2ull, 0xa27043030c496818ull, 0xa43515ae09e6809eull, \
    0xa5fed6a9b15138eaull, 0xa7cd93b4e9653569ull, 0xa9a15ab4ea7c0ef8ull, 0xab7a39b5a93ed337ull, 0xad583eea42a14ac6ull, 0xaf3b78ad690a4374ull, \
    0xb123f581d2ac258full, 0xb311c412a9112489ull, 0xb504f333f9de6484ull, 0xb6fd91e328d17791ull, 0xb8fbaf4762fb9ee9ull, 0xbaff5ab2133e45fbull, \
    0xbd08a39f580c36beull, 0xbf1799b67a731082ull, 0xc12c4cca66709456ull, 0xc346ccda24976407ull, 0xc5672a115506daddull, 0xc78d74c8abb9b15cull, \
    0xc9b9bd866e2f27a2ull, 0xcbec14fef2727c5cull, 0xce248c151f8480e3ull, 0xd06333daef2b2594ull, 0xd2a81d91f12ae45aull, 0xd4f35aabcfedfa1full, \
    0xd744fccad69d6af4ull, 0xd99d15c278afd7b5ull, 0xdbfbb797daf23755ull, 0xde60f4825e0e9123ull, 0xe0ccdeec2a94e111ull, 0xe33f8972be8a5a51ull, \
    0xe5b906e77c8348a8ull, 0xe8396a503c4bdc68ull, 0xeac0c6e7dd24392eull, 0xed4f301ed9942b84ull, 0xefe4b99bdcdaf5cbull, 0xf281773c59ffb139ull, \
    0xf5257d152486cc2cull, 0xf7d0df730ad13bb8ull, 0xfa83b2db722a033aull, 0xfd3e0c0cf486c174ull

struct FixedTables {
    uint64_t log_l[128];
    uint64_t exp_t[64];
    uint16_t log_c[128];
};

// Per-axis constants of a uniform log10 axis: x = log2(v) - lo, clamped to [0, span] (Q52), times the
// cells per octave a (a 2^-fb after the normalising shift zs).
struct FixedAxis {
    int64_t lo, span;
    uint64_t a;
    int zs, fb, n;
};

constexpr int64_t kLog2Inf = int64_t(1) << 62;   // log2_q52 of +infinity; its negative of zero, NaN and negatives
constexpr double kFixedMax = 500.0;              // |ln value| the fixed-point tables hold (Q53 in 64 bits)

__host__ __device__ __forceinline__ uint64_t mulhi_u64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

__host__ __device__ __forceinline__ uint32_t mulhi_u32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

__host__ __device__ __forceinline__ uint64_t word_of(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

// log2(x) as Q52; any double (see kLog2Inf)
__host__ __device__ __forceinline__ int64_t log2_q52(double x, const FixedTables& ft) {
    uint64_t u = word_of(x);
    int e = (int)(u >> 52) - 1023;   // a set sign bit makes it >= 1025
    if ((unsigned)(e + 1022) > 2045u) {   // zero, denormal, negative, infinite or NaN
        if (u == 0x7ff0000000000000ull) return kLog2Inf;
        if (!(x > 0.0)) return -kLog2Inf;
        u = word_of(x * 18014398509481984.0);   // 2^54
        e = (int)(u >> 52) - 1023 - 54;
    }
    const uint64_t m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
    const int i = (int)(m >> 45) & 127;
    const uint64_t z = (m * ft.log_c[i]) << 4;   // r 2^7 as Q64: the product's integer part falls off the top
    const uint32_t zh = (uint32_t)(z >> 32);
    uint32_t s = 0x1ec71u - mulhi_u32(zh, 0x34cu);                       // Q54
    s = 0x12776c5u - mulhi_u32(zh, s);
    s = 0xb8aa3b29u - mulhi_u32(zh, s);
    const uint64_t q3 = 0x1ec709dc3a040ull - (((uint64_t)zh * s) >> 22);   // Q64
    const uint64_t q2 = 0x171547652b82fe1ull - (((uint64_t)zh * (uint32_t)(q3 >> 17)) >> 15);
    const uint64_t q1 = 0xb8aa3b295c17f0bcull - (mulhi_u64(z, q2) >> 1);   // Q63
    return ((int64_t)e << 52) + (int64_t)((ft.log_l[i] + (mulhi_u64(z, q1) >> 10) + 128) >> 8);
}

// e^v for v as Q53, |v| <= 512: the double nearest to within an ulp
__device__ __forceinline__ double exp_q53(int64_t v, const FixedTables& ft) {
    const uint64_t w = (uint64_t)(v + 0x401db9a90b4f7777ll);   // + 740 ln 2: non-negative
    const uint64_t kL2e = 0xb8aa3b295c17f0bcull;               // log2 e, Q63
    const uint64_t h = mulhi_u64(w, kL2e), f = (h << 12) | ((w * kL2e) >> 52);   // w log2 e: h as Q52, fraction f as Q64
    const int k = (int)(h >> 52) - 740, j = (int)(f >> 58);
    const uint64_t z = f << 6;
    const uint32_t zh = (uint32_t)(z >> 32);
    uint32_t s = 0x576200u + mulhi_u32(zh, 0x2861u);                       // Q62
    s = 0x9d955b7eu + mulhi_u32(zh, s);
    const uint64_t q3 = 0x38d611ae094ull + (((uint64_t)zh * s) >> 30);    // Q64
    const uint64_t q2 = 0x3d7f7bff058b2ull + (((uint64_t)zh * (uint32_t)(q3 >> 10)) >> 22);
    const uint64_t q1 = 0x2c5c85fdf473de7ull + mulhi_u64(z, q2);
    const uint64_t t = ft.exp_t[j];
    const uint64_t r = t + mulhi_u64(t, mulhi_u64(z, q1));            // Q63, in [1, 2)
    const uint64_t m = (r >> 11) + ((r >> 10) & 1);
    return __longlong_as_double((long long)(((uint64_t)(int64_t)(k + 1022) << 52) + m));
}

// a + (b - a) t, t as Q63
__device__ __forceinline__ int64_t lerp_q(int64_t a, int64_t b, int64_t t) { return a + 2 * __mul64hi(b - a, t); }

}  // namespace nmc
