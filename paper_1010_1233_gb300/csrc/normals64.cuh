// FP64 unit normals in 64-bit fixed-point arithmetic.
//
// GB300 executes 2 FP64 instructions per clock and SM, 1/64 of its integer rate, and the
// FP64 step kernels are bound by that pipe.  A Box-Muller pair through log, sqrt and sincospi
// is about 100 FP64 instructions, two thirds of a D2Q9 or D3Q15 site update.  Its inputs are
// integers, u = (w + 1/2) 2^-32 exactly, so the whole transform runs here in integer
// multiply-adds instead (about 300 instructions of the wide pipes and none of FP64) and only
// the two results are written as doubles.
//
// N0 = r cos(2 pi ub), N1 = r sin(2 pi ub), r = sqrt(-2 ln ua).  Qk: an integer in units of 2^-k.
//   ln:  ua = x 2^-33, x = 2 wa + 1 = 2^e m, m in [1, 2) exact in Q32.  Table-driven reduction
//        (Tang, ACM TOMS 16, 1990): c ~ 1/m to 9 bits by the top 7 fraction bits of m, z = m c - 1
//        exactly, |z| < 2^-7.7, -ln ua = (33 - e) ln 2 + ln c - ln(1 + z), the last by its Taylor
//        series to z^7 (z^8 / 8 < 2^-64); result in Q59, or in Q63 for ua >= 1/2, where it can be
//        small.  The last entry is c = 1/2 exactly, so that for ua >= 1 - 2^-8 the first two terms
//        cancel and z = -(1 - ua) is all of the argument: it keeps its leading zeros apart (an even
//        number of them), and the result has 61 significant bits however small it is.
//   sqrt: a 23-bit reciprocal root y of the mantissa v, h = v y, e = 1 - h y, sqrt v = h / sqrt(1 - e)
//        by its binomial series to e^2 (5/16 e^3 < 2^-61).
//   sin, cos: 256 table angles (i + 1/2) 2 pi / 256 by the top 8 bits of ub, the remainder
//        |delta| <= pi / 256 by Taylor series (errors below 2^-66) and the addition theorems.
// The result is the product of two fixed-point numbers and a power of two, so its error goes with r: at
// most 1.2e-16 r for every scale of 1 - ua down to 2^-33 (2.9e-16 r with FP64 log and sqrt and correctly
// rounded sine and cosine); where the sine or cosine is small it stays below 2^-60 r, but not below the
// last bit of the product.  The root-mean-square error of 3 10^6 random pairs is 4.7e-17, that of the
// final rounding (8.1e-17).
#pragma once
#include <cstdint>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define FLB_HD __host__ __device__ __forceinline__
#define FLB_TAB static __device__ const
#else
#define FLB_HD static inline
#define FLB_TAB static const
#endif

namespace flb {

struct alignas(16) Fx2 { uint64_t a, b; };

// by the top 7 fraction bits of m: c = round(2^9 / (1 + (i + 1/2) / 128)), the last 2^8, and -ln(c / 512) in Q63
FLB_TAB Fx2 kFxLog[128] = {
  {510, 0x0080402acac459acull}, {506, 0x0182448a388a2aa2ull}, {502, 0x02865524b3019814ull},
  {498, 0x038c7a5d82955e32ull}, {495, 0x045278f90016a33bull}, {491, 0x055c571300f3bbb9ull},
  {487, 0x066861ed5cf79ee9ull}, {484, 0x0732dcf3776cb2e2ull}, {480, 0x0842cc5acf1d0344ull},
  {477, 0x09103dae3c2a4ec6ull}, {473, 0x0a242f01edefd6a3ull}, {470, 0x0af4ad26cbc8e5beull},
  {466, 0x0c0cbf17a071f80eull}, {463, 0x0ce06196a692a420ull}, {460, 0x0db56446d6ad8df0ull},
  {457, 0x0e8bcbc410c9b21aull}, {454, 0x0f639cc185088fe6ull}, {450, 0x108598b59e3a0689ull},
  {447, 0x1160c8024b27b0b5ull}, {444, 0x123d712a49c201a4ull}, {441, 0x131b994d3a4f84c7ull},
  {438, 0x13fb45a59928cb8aull}, {435, 0x14dc7b897bc1c79bull}, {433, 0x15737cc9018cdd54ull},
  {430, 0x16574ebe8c1339f1ull}, {427, 0x173cb9074fd14cabull}, {424, 0x1823c16551a3c1bbull},
  {421, 0x190c6db9fcbcd941ull}, {419, 0x19a8778debaa387dull}, {416, 0x1a93ed3c8ad9e36full},
  {413, 0x1b811730b823d20dull}, {411, 0x1c2028ab17f9b47cull}, {408, 0x1d1037f2655e7b58ull},
  {406, 0x1db13db0d4894035ull}, {403, 0x1ea4449f04aaf48bull}, {401, 0x1f474b134df228dbull},
  {398, 0x203d5cac4d8d21eeull}, {396, 0x20e270c09ab0c4e7ull}, {394, 0x21885acec2c5c623ull},
  {391, 0x2282cfde6cef0604ull}, {389, 0x232ada773785f4beull}, {387, 0x23d3c2cf1133e8a9ull},
  {384, 0x24d2c42269b724f0ull}, {382, 0x257de0f9b926a73full}, {380, 0x2629e3c3a6b9c761ull},
  {378, 0x26d6ceed7c222ddaull}, {376, 0x2784a4ee6663076bull}, {373, 0x288b23c0a73e916aull},
  {371, 0x293b4fe779883d9aull}, {369, 0x29ec6fd775301f54ull}, {367, 0x2a9e8636f7c3512bull},
  {365, 0x2b5195b77dbf41c3ull}, {363, 0x2c05a115e123d7d2ull}, {361, 0x2cbaab1a99c01545ull},
  {359, 0x2d70b699ff47f99dull}, {357, 0x2e27c6748d42f736ull}, {355, 0x2edfdd9728e2e977ull},
  {353, 0x2f98fefb68d41b3eull}, {351, 0x30532da7df17956bull}, {350, 0x30b0aaeedb97f55cull},
  {348, 0x316c7351165be948ull}, {346, 0x322950c6b7ed1329ull}, {344, 0x32e7468626ad5b9eull},
  {342, 0x33a657d42bda7618ull}, {340, 0x3466880449f4f191ull}, {339, 0x34c70cbf57a1d7bbull},
  {337, 0x3588f1a040a0de07ull}, {335, 0x364bfdf6c1965c18ull}, {334, 0x36adf4088c5212a5ull},
  {332, 0x3772c23701c5f617ull}, {330, 0x3838c0d27f473b20ull}, {329, 0x389c33708e478349ull},
  {327, 0x396401a59d6c85cfull}, {325, 0x3a2d09a93e8d5cedull}, {324, 0x3a92048dbdf4d6ecull},
  {322, 0x3b5cea90992c2b7aull}, {320, 0x3c2914344e4d9b2aull}, {319, 0x3c8fa3a65ccefc33ull},
  {317, 0x3d5dba5d59321867ull}, {316, 0x3dc542ad6827c9fdull}, {314, 0x3e954fdc063259bdull},
  {313, 0x3efdd5cd6aec3980ull}, {311, 0x3fcfe31d607a7c2cull}, {310, 0x40396b96c81eac46ull},
  {308, 0x410d82f9d80eb3baull}, {307, 0x41781306a8b0180cull}, {306, 0x41e2fc14cf15a049ull},
  {304, 0x42b9db8b4153e90dull}, {303, 0x4325d32250c73703ull}, {301, 0x43fed5084e91d77cull},
  {300, 0x446be08f1d6a9e6eull}, {299, 0x44d9494afc21930bull}, {297, 0x45b534e30467e9d7ull},
  {296, 0x4623b903c8f2998aull}, {295, 0x46929ce2de8cf159ull}, {293, 0x4771867781a5106dull},
  {292, 0x47e18d7f1859636full}, {291, 0x4851f6e91e8e4eacull}, {289, 0x4933f39be03669a5ull},
  {288, 0x49a58844d36e49e1ull}, {287, 0x4a178210b28e0e27ull}, {286, 0x4a89e1b43b041b4bull},
  {284, 0x4b6fd55ec37d0b23ull}, {283, 0x4be36ad8d8cde668ull}, {282, 0x4c576910d01a2c5bull},
  {281, 0x4ccbd0c52b5e5694ull}, {279, 0x4db5dfa74d3f5afdull}, {278, 0x4e2b885c65db9d21ull},
  {277, 0x4ea19d9c95c444b8ull}, {276, 0x4f182030dafed48dull}, {275, 0x4f8f10e463ddb159ull},
  {274, 0x50067084972a4c62ull}, {272, 0x50f67fcbe48f133eull}, {271, 0x516f31193224e851ull},
  {270, 0x51e8549fa28b4d25ull}, {269, 0x5261eb3836aec1f7ull}, {268, 0x52dbf5be5c307dc4ull},
  {267, 0x5356750ff6ae87b3ull}, {266, 0x53d16a0d693864ecull}, {265, 0x544cd5999ff15ce5ull},
  {264, 0x54c8b89a19e15cccull}, {263, 0x554513f6f2f589d6ull}, {262, 0x55c1e89aee319981ull},
  {261, 0x563f377380130e38ull}, {260, 0x56bd0170d9277e99ull}, {259, 0x573b4785f0d71568ull},
  {258, 0x57ba0aa89064808eull}, {256, 0x58b90bfbe8e7bcd6ull},
};

// cos and sin of 2 pi (i + 1/2) / 256 in Q62 (two's complement)
FLB_TAB Fx2 kFxTrig[256] = {
  {0x3ffec42d3725b6afull, 0x00c90e8fe6f63c23ull}, {0x3ff4e5dffdeeb93aull, 0x025b0caeb28ab9a3ull},
  {0x3fe12acb1ce35a81ull, 0x03ecadcf3f041bfeull}, {0x3fc395f97ab61234ull, 0x057db402a6a90630ull},
  {0x3f9c2bfadb4cf5a9ull, 0x070de171e7b0b53dull}, {0x3f6af2e32bae8247ull, 0x089cf8676d7abb56ull},
  {0x3f2ff2499213350full, 0x0a2abb58949f2cedull}, {0x3eeb33474240eec2ull, 0x0bb6ecef285f98a4ull},
  {0x3e9cc076165e599cull, 0x0d415012d802284full}, {0x3e44a5eeec75b370ull, 0x0ec9a7f2a2a188afull},
  {0x3de2f147c8e784b2ull, 0x104fb80e37fdadffull}, {0x3d77b191be16e872ull, 0x11d3443f4cdb3dd2ull},
  {0x3d02f75699a2198cull, 0x135410c2e18151b1ull}, {0x3c84d4965782fcd4ull, 0x14d1e24278e76a25ull},
  {0x3bfd5cc45b7c5557ull, 0x164c7ddd3f27c611ull}, {0x3b6ca4c471413595ull, 0x17c3a9311dcce702ull},
  {0x3ad2c2e793cd1586ull, 0x19372a63bc93d72dull}, {0x3a2fcee87c6bb7efull, 0x1aa6c82b6d3fc98bull},
  {0x3983e1e7f9f8b879ull, 0x1c1249d8011ee6a0ull}, {0x38cf166910e7363bull, 0x1d79775b86e38955ull},
  {0x3811884ce4aa921bull, 0x1edc1952ef78d589ull}, {0x374b54ce6b21a4bfull, 0x2039f90e987d6db3ull},
  {0x367c9a7deaae230aull, 0x2192e09abb131d39ull}, {0x35a5793c43aa215cull, 0x22e69ac7bdb69141ull},
  {0x34c6123605f5c386ull, 0x2434f33267d6b163ull}, {0x33de87de535f286cull, 0x257db64bf5e7d3efull},
  {0x32eefde98fae8375ull, 0x26c0b1620cb3e570ull}, {0x31f79947df2819d2ull, 0x27fdb2a68aada89bull},
  {0x30f8801f745d7d69ull, 0x293489373612716cull}, {0x2ff1d9c6ae2ee132ull, 0x2a65052546ab2b98ull},
  {0x2ee3cebe06e4c257ull, 0x2b8ef77cca031883ull}, {0x2dce88a9d5515d12ull, 0x2cb2324be0f07ae2ull},
  {0x2cb2324be0f07ae2ull, 0x2dce88a9d5515d12ull}, {0x2b8ef77cca031883ull, 0x2ee3cebe06e4c257ull},
  {0x2a65052546ab2b98ull, 0x2ff1d9c6ae2ee132ull}, {0x293489373612716cull, 0x30f8801f745d7d69ull},
  {0x27fdb2a68aada89bull, 0x31f79947df2819d2ull}, {0x26c0b1620cb3e570ull, 0x32eefde98fae8375ull},
  {0x257db64bf5e7d3efull, 0x33de87de535f286cull}, {0x2434f33267d6b163ull, 0x34c6123605f5c386ull},
  {0x22e69ac7bdb69141ull, 0x35a5793c43aa215cull}, {0x2192e09abb131d39ull, 0x367c9a7deaae230aull},
  {0x2039f90e987d6db3ull, 0x374b54ce6b21a4bfull}, {0x1edc1952ef78d589ull, 0x3811884ce4aa921bull},
  {0x1d79775b86e38955ull, 0x38cf166910e7363bull}, {0x1c1249d8011ee6a0ull, 0x3983e1e7f9f8b879ull},
  {0x1aa6c82b6d3fc98bull, 0x3a2fcee87c6bb7efull}, {0x19372a63bc93d72dull, 0x3ad2c2e793cd1586ull},
  {0x17c3a9311dcce702ull, 0x3b6ca4c471413595ull}, {0x164c7ddd3f27c611ull, 0x3bfd5cc45b7c5557ull},
  {0x14d1e24278e76a25ull, 0x3c84d4965782fcd4ull}, {0x135410c2e18151b1ull, 0x3d02f75699a2198cull},
  {0x11d3443f4cdb3dd2ull, 0x3d77b191be16e872ull}, {0x104fb80e37fdadffull, 0x3de2f147c8e784b2ull},
  {0x0ec9a7f2a2a188afull, 0x3e44a5eeec75b370ull}, {0x0d415012d802284full, 0x3e9cc076165e599cull},
  {0x0bb6ecef285f98a4ull, 0x3eeb33474240eec2ull}, {0x0a2abb58949f2cedull, 0x3f2ff2499213350full},
  {0x089cf8676d7abb56ull, 0x3f6af2e32bae8247ull}, {0x070de171e7b0b53dull, 0x3f9c2bfadb4cf5a9ull},
  {0x057db402a6a90630ull, 0x3fc395f97ab61234ull}, {0x03ecadcf3f041bfeull, 0x3fe12acb1ce35a81ull},
  {0x025b0caeb28ab9a3ull, 0x3ff4e5dffdeeb93aull}, {0x00c90e8fe6f63c23ull, 0x3ffec42d3725b6afull},
  {0xff36f1701909c3ddull, 0x3ffec42d3725b6afull}, {0xfda4f3514d75465dull, 0x3ff4e5dffdeeb93aull},
  {0xfc135230c0fbe402ull, 0x3fe12acb1ce35a81ull}, {0xfa824bfd5956f9d0ull, 0x3fc395f97ab61234ull},
  {0xf8f21e8e184f4ac3ull, 0x3f9c2bfadb4cf5a9ull}, {0xf7630798928544aaull, 0x3f6af2e32bae8247ull},
  {0xf5d544a76b60d313ull, 0x3f2ff2499213350full}, {0xf4491310d7a0675cull, 0x3eeb33474240eec2ull},
  {0xf2beafed27fdd7b1ull, 0x3e9cc076165e599cull}, {0xf136580d5d5e7751ull, 0x3e44a5eeec75b370ull},
  {0xefb047f1c8025201ull, 0x3de2f147c8e784b2ull}, {0xee2cbbc0b324c22eull, 0x3d77b191be16e872ull},
  {0xecabef3d1e7eae4full, 0x3d02f75699a2198cull}, {0xeb2e1dbd871895dbull, 0x3c84d4965782fcd4ull},
  {0xe9b38222c0d839efull, 0x3bfd5cc45b7c5557ull}, {0xe83c56cee23318feull, 0x3b6ca4c471413595ull},
  {0xe6c8d59c436c28d3ull, 0x3ad2c2e793cd1586ull}, {0xe55937d492c03675ull, 0x3a2fcee87c6bb7efull},
  {0xe3edb627fee11960ull, 0x3983e1e7f9f8b879ull}, {0xe28688a4791c76abull, 0x38cf166910e7363bull},
  {0xe123e6ad10872a77ull, 0x3811884ce4aa921bull}, {0xdfc606f16782924dull, 0x374b54ce6b21a4bfull},
  {0xde6d1f6544ece2c7ull, 0x367c9a7deaae230aull}, {0xdd19653842496ebfull, 0x35a5793c43aa215cull},
  {0xdbcb0ccd98294e9dull, 0x34c6123605f5c386ull}, {0xda8249b40a182c11ull, 0x33de87de535f286cull},
  {0xd93f4e9df34c1a90ull, 0x32eefde98fae8375ull}, {0xd8024d5975525765ull, 0x31f79947df2819d2ull},
  {0xd6cb76c8c9ed8e94ull, 0x30f8801f745d7d69ull}, {0xd59afadab954d468ull, 0x2ff1d9c6ae2ee132ull},
  {0xd471088335fce77dull, 0x2ee3cebe06e4c257ull}, {0xd34dcdb41f0f851eull, 0x2dce88a9d5515d12ull},
  {0xd23177562aaea2eeull, 0x2cb2324be0f07ae2ull}, {0xd11c3141f91b3da9ull, 0x2b8ef77cca031883ull},
  {0xd00e263951d11eceull, 0x2a65052546ab2b98ull}, {0xcf077fe08ba28297ull, 0x293489373612716cull},
  {0xce0866b820d7e62eull, 0x27fdb2a68aada89bull}, {0xcd11021670517c8bull, 0x26c0b1620cb3e570ull},
  {0xcc217821aca0d794ull, 0x257db64bf5e7d3efull}, {0xcb39edc9fa0a3c7aull, 0x2434f33267d6b163ull},
  {0xca5a86c3bc55dea4ull, 0x22e69ac7bdb69141ull}, {0xc98365821551dcf6ull, 0x2192e09abb131d39ull},
  {0xc8b4ab3194de5b41ull, 0x2039f90e987d6db3ull}, {0xc7ee77b31b556de5ull, 0x1edc1952ef78d589ull},
  {0xc730e996ef18c9c5ull, 0x1d79775b86e38955ull}, {0xc67c1e1806074787ull, 0x1c1249d8011ee6a0ull},
  {0xc5d0311783944811ull, 0x1aa6c82b6d3fc98bull}, {0xc52d3d186c32ea7aull, 0x19372a63bc93d72dull},
  {0xc4935b3b8ebeca6bull, 0x17c3a9311dcce702ull}, {0xc402a33ba483aaa9ull, 0x164c7ddd3f27c611ull},
  {0xc37b2b69a87d032cull, 0x14d1e24278e76a25ull}, {0xc2fd08a9665de674ull, 0x135410c2e18151b1ull},
  {0xc2884e6e41e9178eull, 0x11d3443f4cdb3dd2ull}, {0xc21d0eb837187b4eull, 0x104fb80e37fdadffull},
  {0xc1bb5a11138a4c90ull, 0x0ec9a7f2a2a188afull}, {0xc1633f89e9a1a664ull, 0x0d415012d802284full},
  {0xc114ccb8bdbf113eull, 0x0bb6ecef285f98a4ull}, {0xc0d00db66deccaf1ull, 0x0a2abb58949f2cedull},
  {0xc0950d1cd4517db9ull, 0x089cf8676d7abb56ull}, {0xc063d40524b30a57ull, 0x070de171e7b0b53dull},
  {0xc03c6a068549edccull, 0x057db402a6a90630ull}, {0xc01ed534e31ca57full, 0x03ecadcf3f041bfeull},
  {0xc00b1a20021146c6ull, 0x025b0caeb28ab9a3ull}, {0xc0013bd2c8da4951ull, 0x00c90e8fe6f63c23ull},
  {0xc0013bd2c8da4951ull, 0xff36f1701909c3ddull}, {0xc00b1a20021146c6ull, 0xfda4f3514d75465dull},
  {0xc01ed534e31ca57full, 0xfc135230c0fbe402ull}, {0xc03c6a068549edccull, 0xfa824bfd5956f9d0ull},
  {0xc063d40524b30a57ull, 0xf8f21e8e184f4ac3ull}, {0xc0950d1cd4517db9ull, 0xf7630798928544aaull},
  {0xc0d00db66deccaf1ull, 0xf5d544a76b60d313ull}, {0xc114ccb8bdbf113eull, 0xf4491310d7a0675cull},
  {0xc1633f89e9a1a664ull, 0xf2beafed27fdd7b1ull}, {0xc1bb5a11138a4c90ull, 0xf136580d5d5e7751ull},
  {0xc21d0eb837187b4eull, 0xefb047f1c8025201ull}, {0xc2884e6e41e9178eull, 0xee2cbbc0b324c22eull},
  {0xc2fd08a9665de674ull, 0xecabef3d1e7eae4full}, {0xc37b2b69a87d032cull, 0xeb2e1dbd871895dbull},
  {0xc402a33ba483aaa9ull, 0xe9b38222c0d839efull}, {0xc4935b3b8ebeca6bull, 0xe83c56cee23318feull},
  {0xc52d3d186c32ea7aull, 0xe6c8d59c436c28d3ull}, {0xc5d0311783944811ull, 0xe55937d492c03675ull},
  {0xc67c1e1806074787ull, 0xe3edb627fee11960ull}, {0xc730e996ef18c9c5ull, 0xe28688a4791c76abull},
  {0xc7ee77b31b556de5ull, 0xe123e6ad10872a77ull}, {0xc8b4ab3194de5b41ull, 0xdfc606f16782924dull},
  {0xc98365821551dcf6ull, 0xde6d1f6544ece2c7ull}, {0xca5a86c3bc55dea4ull, 0xdd19653842496ebfull},
  {0xcb39edc9fa0a3c7aull, 0xdbcb0ccd98294e9dull}, {0xcc217821aca0d794ull, 0xda8249b40a182c11ull},
  {0xcd11021670517c8bull, 0xd93f4e9df34c1a90ull}, {0xce0866b820d7e62eull, 0xd8024d5975525765ull},
  {0xcf077fe08ba28297ull, 0xd6cb76c8c9ed8e94ull}, {0xd00e263951d11eceull, 0xd59afadab954d468ull},
  {0xd11c3141f91b3da9ull, 0xd471088335fce77dull}, {0xd23177562aaea2eeull, 0xd34dcdb41f0f851eull},
  {0xd34dcdb41f0f851eull, 0xd23177562aaea2eeull}, {0xd471088335fce77dull, 0xd11c3141f91b3da9ull},
  {0xd59afadab954d468ull, 0xd00e263951d11eceull}, {0xd6cb76c8c9ed8e94ull, 0xcf077fe08ba28297ull},
  {0xd8024d5975525765ull, 0xce0866b820d7e62eull}, {0xd93f4e9df34c1a90ull, 0xcd11021670517c8bull},
  {0xda8249b40a182c11ull, 0xcc217821aca0d794ull}, {0xdbcb0ccd98294e9dull, 0xcb39edc9fa0a3c7aull},
  {0xdd19653842496ebfull, 0xca5a86c3bc55dea4ull}, {0xde6d1f6544ece2c7ull, 0xc98365821551dcf6ull},
  {0xdfc606f16782924dull, 0xc8b4ab3194de5b41ull}, {0xe123e6ad10872a77ull, 0xc7ee77b31b556de5ull},
  {0xe28688a4791c76abull, 0xc730e996ef18c9c5ull}, {0xe3edb627fee11960ull, 0xc67c1e1806074787ull},
  {0xe55937d492c03675ull, 0xc5d0311783944811ull}, {0xe6c8d59c436c28d3ull, 0xc52d3d186c32ea7aull},
  {0xe83c56cee23318feull, 0xc4935b3b8ebeca6bull}, {0xe9b38222c0d839efull, 0xc402a33ba483aaa9ull},
  {0xeb2e1dbd871895dbull, 0xc37b2b69a87d032cull}, {0xecabef3d1e7eae4full, 0xc2fd08a9665de674ull},
  {0xee2cbbc0b324c22eull, 0xc2884e6e41e9178eull}, {0xefb047f1c8025201ull, 0xc21d0eb837187b4eull},
  {0xf136580d5d5e7751ull, 0xc1bb5a11138a4c90ull}, {0xf2beafed27fdd7b1ull, 0xc1633f89e9a1a664ull},
  {0xf4491310d7a0675cull, 0xc114ccb8bdbf113eull}, {0xf5d544a76b60d313ull, 0xc0d00db66deccaf1ull},
  {0xf7630798928544aaull, 0xc0950d1cd4517db9ull}, {0xf8f21e8e184f4ac3ull, 0xc063d40524b30a57ull},
  {0xfa824bfd5956f9d0ull, 0xc03c6a068549edccull}, {0xfc135230c0fbe402ull, 0xc01ed534e31ca57full},
  {0xfda4f3514d75465dull, 0xc00b1a20021146c6ull}, {0xff36f1701909c3ddull, 0xc0013bd2c8da4951ull},
  {0x00c90e8fe6f63c23ull, 0xc0013bd2c8da4951ull}, {0x025b0caeb28ab9a3ull, 0xc00b1a20021146c6ull},
  {0x03ecadcf3f041bfeull, 0xc01ed534e31ca57full}, {0x057db402a6a90630ull, 0xc03c6a068549edccull},
  {0x070de171e7b0b53dull, 0xc063d40524b30a57ull}, {0x089cf8676d7abb56ull, 0xc0950d1cd4517db9ull},
  {0x0a2abb58949f2cedull, 0xc0d00db66deccaf1ull}, {0x0bb6ecef285f98a4ull, 0xc114ccb8bdbf113eull},
  {0x0d415012d802284full, 0xc1633f89e9a1a664ull}, {0x0ec9a7f2a2a188afull, 0xc1bb5a11138a4c90ull},
  {0x104fb80e37fdadffull, 0xc21d0eb837187b4eull}, {0x11d3443f4cdb3dd2ull, 0xc2884e6e41e9178eull},
  {0x135410c2e18151b1ull, 0xc2fd08a9665de674ull}, {0x14d1e24278e76a25ull, 0xc37b2b69a87d032cull},
  {0x164c7ddd3f27c611ull, 0xc402a33ba483aaa9ull}, {0x17c3a9311dcce702ull, 0xc4935b3b8ebeca6bull},
  {0x19372a63bc93d72dull, 0xc52d3d186c32ea7aull}, {0x1aa6c82b6d3fc98bull, 0xc5d0311783944811ull},
  {0x1c1249d8011ee6a0ull, 0xc67c1e1806074787ull}, {0x1d79775b86e38955ull, 0xc730e996ef18c9c5ull},
  {0x1edc1952ef78d589ull, 0xc7ee77b31b556de5ull}, {0x2039f90e987d6db3ull, 0xc8b4ab3194de5b41ull},
  {0x2192e09abb131d39ull, 0xc98365821551dcf6ull}, {0x22e69ac7bdb69141ull, 0xca5a86c3bc55dea4ull},
  {0x2434f33267d6b163ull, 0xcb39edc9fa0a3c7aull}, {0x257db64bf5e7d3efull, 0xcc217821aca0d794ull},
  {0x26c0b1620cb3e570ull, 0xcd11021670517c8bull}, {0x27fdb2a68aada89bull, 0xce0866b820d7e62eull},
  {0x293489373612716cull, 0xcf077fe08ba28297ull}, {0x2a65052546ab2b98ull, 0xd00e263951d11eceull},
  {0x2b8ef77cca031883ull, 0xd11c3141f91b3da9ull}, {0x2cb2324be0f07ae2ull, 0xd23177562aaea2eeull},
  {0x2dce88a9d5515d12ull, 0xd34dcdb41f0f851eull}, {0x2ee3cebe06e4c257ull, 0xd471088335fce77dull},
  {0x2ff1d9c6ae2ee132ull, 0xd59afadab954d468ull}, {0x30f8801f745d7d69ull, 0xd6cb76c8c9ed8e94ull},
  {0x31f79947df2819d2ull, 0xd8024d5975525765ull}, {0x32eefde98fae8375ull, 0xd93f4e9df34c1a90ull},
  {0x33de87de535f286cull, 0xda8249b40a182c11ull}, {0x34c6123605f5c386ull, 0xdbcb0ccd98294e9dull},
  {0x35a5793c43aa215cull, 0xdd19653842496ebfull}, {0x367c9a7deaae230aull, 0xde6d1f6544ece2c7ull},
  {0x374b54ce6b21a4bfull, 0xdfc606f16782924dull}, {0x3811884ce4aa921bull, 0xe123e6ad10872a77ull},
  {0x38cf166910e7363bull, 0xe28688a4791c76abull}, {0x3983e1e7f9f8b879ull, 0xe3edb627fee11960ull},
  {0x3a2fcee87c6bb7efull, 0xe55937d492c03675ull}, {0x3ad2c2e793cd1586ull, 0xe6c8d59c436c28d3ull},
  {0x3b6ca4c471413595ull, 0xe83c56cee23318feull}, {0x3bfd5cc45b7c5557ull, 0xe9b38222c0d839efull},
  {0x3c84d4965782fcd4ull, 0xeb2e1dbd871895dbull}, {0x3d02f75699a2198cull, 0xecabef3d1e7eae4full},
  {0x3d77b191be16e872ull, 0xee2cbbc0b324c22eull}, {0x3de2f147c8e784b2ull, 0xefb047f1c8025201ull},
  {0x3e44a5eeec75b370ull, 0xf136580d5d5e7751ull}, {0x3e9cc076165e599cull, 0xf2beafed27fdd7b1ull},
  {0x3eeb33474240eec2ull, 0xf4491310d7a0675cull}, {0x3f2ff2499213350full, 0xf5d544a76b60d313ull},
  {0x3f6af2e32bae8247ull, 0xf7630798928544aaull}, {0x3f9c2bfadb4cf5a9ull, 0xf8f21e8e184f4ac3ull},
  {0x3fc395f97ab61234ull, 0xfa824bfd5956f9d0ull}, {0x3fe12acb1ce35a81ull, 0xfc135230c0fbe402ull},
  {0x3ff4e5dffdeeb93aull, 0xfda4f3514d75465dull}, {0x3ffec42d3725b6afull, 0xff36f1701909c3ddull},
};

FLB_HD uint64_t fx_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
FLB_HD int64_t fx_mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
FLB_HD int fx_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}
FLB_HD Fx2 fx_load(const Fx2* p) {
#ifdef __CUDA_ARCH__
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
  return Fx2{v.x, v.y};
#else
  return *p;
#endif
}
// (a b) >> 32 for a 64-bit a and a 32-bit b (bits 32 .. 95 of the product)
FLB_HD uint64_t fx_mul64x32(uint64_t a, uint32_t b) {
  return (a >> 32) * b + (((a & 0xFFFFFFFFull) * b) >> 32);
}

// sqrt(-2 ln((w + 1/2) 2^-32)) = s 2^-(60 + k): returns s < 2^63
FLB_HD int64_t fx_radius(uint32_t w, int& k) {
  const uint64_t x = 2 * (uint64_t)w + 1;
  const int e = 63 - fx_clz(x);                                   // 0 .. 32
  const uint64_t m = x << (32 - e);                               // Q32, [1, 2)
  const int i = (int)(m >> 25) & 127;
  const Fx2 t = fx_load(&kFxLog[i]);
  const int64_t z = (int64_t)(m * (uint32_t)t.a) - (1ll << 41);   // Q41, exact, |z| < 2^33.3
  const int32_t zs = (int32_t)(z >> 3);                           // Q38
  // 1/4 - z (1/5 - z (1/6 - z / 7)) in Q32
  const int64_t t6 = 0x2aaaaaab - (((int64_t)zs * 0x24924925) >> 38);
  const int64_t t5 = 0x33333333 - (((int64_t)zs * (int32_t)t6) >> 38);
  const int64_t t4 = 0x40000000 - (((int64_t)zs * (int32_t)t5) >> 38);
  const int64_t t3 = 0x1555555555555555ll - (((int64_t)zs * (int32_t)t4) >> 8);   // 1/3 - z t4, Q62
  const uint64_t t2 = (1ull << 63) - ((uint64_t)fx_mulhi_s((int64_t)((uint64_t)z << 22), t3) << 3);   // 1/2 - z t3, Q64
  const uint64_t az = (uint64_t)(z < 0 ? -z : z) << 23;           // |z|, Q64
  // near: ln 2 - ln c = 0, and all from here is scaled by 2^sn
  const bool top = e == 32;
  const int sn = top && i == 127 ? fx_clz(az) & ~1 : 0;
  const uint64_t q = fx_mulhi(az << sn, fx_mulhi(az, t2));        // z^2 t2, Q64
  const uint64_t l1 = ((uint64_t)z << (22 + sn)) - (q >> 1);      // ln(1 + z), Q63 (two's complement)
  // ln 2 - ln m in Q63, the whole of -ln ua for ua >= 1/2; otherwise plus (32 - e) ln 2 in Q59
  const uint64_t f = 0x58b90bfbe8e7bcd6ull - t.b - l1;
  const uint64_t a = top ? f : (f >> 4) + (uint64_t)(32 - e) * 0x058b90bfbe8e7bcdull;
  // sqrt(2 a 2^-59), a = v 2^-sh: 2^(3 - sh/2) sqrt(v 2^-64), two halvings fewer for Q63
  const int sh = fx_clz(a) & ~1;
  const uint64_t v = a << sh;                                     // Q64, [1/4, 1)
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint2float_rz((uint32_t)(v >> 32)) * 0x1p-32f));
  uint32_t Y = __float2uint_rz(y * 0x1p30f);
#else
  uint32_t Y = (uint32_t)(0x1p30f / __builtin_sqrtf((float)(uint32_t)(v >> 40) * 0x1p-24f));
#endif
  Y -= (Y >> 22) + 1;                     // below 1 / sqrt v, so that h stays below 1
  // h = v y in Q64: bits 30 .. 93 of v Y (y in Q30)
  const uint64_t h = (fx_mul64x32(v, Y) << 2) | (((uint32_t)v * Y) >> 30);
  // e = 1 - h y, 0 < e < 2^-20, in Q64: the low 64 bits of -(h Y >> 30)
  const int64_t er = -(int64_t)((fx_mul64x32(h, Y) << 2) | (((uint32_t)h * Y) >> 30));
  const int32_t e32 = (int32_t)(er >> 16);                        // Q48
  const int64_t c = (er >> 1) + (int64_t)((((uint64_t)((int64_t)e32 * e32) >> 32) * 3) >> 3);   // e / 2 + 3/8 e^2
  const int64_t s = (int64_t)(h >> 1) + fx_mulhi_s((int64_t)(h >> 1), c);         // Q63
  k = ((sh + sn) >> 1) + (top ? 2 : 0);
  return s;
}

// cos and sin of 2 pi (w + 1/2) 2^-32 in Q62
FLB_HD void fx_sincos(uint32_t w, int64_t& c, int64_t& s) {
  const uint64_t x = 2 * (uint64_t)w + 1;                         // in units of 2^-33 turns
  const Fx2 t = fx_load(&kFxTrig[x >> 25]);
  const int32_t rem = (int32_t)(x & 0x1FFFFFFu) - (1 << 24);
  const uint32_t ar = (uint32_t)(rem < 0 ? -rem : rem);
  // |delta| = |rem| 2^-33 2 pi in Q70 (2 pi in Q61: the product is in Q94)
  const uint64_t K = 0xc90fdaa22168c235ull;
  const uint64_t lo = (K & 0xFFFFFFFFull) * ar, p = (K >> 32) * ar + (lo >> 32);   // Q62
  const uint64_t d = (p << 8) | ((uint32_t)lo >> 24);             // Q70, < 2^63.7
  const uint64_t d2 = fx_mulhi(d, d);                             // Q76, < 2^63.4
  const uint32_t d2h = (uint32_t)(d2 >> 32);                      // Q44
  // sin: d (1 - d2 (1/6 - d2 (1/120 - d2 / 5040)))
  const uint32_t b1 = 0x88888889u - (uint32_t)(((uint64_t)d2h * 0xd00d00d0u) >> 50);         // Q38
  const uint64_t s1 = 0xaaaaaaaaaaaaaaabull - (fx_mul64x32(d2, b1) >> 16);                   // Q66
  const int64_t sd = (int64_t)((d - (fx_mulhi(d, fx_mulhi(d2, s1)) >> 14)) >> 1);            // Q69
  // 1 - cos: d2 (1/2 - d2 (1/24 - d2 / 720))
  const uint64_t b2 = 0x2aaaaaaaaaaaaaabull - (fx_mul64x32(d2, 0xb60b60b6u) >> 19);          // Q66
  const int64_t cm = (int64_t)fx_mulhi(d2, (1ull << 63) - (fx_mulhi(d2, b2) >> 14));         // Q76
  const int64_t C = (int64_t)t.a, S = (int64_t)t.b, sn = rem < 0 ? -sd : sd;
  c = C - (fx_mulhi_s(C, cm) >> 12) - (fx_mulhi_s(S, sn) >> 5);   // Q74 >> 12, Q67 >> 5
  s = S - (fx_mulhi_s(S, cm) >> 12) + (fx_mulhi_s(C, sn) >> 5);
}

// a 2^-p rounded to a double (assembled from its bits: a conversion would use the FP64 pipe)
FLB_HD double fx_to_double(int64_t a, int p) {
  const uint64_t m = (uint64_t)(a < 0 ? -a : a);
  const int lz = fx_clz(m);
  const uint64_t t = m << (lz & 63);
  uint64_t b = ((uint64_t)(1023 + 63 - 1 - p - lz) << 52) + (t >> 11) + ((t >> 10) & 1);
  if (m == 0) b = 0;
  b |= (uint64_t)a & (1ull << 63);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double r;
  __builtin_memcpy(&r, &b, 8);
  return r;
#endif
}

// Box-Muller on a word pair, FP64 results
FLB_HD void fx_box_muller(uint32_t wa, uint32_t wb, double& n0, double& n1) {
  int k;
  const int64_t r = fx_radius(wa, k);                             // r 2^-(60 + k) < 6.8
  int64_t c, s;
  fx_sincos(wb, c, s);
  n0 = fx_to_double(fx_mulhi_s(r, c), 58 + k);                    // 60 + k + 62 - 64
  n1 = fx_to_double(fx_mulhi_s(r, s), 58 + k);
}

}  // namespace flb
