// log10 and 10^v for the opacity tables, with few FP64 instructions (see fix64.cuh for why): 9 and
// 11, about 30 each in the CUDA library's. Both are table-driven argument reductions
// (P. T. P. Tang, "Table-driven implementation of the logarithm function in IEEE floating-point
// arithmetic", ACM TOMS 16, 1990, and of the exponential function, TOMS 15, 1989):
//   x = 2^e m,  c ~ 1/m to 7 bits (10-bit numbers, so that m c - 1 is one exact FMA),
//   log10 x = e log10 2 - log10 c + log10(1 + r),  r = m c - 1, |r| < 2^-7.6;
//   10^v = 2^(n/128) e^z,  n = round(128 v / log10 2),  z = (v - n log10(2)/128) ln 10, |z| < 2^-8.5.
// The leading terms of the two short series are FP64, the rest (below 2^-17 of the sum) FP32. The
// tables hold c, -log10 c in two parts, and 2^(j/128), rounded from 200-bit values.
//
// Against 200-bit values 10^v is within a unit of the last place, and log10 x within half a unit
// where |log10 x| is above 0.1. Near x = 1 the sum cancels: the absolute error stays below 5e-18
// (a table's coordinate, log10 x less the table's start over its spacing, does not see it), but
// it is no longer small beside log10 x itself. Not a replacement for log10 elsewhere.
#pragma once
#include "fix64.cuh"

namespace fld {

struct __align__(32) LogRow {
    double c, l, lo, pad;
};
static __device__ const LogRow k_log10_tab[128] = {
    {0x1.fe00000000000p-1, 0x1.bd96a1d800000p-10, -0x1.31a1eb97093b9p-45, 0.0},
    {0x1.fa00000000000p-1, 0x1.4f82052340000p-8, 0x1.102c95c0dc644p-44, 0.0},
    {0x1.f600000000000p-1, 0x1.18b2dc8d20000p-7, 0x1.7721c86a32e2ap-44, 0.0},
    {0x1.f280000000000p-1, 0x1.7c441aa5e0000p-7, 0x1.b4533966c4829p-45, 0.0},
    {0x1.ee80000000000p-1, 0x1.eeeab9b440000p-7, -0x1.77467df16102ap-44, 0.0},
    {0x1.eb00000000000p-1, 0x1.29fff7b8d0000p-6, -0x1.618b4ef79c38fp-44, 0.0},
    {0x1.e780000000000p-1, 0x1.5ce72239a0000p-6, -0x1.d1a132eeb5289p-44, 0.0},
    {0x1.e380000000000p-1, 0x1.9786f287a0000p-6, -0x1.d651a345db748p-49, 0.0},
    {0x1.e000000000000p-1, 0x1.cb38fccd90000p-6, -0x1.00925a535ae72p-44, 0.0},
    {0x1.dc80000000000p-1, 0x1.ff4be13b90000p-6, 0x1.48fd764dea1d9p-45, 0.0},
    {0x1.d900000000000p-1, 0x1.19e086b3b8000p-5, 0x1.99ac1fd443e40p-48, 0.0},
    {0x1.d600000000000p-1, 0x1.30838cdc30000p-5, -0x1.00c12f7a1b586p-47, 0.0},
    {0x1.d280000000000p-1, 0x1.4b1b588128000p-5, 0x1.20287dac177e6p-45, 0.0},
    {0x1.cf00000000000p-1, 0x1.65e6692548000p-5, -0x1.d8cf527f38ac6p-48, 0.0},
    {0x1.cc00000000000p-1, 0x1.7d070145f8000p-5, -0x1.8145a563de9f8p-44, 0.0},
    {0x1.c880000000000p-1, 0x1.98335cd4a0000p-5, 0x1.6c2c0931d0032p-45, 0.0},
    {0x1.c580000000000p-1, 0x1.afa88992b0000p-5, -0x1.5e6edad46beacp-45, 0.0},
    {0x1.c280000000000p-1, 0x1.c74591df70000p-5, 0x1.22aea9b40f263p-44, 0.0},
    {0x1.bf80000000000p-1, 0x1.df0afe1508000p-5, -0x1.463f99aa83d1ap-44, 0.0},
    {0x1.bc80000000000p-1, 0x1.f6f9594de8000p-5, -0x1.f0f9c4cf885d9p-45, 0.0},
    {0x1.b980000000000p-1, 0x1.078898bc04000p-4, 0x1.bf44e72402874p-44, 0.0},
    {0x1.b680000000000p-1, 0x1.13a98bb450000p-4, 0x1.f0168af5d72d9p-45, 0.0},
    {0x1.b380000000000p-1, 0x1.1fdfcf7838000p-4, 0x1.8038fc483bdc1p-44, 0.0},
    {0x1.b080000000000p-1, 0x1.2c2baf7880000p-4, 0x1.7b6b8c091127dp-44, 0.0},
    {0x1.ad80000000000p-1, 0x1.388d78b934000p-4, 0x1.0feadd5856604p-44, 0.0},
    {0x1.ab00000000000p-1, 0x1.42efeb4b50000p-4, 0x1.ba270494ee73dp-46, 0.0},
    {0x1.a800000000000p-1, 0x1.4f7aad9bbc000p-4, 0x1.75da8a5871b9ap-45, 0.0},
    {0x1.a580000000000p-1, 0x1.59ffb662b8000p-4, 0x1.5bcd1450d31d8p-48, 0.0},
    {0x1.a300000000000p-1, 0x1.6494c46ac8000p-4, -0x1.1b294ba31c9a5p-44, 0.0},
    {0x1.a000000000000p-1, 0x1.715d0ce368000p-4, -0x1.41149840eaa65p-46, 0.0},
    {0x1.9d80000000000p-1, 0x1.7c1607b7d8000p-4, -0x1.cdee31de0d912p-48, 0.0},
    {0x1.9b00000000000p-1, 0x1.86dfa808d4000p-4, -0x1.2c09bb60238bap-45, 0.0},
    {0x1.9880000000000p-1, 0x1.91ba21d6c0000p-4, -0x1.088de1de62c8cp-44, 0.0},
    {0x1.9600000000000p-1, 0x1.9ca5aa1728000p-4, 0x1.f44a74b04a5b6p-44, 0.0},
    {0x1.9380000000000p-1, 0x1.a7a276badc000p-4, 0x1.2c79e9957c9d4p-44, 0.0},
    {0x1.9100000000000p-1, 0x1.b2b0beb418000p-4, 0x1.ad02ad13bc4d7p-44, 0.0},
    {0x1.8e80000000000p-1, 0x1.bdd0b9fd08000p-4, 0x1.a0fc2eafba507p-44, 0.0},
    {0x1.8c00000000000p-1, 0x1.c902a19e64000p-4, 0x1.1117390924cd5p-44, 0.0},
    {0x1.8980000000000p-1, 0x1.d446afb64c000p-4, 0x1.f95fec4153145p-46, 0.0},
    {0x1.8780000000000p-1, 0x1.dd5727676c000p-4, 0x1.2b2443f2d9850p-45, 0.0},
    {0x1.8500000000000p-1, 0x1.e8bc77271c000p-4, -0x1.a197240569ddfp-46, 0.0},
    {0x1.8280000000000p-1, 0x1.f4349618fc000p-4, -0x1.6e6791f17a5c9p-44, 0.0},
    {0x1.8080000000000p-1, 0x1.fd6f308ce4000p-4, 0x1.b51fe006d8435p-44, 0.0},
    {0x1.7e00000000000p-1, 0x1.0484e4942a000p-3, 0x1.4867cc62a8c08p-44, 0.0},
    {0x1.7c00000000000p-1, 0x1.093025a19a000p-3, -0x1.128d0950e065ap-44, 0.0},
    {0x1.7980000000000p-1, 0x1.0f0f17a062000p-3, 0x1.a9547d2cbfbb2p-46, 0.0},
    {0x1.7780000000000p-1, 0x1.13c8a1e350000p-3, -0x1.0bfa55f697578p-44, 0.0},
    {0x1.7580000000000p-1, 0x1.1888a1c996000p-3, -0x1.b3c1301ae9ac8p-45, 0.0},
    {0x1.7380000000000p-1, 0x1.1d4f291514000p-3, -0x1.fed10b114338bp-47, 0.0},
    {0x1.7100000000000p-1, 0x1.23509c1e6e000p-3, -0x1.b2215ab3ec84fp-45, 0.0},
    {0x1.6f00000000000p-1, 0x1.2826167a6c000p-3, -0x1.b1d5505664200p-46, 0.0},
    {0x1.6d00000000000p-1, 0x1.2d0253f67e000p-3, 0x1.32ac22596b4a0p-45, 0.0},
    {0x1.6b00000000000p-1, 0x1.31e56798aa000p-3, -0x1.debad218b9aa2p-44, 0.0},
    {0x1.6900000000000p-1, 0x1.36cf64b7a8000p-3, 0x1.72f237e0ce5c8p-46, 0.0},
    {0x1.6700000000000p-1, 0x1.3bc05efcbc000p-3, -0x1.cf6e4c905eeddp-44, 0.0},
    {0x1.6500000000000p-1, 0x1.40b86a657c000p-3, 0x1.479a53a17bd7cp-44, 0.0},
    {0x1.6300000000000p-1, 0x1.45b79b45c8000p-3, 0x1.5459420146650p-45, 0.0},
    {0x1.6180000000000p-1, 0x1.497bbcf096000p-3, -0x1.afdef4b07dcb4p-45, 0.0},
    {0x1.5f80000000000p-1, 0x1.4e87a15648000p-3, -0x1.2643fb03d92d0p-45, 0.0},
    {0x1.5d80000000000p-1, 0x1.539ae4e6fa000p-3, -0x1.9236ae719d455p-50, 0.0},
    {0x1.5b80000000000p-1, 0x1.58b59d4bcc000p-3, 0x1.d25c440efd186p-46, 0.0},
    {0x1.5a00000000000p-1, 0x1.5c8e998072000p-3, 0x1.fc353e9430bfbp-44, 0.0},
    {0x1.5800000000000p-1, 0x1.61b6939984000p-3, -0x1.f70dc69c572dap-44, 0.0},
    {0x1.5600000000000p-1, 0x1.66e6400da4000p-3, -0x1.1116ad28239b0p-48, 0.0},
    {0x1.5480000000000p-1, 0x1.6acf1c53f8000p-3, -0x1.35947f360dcefp-45, 0.0},
    {0x1.5280000000000p-1, 0x1.700c78c3e6000p-3, 0x1.089422f108989p-47, 0.0},
    {0x1.5100000000000p-1, 0x1.73ffb42e56000p-3, 0x1.2141b769b4890p-44, 0.0},
    {0x1.4f00000000000p-1, 0x1.794b099a26000p-3, -0x1.84765db2f226ap-47, 0.0},
    {0x1.4d80000000000p-1, 0x1.7d48dbc3aa000p-3, -0x1.af4c54295627bp-46, 0.0},
    {0x1.4c00000000000p-1, 0x1.814b4921be000p-3, -0x1.5a928400b36a5p-44, 0.0},
    {0x1.4a00000000000p-1, 0x1.86ab17c10c000p-3, -0x1.c0b434f5d2b7ap-46, 0.0},
    {0x1.4880000000000p-1, 0x1.8ab86e6288000p-3, 0x1.9ad1afab13d0fp-44, 0.0},
    {0x1.4700000000000p-1, 0x1.8eca84642a000p-3, -0x1.68dc92d80a93bp-44, 0.0},
    {0x1.4500000000000p-1, 0x1.943f6cfd3e000p-3, 0x1.2de43955d0f41p-44, 0.0},
    {0x1.4380000000000p-1, 0x1.985cc29a14000p-3, -0x1.dc7d9674ea185p-48, 0.0},
    {0x1.4200000000000p-1, 0x1.9c7efd734a000p-3, 0x1.7c9690248757ep-46, 0.0},
    {0x1.4080000000000p-1, 0x1.a0a6293cf6000p-3, -0x1.e2dcb81d6c8acp-45, 0.0},
    {0x1.3f00000000000p-1, 0x1.a4d251d554000p-3, 0x1.250e2ae44fb70p-44, 0.0},
    {0x1.3d80000000000p-1, 0x1.a90383459c000p-3, -0x1.64ad9d61e75bap-46, 0.0},
    {0x1.3c00000000000p-1, 0x1.ad39c9c2c6000p-3, 0x1.fe6eb5a4df1dfp-49, 0.0},
    {0x1.3a80000000000p-1, 0x1.b17531ae6a000p-3, -0x1.19e07db80ab20p-44, 0.0},
    {0x1.3900000000000p-1, 0x1.b5b5c79792000p-3, 0x1.f3ccebba162e0p-46, 0.0},
    {0x1.3780000000000p-1, 0x1.b9fb983ba2000p-3, 0x1.bed561985d699p-47, 0.0},
    {0x1.3600000000000p-1, 0x1.be46b08736000p-3, -0x1.688bb48fc920cp-44, 0.0},
    {0x1.3480000000000p-1, 0x1.c2971d970e000p-3, -0x1.9d2c5af984a28p-44, 0.0},
    {0x1.3300000000000p-1, 0x1.c6ececb900000p-3, 0x1.3fd129ff7a4c9p-44, 0.0},
    {0x1.3180000000000p-1, 0x1.cb482b6cf2000p-3, 0x1.06c668ba18341p-48, 0.0},
    {0x1.3000000000000p-1, 0x1.cfa8e765cc000p-3, -0x1.2386ad8b819b8p-45, 0.0},
    {0x1.2e80000000000p-1, 0x1.d40f2e8a82000p-3, 0x1.4001cf4159b54p-45, 0.0},
    {0x1.2d80000000000p-1, 0x1.d701240630000p-3, 0x1.a1d9a58fffce3p-45, 0.0},
    {0x1.2c00000000000p-1, 0x1.db70c7e96e000p-3, 0x1.fcc16f3ba09cbp-45, 0.0},
    {0x1.2a80000000000p-1, 0x1.dfe61d1174000p-3, 0x1.dce090ac2ac30p-44, 0.0},
    {0x1.2900000000000p-1, 0x1.e461322d16000p-3, 0x1.229d2281d2fc1p-45, 0.0},
    {0x1.2800000000000p-1, 0x1.e76124046c000p-3, -0x1.81a1e23fe0fb6p-44, 0.0},
    {0x1.2680000000000p-1, 0x1.ebe5ef9d44000p-3, 0x1.af78ae52b6fecp-50, 0.0},
    {0x1.2500000000000p-1, 0x1.f070a36b8e000p-3, -0x1.8fcf23ae5e081p-45, 0.0},
    {0x1.2400000000000p-1, 0x1.f37b15bab0000p-3, 0x1.1a1fc3b7d53cep-44, 0.0},
    {0x1.2280000000000p-1, 0x1.f80fc47f58000p-3, 0x1.43c4b84b5cd38p-50, 0.0},
    {0x1.2180000000000p-1, 0x1.fb20ecc2ca000p-3, -0x1.abf710c2dc032p-49, 0.0},
    {0x1.2000000000000p-1, 0x1.ffbfc2bbc8000p-3, -0x1.ff229f20ed3d2p-45, 0.0},
    {0x1.1f00000000000p-1, 0x1.016bdf6a18000p-2, 0x1.77bf652b01c58p-50, 0.0},
    {0x1.1d80000000000p-1, 0x1.03c074b41e000p-2, 0x1.25d1d88d0d718p-44, 0.0},
    {0x1.1c80000000000p-1, 0x1.054febffc6000p-2, -0x1.b7ddde0c4a9c8p-44, 0.0},
    {0x1.1b00000000000p-1, 0x1.07a9c2e44b000p-2, -0x1.81f0ce0292635p-46, 0.0},
    {0x1.1a00000000000p-1, 0x1.093cc32c91000p-2, -0x1.f171b2c5f2274p-48, 0.0},
    {0x1.1880000000000p-1, 0x1.0b9bf3979e000p-2, 0x1.e178275604cd7p-46, 0.0},
    {0x1.1780000000000p-1, 0x1.0d328d059b000p-2, 0x1.b8ad13536e28dp-44, 0.0},
    {0x1.1680000000000p-1, 0x1.0eca9b8862000p-2, -0x1.74ab3cc3b5f91p-44, 0.0},
    {0x1.1500000000000p-1, 0x1.113172b49d000p-2, -0x1.83fe713bee31dp-44, 0.0},
    {0x1.1400000000000p-1, 0x1.12cd31b9ca000p-2, -0x1.80449aa0fa56fp-44, 0.0},
    {0x1.1300000000000p-1, 0x1.146a6f5973000p-2, -0x1.f17153840e292p-44, 0.0},
    {0x1.1180000000000p-1, 0x1.16d91f45d1000p-2, -0x1.de16dc4a9ab54p-44, 0.0},
    {0x1.1080000000000p-1, 0x1.187a25ab01000p-2, 0x1.15df26e15bf12p-44, 0.0},
    {0x1.0f80000000000p-1, 0x1.1a1cb48ee9000p-2, 0x1.a49960989de3ep-45, 0.0},
    {0x1.0e80000000000p-1, 0x1.1bc0ced713000p-2, 0x1.387d1621bc3bep-44, 0.0},
    {0x1.0d00000000000p-1, 0x1.1e39e209bd000p-2, 0x1.5ffaaed015cf1p-47, 0.0},
    {0x1.0c00000000000p-1, 0x1.1fe1e5af2c000p-2, 0x1.40eb9b53054c3p-46, 0.0},
    {0x1.0b00000000000p-1, 0x1.218b7f1df6000p-2, -0x1.a78f9277107fbp-44, 0.0},
    {0x1.0a00000000000p-1, 0x1.2336b161b3000p-2, 0x1.9bbc8038401fcp-45, 0.0},
    {0x1.0900000000000p-1, 0x1.24e37f8ece000p-2, -0x1.461fa8e29bedbp-44, 0.0},
    {0x1.0780000000000p-1, 0x1.2769bffab3000p-2, -0x1.00013af9a67f0p-45, 0.0},
    {0x1.0680000000000p-1, 0x1.291aa1a385000p-2, -0x1.a1fdb1804ed40p-44, 0.0},
    {0x1.0580000000000p-1, 0x1.2acd2a4473000p-2, 0x1.9a1c74363b9dfp-45, 0.0},
    {0x1.0480000000000p-1, 0x1.2c815d1b3b000p-2, 0x1.41dd7e925a2f3p-47, 0.0},
    {0x1.0380000000000p-1, 0x1.2e373d6f2b000p-2, 0x1.7c6c96cbf5706p-44, 0.0},
    {0x1.0280000000000p-1, 0x1.2feece914c000p-2, 0x1.e22db36384cc2p-45, 0.0},
    {0x1.0180000000000p-1, 0x1.31a813dc85000p-2, 0x1.01f0aec835f54p-47, 0.0},
    {0x1.0080000000000p-1, 0x1.336310b5c4000p-2, -0x1.21b425357b11fp-45, 0.0},
};
static __device__ const double k_exp2_tab[128] = {
    0x1.0000000000000p+0, 0x1.0163da9fb3335p+0, 0x1.02c9a3e778061p+0, 0x1.04315e86e7f85p+0,
    0x1.059b0d3158574p+0, 0x1.0706b29ddf6dep+0, 0x1.0874518759bc8p+0, 0x1.09e3ecac6f383p+0,
    0x1.0b5586cf9890fp+0, 0x1.0cc922b7247f7p+0, 0x1.0e3ec32d3d1a2p+0, 0x1.0fb66affed31bp+0,
    0x1.11301d0125b51p+0, 0x1.12abdc06c31ccp+0, 0x1.1429aaea92de0p+0, 0x1.15a98c8a58e51p+0,
    0x1.172b83c7d517bp+0, 0x1.18af9388c8deap+0, 0x1.1a35beb6fcb75p+0, 0x1.1bbe084045cd4p+0,
    0x1.1d4873168b9aap+0, 0x1.1ed5022fcd91dp+0, 0x1.2063b88628cd6p+0, 0x1.21f49917ddc96p+0,
    0x1.2387a6e756238p+0, 0x1.251ce4fb2a63fp+0, 0x1.26b4565e27cddp+0, 0x1.284dfe1f56381p+0,
    0x1.29e9df51fdee1p+0, 0x1.2b87fd0dad990p+0, 0x1.2d285a6e4030bp+0, 0x1.2ecafa93e2f56p+0,
    0x1.306fe0a31b715p+0, 0x1.32170fc4cd831p+0, 0x1.33c08b26416ffp+0, 0x1.356c55f929ff1p+0,
    0x1.371a7373aa9cbp+0, 0x1.38cae6d05d866p+0, 0x1.3a7db34e59ff7p+0, 0x1.3c32dc313a8e5p+0,
    0x1.3dea64c123422p+0, 0x1.3fa4504ac801cp+0, 0x1.4160a21f72e2ap+0, 0x1.431f5d950a897p+0,
    0x1.44e086061892dp+0, 0x1.46a41ed1d0057p+0, 0x1.486a2b5c13cd0p+0, 0x1.4a32af0d7d3dep+0,
    0x1.4bfdad5362a27p+0, 0x1.4dcb299fddd0dp+0, 0x1.4f9b2769d2ca7p+0, 0x1.516daa2cf6642p+0,
    0x1.5342b569d4f82p+0, 0x1.551a4ca5d920fp+0, 0x1.56f4736b527dap+0, 0x1.58d12d497c7fdp+0,
    0x1.5ab07dd485429p+0, 0x1.5c9268a5946b7p+0, 0x1.5e76f15ad2148p+0, 0x1.605e1b976dc09p+0,
    0x1.6247eb03a5585p+0, 0x1.6434634ccc320p+0, 0x1.6623882552225p+0, 0x1.68155d44ca973p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6c012750bdabfp+0, 0x1.6dfb23c651a2fp+0, 0x1.6ff7df9519484p+0,
    0x1.71f75e8ec5f74p+0, 0x1.73f9a48a58174p+0, 0x1.75feb564267c9p+0, 0x1.780694fde5d3fp+0,
    0x1.7a11473eb0187p+0, 0x1.7c1ed0130c132p+0, 0x1.7e2f336cf4e62p+0, 0x1.80427543e1a12p+0,
    0x1.82589994cce13p+0, 0x1.8471a4623c7adp+0, 0x1.868d99b4492edp+0, 0x1.88ac7d98a6699p+0,
    0x1.8ace5422aa0dbp+0, 0x1.8cf3216b5448cp+0, 0x1.8f1ae99157736p+0, 0x1.9145b0b91ffc6p+0,
    0x1.93737b0cdc5e5p+0, 0x1.95a44cbc8520fp+0, 0x1.97d829fde4e50p+0, 0x1.9a0f170ca07bap+0,
    0x1.9c49182a3f090p+0, 0x1.9e86319e32323p+0, 0x1.a0c667b5de565p+0, 0x1.a309bec4a2d33p+0,
    0x1.a5503b23e255dp+0, 0x1.a799e1330b358p+0, 0x1.a9e6b5579fdbfp+0, 0x1.ac36bbfd3f37ap+0,
    0x1.ae89f995ad3adp+0, 0x1.b0e07298db666p+0, 0x1.b33a2b84f15fbp+0, 0x1.b59728de5593ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.ba5b030a1064ap+0, 0x1.bcc1e904bc1d2p+0, 0x1.bf2c25bd71e09p+0,
    0x1.c199bdd85529cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c67f12e57d14bp+0, 0x1.c8f6d9406e7b5p+0,
    0x1.cb720dcef9069p+0, 0x1.cdf0b555dc3fap+0, 0x1.d072d4a07897cp+0, 0x1.d2f87080d89f2p+0,
    0x1.d5818dcfba487p+0, 0x1.d80e316c98398p+0, 0x1.da9e603db3285p+0, 0x1.dd321f301b460p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e264614f5a129p+0, 0x1.e502ee78b3ff6p+0, 0x1.e7a51fbc74c83p+0,
    0x1.ea4afa2a490dap+0, 0x1.ecf482d8e67f1p+0, 0x1.efa1bee615a27p+0, 0x1.f252b376bba97p+0,
    0x1.f50765b6e4540p+0, 0x1.f7bfdad9cbe14p+0, 0x1.fa7c1819e90d8p+0, 0x1.fd3c22b8f71f1p+0,
};

// signed FP32 images by integer arithmetic (zero for magnitudes below 2^-126)
__device__ __forceinline__ float f32_cut(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7FFu;
    const unsigned u = __funnelshift_l(lo, hi & 0x7FFFFFFFu, 3) - (896u << 23);
    return e < 897u ? 0.f : __uint_as_float(u | (hi & 0x80000000u));
}
// the FP64 value of a small non-negative integer
__device__ __forceinline__ double f64_of_count(int n) {
    const int z = __clz(n);                    // 32 for zero
    const unsigned m = (unsigned)n << (z & 31);   // leading one at bit 31
    const unsigned hi = ((unsigned)(1023 + 31 - z - 1) << 20) + (m >> 11);
    return n ? __hiloint2double((int)hi, (int)(m << 21)) : 0.0;
}

static __device__ __noinline__ double log10_far(double x) { return log10(x); }
static __device__ __noinline__ double exp10_far(double v) { return exp10(v); }

// log10 of a positive finite number
__device__ __forceinline__ double tab_log10(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (hi < 0x00100000u) return log10_far(x);                 // subnormal
    const int e = (int)(hi >> 20) - 1023;
    const double m = __hiloint2double((int)((hi & 0xFFFFFu) | 0x3FF00000u), __double2loint(x));
    const LogRow t = k_log10_tab[(hi >> 13) & 127u];
    const double r = fma(m, t.c, -1.0);
    const float rf = f32_cut(r);
    // log(1 + r) = r + r^2 (-1/2 + r/3 - r^2 (1/4 - r/5 + r^2/6 - ..))
    const float tail = rf * rf * fmaf(rf, fmaf(rf, fmaf(rf, -1.f / 7, 1.f / 6), -0.2f), 0.25f);
    const double q = fma(tail > 1e-30f ? f64_of_pos(tail) : 0.0, -1.0, fma(r, 1.0 / 3.0, -0.5));
    const double l = fma(r * r, q, r);
    const double de = e >= 0 ? f64_of_count(e) : -f64_of_count(-e);
    // log10 2 and the table's -log10 c in two parts each: the leading ones are multiples of 2^-42,
    // their sum is exact, and only the final addition rounds
    return fma(de, 0x1.34413509f8000p-2, t.l) + fma(l, 0x1.bcb7b1526e50ep-2, fma(de, -0x1.80433b83b532ap-44, t.lo));
}

// 10^v
__device__ __forceinline__ double tab_exp10(double v) {
    if (((unsigned)__double2hiint(v) & 0x7FFFFFFFu) >= 0x4072C000u) return exp10_far(v);   // |v| >= 300
    const double big = 6755399441055744.0;                     // 1.5 * 2^52: rounds to an integer
    const double t = fma(v, 0x1.a934f0979a371p+8, big);
    const int n = __double2loint(t);
    const double nd = t - big;
    const double z = fma(nd, -0x1.e7fbcc47c4acdp-47, fma(nd, -0x1.34413509f0000p-9, v)) * 0x1.26bb1bbb55516p+1;
    const float zf = f32_cut(z);
    // e^z - 1 = z + z^2 (1/2 + z/6 + z^2 (1/24 + z/120))
    const float tail = zf * zf * fmaf(zf, 1.f / 120, 1.f / 24);
    const double p = fma(tail > 1e-30f ? f64_of_pos(tail) : 0.0, 1.0, fma(z, 1.0 / 6.0, 0.5));
    const double s = fma(z * z, p, z);
    const double T = k_exp2_tab[n & 127];
    const double w = fma(T, s, T);
    return __hiloint2double(__double2hiint(w) + ((n >> 7) << 20), __double2loint(w));
}

}  // namespace fld
