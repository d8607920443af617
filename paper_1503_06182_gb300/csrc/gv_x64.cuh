// gv_x64.cuh -- the FP64 form's arithmetic on the integer pipes.
//
// This chip issues one warp-wide FP64 instruction per SM every ~19 cycles: an
// FP64 operation costs as much as ~76 issue slots of the other pipes, and the
// FP64 fills were bound by nothing else.  A 64 x 64 -> 64 bit product takes
// ~8 integer instructions, so the FP64 form evaluates its events in numbers
// with a 64-bit significand instead (GvX), or in 64-bit fixed point where a
// quantity is bounded: 11 bits more than FP64 keeps, in less time.  A weight
// is rounded once, to FP64, at the end.  One fill of 1e6 Drell-Yan events on 4
// axes: 350 us on the FP64 pipe (a warp instruction per ~19 cycles per SM, the
// pipe full), 95 us here (about 2100 instructions per event);
// 1e5 events of the NLO-shaped weight on 13 axes: 230 us there, 50 with an
// exponential per axis and fewer with one per event.  Weights at
// random points: 2^-54.2 rms from 200-bit values, of which the final rounding
// alone makes 2^-54.8.
//
//   GvX: (-1)^s m 2^e, m in [2^63, 2^64), or m = 0 with a very negative e.
//   Q64: an unsigned 64-bit fraction of 1.
//
// exp2 and log2 reduce their argument by a 256-entry table and sum a Taylor
// series (the methods of P. T. P. Tang, ACM TOMS 15 (1989) and 16 (1990), in
// integers); sine and cosine are Taylor series after reduction to an eighth
// of a turn; 1/x and its seed are Newton-Raphson steps from the hardware's
// FP32 approximation.  Tables: gv_x_exp2_tab[j] = floor(2^(j/256) 2^63);
// gv_x_log2_tab[j] = (R, floor(-log2(R 2^-31) 2^64)), R = ceil(2^31 / (1 +
// j/256)).  The test suite recomputes every entry and runs this file on the
// host against 300-bit arithmetic: relative errors stay below 2^-59 for one
// operation or function, against 2^-53 for one FP64 rounding.
#pragma once
#include <cstdint>

// clang-format off
#ifndef __CUDACC__
struct ulonglong2 {
  unsigned long long x, y;
};
#define __device__
#define __align__(n)
#endif
static __device__ __align__(16) const unsigned long long gv_x_exp2_tab[256] = {
    0x8000000000000000ull, 0x8058d7d2d5e5f6b0ull, 0x80b1ed4fd999ab6cull, 0x810b40a1d81406d4ull,
    0x8164d1f3bc030773ull, 0x81bea1708dde6055ull, 0x8218af4373fc25ebull, 0x8272fb97b2a5894cull,
    0x82cd8698ac2ba1d7ull, 0x83285071e0fc4546ull, 0x8383594eefb6ee36ull, 0x83dea15b9541b132ull,
    0x843a28c3acde4046ull, 0x8495efb3303efd2full, 0x84f1f656379c1a29ull, 0x854e3cd8f9c8c95dull,
    0x85aac367cc487b14ull, 0x86078a2f23642a9full, 0x8664915b923fba03ull, 0x86c1d919caef5c87ull,
    0x871f61969e8d1010ull, 0x877d2afefd4e256cull, 0x87db357ff698d791ull, 0x88398146b919f1d4ull,
    0x88980e8092da8527ull, 0x88f6dd5af155ac6bull, 0x8955ee03618e5fdcull, 0x89b540a7902557a3ull,
    0x8a14d575496efd9aull, 0x8a74ac9a79896e46ull, 0x8ad4c6452c728924ull, 0x8b3522a38e1e1031ull,
    0x8b95c1e3ea8bd6e6ull, 0x8bf6a434adde0084ull, 0x8c57c9c4646f4dddull, 0x8cb932c1bae97a95ull,
    0x8d1adf5b7e5ba9e5ull, 0x8d7ccfc09c50e2f7ull, 0x8ddf042022e69cd5ull, 0x8e417ca940e35a01ull,
    0x8ea4398b45cd53c0ull, 0x8f073af5a2013520ull, 0x8f6a8117e6c8e5c4ull, 0x8fce0c21c6726481ull,
    0x9031dc431466b1dcull, 0x9095f1abc540ca6bull, 0x90fa4c8beee4b12aull, 0x915eed13c89689d3ull,
    0x91c3d373ab11c336ull, 0x9228ffdc10a051acull, 0x928e727d9531f9acull, 0x92f42b88f673aa7cull,
    0x935a2b2f13e6e92bull, 0x93c071a0eef94bc0ull, 0x9426ff0fab1c04b6ull, 0x948dd3ac8ddb7ed3ull,
    0x94f4efa8fef70961ull, 0x955c5336887894d5ull, 0x95c3fe86d6cc7feeull, 0x962bf1cbb8d9755full,
    0x96942d3720185a00ull, 0x96fcb0fb20ac4ba2ull, 0x97657d49f17ab08eull, 0x97ce9255ec4357abull,
    0x9837f0518db8a96full, 0x98a1976f7597e995ull, 0x990b87e266c189a9ull, 0x9975c1dd47518c77ull,
    0x99e0459320b7fa64ull, 0x9a4b13371fd166caull, 0x9ab62afc94ff864aull, 0x9b218d16f441d63cull,
    0x9b8d39b9d54e5538ull, 0x9bf93118f3aa4cc1ull, 0x9c6573682ec32c2dull, 0x9cd200db8a0774caull,
    0x9d3ed9a72cffb750ull, 0x9dabfdff6367a2a9ull, 0x9e196e189d472420ull, 0x9e872a276f0b98ffull,
    0x9ef5326091a111adull, 0x9f6386f8e28ba650ull, 0x9fd228256400dd05ull, 0xa041161b3d0121bdull,
    0xa0b0510fb9714fc2ull, 0xa11fd9384a344cf7ull, 0xa18faeca8544b6e3ull, 0xa1ffd1fc25cea188ull,
    0xa27043030c496818ull, 0xa2e102153e918f9eull, 0xa3520f68e802bb92ull, 0xa3c36b345991b47bull,
    0xa43515ae09e6809eull, 0xa4a70f0c95768ec4ull, 0xa5195786be9ef339ull, 0xa58bef536dbeb6edull,
    0xa5fed6a9b15138eaull, 0xa6720dc0be08a20bull, 0xa6e594cfeee86b1dull, 0xa7596c0ec55ff55bull,
    0xa7cd93b4e9653569ull, 0xa8420bfa298f70d1ull, 0xa8b6d5167b320e08ull, 0xa92bef41fa77771bull,
    0xa9a15ab4ea7c0ef8ull, 0xaa1717a7b5693979ull, 0xaa8d2652ec907629ull, 0xab0386ef48868de0ull,
    0xab7a39b5a93ed337ull, 0xabf13edf162675e8ull, 0xac6896a4be3fe929ull, 0xace0413ff83e5d03ull,
    0xad583eea42a14ac6ull, 0xadd08fdd43d01491ull, 0xae493452ca35b80eull, 0xaec22c84cc5c9465ull,
    0xaf3b78ad690a4374ull, 0xafb51906e75b8661ull, 0xb02f0dcbb6e04583ull, 0xb0a957366fb7a3c9ull,
    0xb123f581d2ac258full, 0xb19ee8e8c94feb08ull, 0xb21a31a66618fe3bull, 0xb295cff5e47db4a3ull,
    0xb311c412a9112489ull, 0xb38e0e38419fae17ull, 0xb40aaea2654b9840ull, 0xb487a58cf4a9c180ull,
    0xb504f333f9de6484ull, 0xb58297d3a8b9f0d1ull, 0xb60093a85ed5f76bull, 0xb67ee6eea3b22b8full,
    0xb6fd91e328d17791ull, 0xb77c94c2c9d725e8ull, 0xb7fbefca8ca41e7cull, 0xb87ba337a1743833ull,
    0xb8fbaf4762fb9ee9ull, 0xb97c143756844dbeull, 0xb9fcd2452c0b9deaull, 0xba7de9aebe5fea08ull,
    0xbaff5ab2133e45fbull, 0xbb81258d5b704b6full, 0xbc034a7ef2e9fb0cull, 0xbc85c9c560e7b269ull,
    0xbd08a39f580c36beull, 0xbd8bd84bb67ed482ull, 0xbe0f6809860993e2ull, 0xbe935317fc378237ull,
    0xbf1799b67a731082ull, 0xbf9c3c248e2486f8ull, 0xc0213aa1f0d08db0ull, 0xc0a6956e8836ca8cull,
    0xc12c4cca66709456ull, 0xc1b260f5ca0fbb33ull, 0xc238d2311e3d6672ull, 0xc2bfa0bcfad907c8ull,
    0xc346ccda24976407ull, 0xc3ce56c98d21b15dull, 0xc4563ecc5334cb32ull, 0xc4de8523c2c07baaull,
    0xc5672a115506daddull, 0xc5f02dd6b0bbc3d9ull, 0xc67990b5aa245f79ull, 0xc70352f04336c51dull,
    0xc78d74c8abb9b15cull, 0xc817f681416452b2ull, 0xc8a2d85c8ffe2c45ull, 0xc92e1a9d517f0ecbull,
    0xc9b9bd866e2f27a2ull, 0xca45c15afcc72623ull, 0xcad2265e4290774dull, 0xcb5eecd3b38597c8ull,
    0xcbec14fef2727c5cull, 0xcc799f23d11510e5ull, 0xcd078b86503dcdd1ull, 0xcd95da6a9ff06444ull,
    0xce248c151f8480e3ull, 0xceb3a0ca5dc6a55dull, 0xcf4318cf191918c1ull, 0xcfd2f4683f94eeb5ull,
    0xd06333daef2b2594ull, 0xd0f3d76c75c5db8cull, 0xd184df6251699ac6ull, 0xd2164c023056bcabull,
    0xd2a81d91f12ae45aull, 0xd33a5457a3029054ull, 0xd3ccf099859ac379ull, 0xd45ff29e0972c560ull,
    0xd4f35aabcfedfa1full, 0xd5872909ab75d189ull, 0xd61b5dfe9f9bce06ull, 0xd6aff9d1e13ba2fdull,
    0xd744fccad69d6af4ull, 0xd7da67311797f569ull, 0xd870394c6db32c84ull, 0xd9067364d44a929bull,
    0xd99d15c278afd7b5ull, 0xda3420adba4d8704ull, 0xdacb946f2ac9cc71ull, 0xdb63714f8e295255ull,
    0xdbfbb797daf23755ull, 0xdc9467913a4f1c91ull, 0xdd2d818508324c20ull, 0xddc705bcd378f7f0ull,
    0xde60f4825e0e9123ull, 0xdefb4e1f9d1037f1ull, 0xdf9612deb8f04420ull, 0xe031430a0d99e627ull,
    0xe0ccdeec2a94e111ull, 0xe168e6cfd3295d23ull, 0xe2055afffe83d368ull, 0xe2a23bc7d7d91225ull,
    0xe33f8972be8a5a51ull, 0xe3dd444c46499618ull, 0xe47b6ca0373da88dull, 0xe51a02ba8e26d680ull,
    0xe5b906e77c8348a8ull, 0xe658797368b3a716ull, 0xe6f85aaaee1fce22ull, 0xe798aadadd5b9cbeull,
    0xe8396a503c4bdc68ull, 0xe8da9958464b42aaull, 0xe97c38406c4f8c56ull, 0xea1e4756550eb27bull,
    0xeac0c6e7dd24392eull, 0xeb63b7431736983full, 0xec0718b64c1cbddcull, 0xecaaeb8ffb03ab40ull,
    0xed4f301ed9942b84ull, 0xedf3e6b1d418a491ull, 0xee990f980da3025bull, 0xef3eab20e032bc6bull,
    0xefe4b99bdcdaf5cbull, 0xf08b3b58cbe8b76aull, 0xf13230a7ad094509ull, 0xf1d999d8b7708cc1ull,
    0xf281773c59ffb139ull, 0xf329c9233b6bae9cull, 0xf3d28fde3a641a5aull, 0xf47bcbbe6db9fddeull,
    0xf5257d152486cc2cull, 0xf5cfa433e6537290ull, 0xf67a416c733f846dull, 0xf7255510c4288238ull,
    0xf7d0df730ad13bb8ull, 0xf87ce0e5b2094d9bull, 0xf92959bb5dd4ba74ull, 0xf9d64a46eb939f35ull,
    0xfa83b2db722a033aull, 0xfb3193cc4227c3f4ull, 0xfbdfed6ce5f09c48ull, 0xfc8ec01121e447bbull,
    0xfd3e0c0cf486c174ull, 0xfdedd1b496a89f34ull, 0xfe9e115c7b8f884bull, 0xff4ecb59511ec8a5ull,
};
static __device__ __align__(16) const ulonglong2 gv_x_log2_tab[256] = {
    {0x80000000ull, 0x0000000000000000ull}, {0x7f807f81ull, 0x01709c456373a836ull}, {0x7f01fc08ull, 0x02dfca16afb67b65ull},
    {0x7e8472a9ull, 0x044d8c431623230full}, {0x7e07e07full, 0x05b9e59e99964172ull}, {0x7d8c42b3ull, 0x0724d8ed32d21434ull},
    {0x7d11967aull, 0x088e68e80ed0de1aull}, {0x7c97d911ull, 0x09f69848dcd08d0full}, {0x7c1f07c2ull, 0x0b5d69ba995434ceull},
    {0x7ba71fe2ull, 0x0cc2dfdeea651a7eull}, {0x7b301ecdull, 0x0e26fd599ce770feull}, {0x7aba01ebull, 0x0f89c4c1510750b4ull},
    {0x7a44c6b0ull, 0x10eb389ee9f55f8aull}, {0x79d06a97ull, 0x124b5b7c25f36678ull}, {0x795ceb25ull, 0x13aa2fda33f8e0a9ull},
    {0x78ea45e8ull, 0x1507b8344ca76a53ull}, {0x78787879ull, 0x1663f6f929941160ull}, {0x78078079ull, 0x17beee93bc01a448ull},
    {0x77975b90ull, 0x1918a16de9de3d19ull}, {0x77280773ull, 0x1a7111dda9382d47ull}, {0x76b981dbull, 0x1bc842405ce14081ull},
    {0x764bc88dull, 0x1d1e34e1b9212c44ull}, {0x75ded953ull, 0x1e72ec111d8b42aeull}, {0x7572b202ull, 0x1fc66a0e86464a0aull},
    {0x75075076ull, 0x2118b116a4204bbfull}, {0x749cb290ull, 0x2269c368e3e1cd34ull}, {0x7432d63eull, 0x23b9a32dcf0cd07cull},
    {0x73c9b972ull, 0x250852931b539cecull}, {0x73615a25ull, 0x2655d3c1ec135c84ull}, {0x72f9b659ull, 0x27a228d815d3ffd4ull},
    {0x7292cc16ull, 0x28ed53f15ce4f193ull}, {0x722c996cull, 0x2a375720bb03e214ull}, {0x71c71c72ull, 0x2b8034733f02d416ull},
    {0x71625345ull, 0x2cc7edf2fd65114bull}, {0x70fe3c08ull, 0x2e0e85a6cd3182e6ull}, {0x709ad4e5ull, 0x2f53fd8ebcc99cdcull},
    {0x70381c0full, 0x3098579d2a93ff77ull}, {0x6fd60fbbull, 0x31db95cd737b4c50ull}, {0x6f74ae27ull, 0x331dba0cb608734dull},
    {0x6f13f597ull, 0x345ec6435be54005ull}, {0x6eb3e454ull, 0x359ebc582adb1da9ull}, {0x6e5478adull, 0x36dd9e2cb4ea6388ull},
    {0x6df5b0f8ull, 0x381b6d99b6c7b9d1ull}, {0x6d978b8full, 0x39582c78dfae448eull}, {0x6d3a06d4ull, 0x3a93dc972188f80aull},
    {0x6cdd212cull, 0x3bce7fc5441c0ffbull}, {0x6c80d902ull, 0x3d0817cd935fe484ull}, {0x6c252cc8ull, 0x3e40a6702e34e479ull},
    {0x6bca1af3ull, 0x3f782d7065510f2bull}, {0x6b6fa1ffull, 0x40aeae86ded2f794ull}, {0x6b15c06cull, 0x41e42b6b98d762eaull},
    {0x6abc74bfull, 0x4318a5d2487eb9edull}, {0x6a63bd82ull, 0x444c1f6a20193709ull}, {0x6a0b9945ull, 0x457e99da1981d1ebull},
    {0x69b4069cull, 0x46b016c7aa58aad6ull}, {0x695d041eull, 0x47e097da1949134eull}, {0x6906906aull, 0x49101ea8caf44d08ull},
    {0x68b0aa20ull, 0x4a3eacd38d9c0355ull}, {0x685b4fe6ull, 0x4b6c43f0e5a043daull}, {0x68068069ull, 0x4c98e58a36d042a5ull},
    {0x67b23a55ull, 0x4dc49337ea43f940ull}, {0x675e7c5eull, 0x4eef4e8161249c0cull}, {0x670b453cull, 0x501918eae3a7681full},
    {0x66b893aaull, 0x5141f3f90bc5d883ull}, {0x66666667ull, 0x5269e12d0a6f7a7eull}, {0x6614bc37ull, 0x5390e200db3cab9eull},
    {0x65c393e1ull, 0x54b6f7ee49ec8f7bull}, {0x6572ec30ull, 0x55dc246b2e6425a7ull}, {0x6522c3f4ull, 0x570068e59730de39ull},
    {0x64d319ffull, 0x5823c6ce89915180ull}, {0x6483ed28ull, 0x59463f8ee9703dbbull}, {0x64353c49ull, 0x5a67d48e9ae262c5ull},
    {0x63e7063full, 0x5b888734614a0f48ull}, {0x639949ecull, 0x5ca858de53bbe40full}, {0x634c0635ull, 0x5dc74ae90f52d3c5ull},
    {0x62ff3a02ull, 0x5ee55eaf95dc16b5ull}, {0x62b2e43eull, 0x6002958b2c5cb0a7ull}, {0x626703d9ull, 0x611ef0cbb7c5c2b5ull},
    {0x621b97c3ull, 0x623a71ca50eea496ull}, {0x61d09ef4ull, 0x635519cb191ab3cbull}, {0x61861862ull, 0x646eea22aeb28eecull},
    {0x613c030aull, 0x6587e41423d2b760ull}, {0x60f25debull, 0x66a008e3ae928c1dull}, {0x60a92807ull, 0x67b759d2c2d709baull},
    {0x60606061ull, 0x68cdd82799cd5e7eull}, {0x60180602ull, 0x69e38519f477a425ull}, {0x5fd017f5ull, 0x6af861e238c4becbull},
    {0x5f889546ull, 0x6c0c6fbd3ab786e0ull}, {0x5f417d06ull, 0x6d1fafdcb3dff3c5ull}, {0x5eface49ull, 0x6e32236eca37e4b2ull},
    {0x5eb48824ull, 0x6f43cba5b981e761ull}, {0x5e6ea9afull, 0x7054a9affa3e9e02ull}, {0x5e293206ull, 0x7164beb43202f500ull},
    {0x5de42047ull, 0x72740bd8df62dba8ull}, {0x5d9f7391ull, 0x73829248367d09d5ull}, {0x5d5b2b09ull, 0x7490531c5219a03bull},
    {0x5d1745d2ull, 0x759d4f7ea1a98a7eull}, {0x5cd3c316ull, 0x76a988843e7137e4ull}, {0x5c90a1feull, 0x77b4ff4d7910ad23ull},
    {0x5c4de1b7ull, 0x78bfb4f1ed5e621eull}, {0x5c0b8171ull, 0x79c9aa8452ca9a48ull}, {0x5bc9805cull, 0x7ad2e11e6a25130eull},
    {0x5b87ddaeull, 0x7bdb59c8ce8027adull}, {0x5b46989bull, 0x7ce3159b0414b8abull}, {0x5b05b05cull, 0x7dea159f3472f5daull},
    {0x5ac5242bull, 0x7ef05ae2334e99e2ull}, {0x5a84f346ull, 0x7ff5e66738e021f7ull}, {0x5a451cebull, 0x80fab9380c06763full},
    {0x5a05a05bull, 0x81fed458b999108cull}, {0x59c67cd9ull, 0x830238cb8c5ffff7ull}, {0x5987b1aaull, 0x8404e790f63912d8ull},
    {0x59493e15ull, 0x8506e1a779280d0bull}, {0x590b2165ull, 0x8608280344ac99c3ull}, {0x58cd5ae3ull, 0x8708bba6f60ff4d7ull},
    {0x588fe9ddull, 0x88089d8689c4753cull}, {0x5852cda1ull, 0x8907ce9c014374b1ull}, {0x58160582ull, 0x8a064fd271c1067dull},
    {0x57d990d1ull, 0x8b0422232f3e6d4bull}, {0x579d6ee4ull, 0x8c0146786cd28fa4ull}, {0x57619f10ull, 0x8cfdbdc655f72403ull},
    {0x572620afull, 0x8df988f1b4c23b16ull}, {0x56eaf31aull, 0x8ef4a8e92daf6fbbull}, {0x56b015adull, 0x8fef1e9448710c10ull},
    {0x567587c5ull, 0x90e8eadbd4d09f2bull}, {0x563b48c3ull, 0x91e20e9d07e0c866ull}, {0x56015806ull, 0x92da8ac30b2f16b4ull},
    {0x55c7b4f2ull, 0x93d26028faec59a7ull}, {0x558e5eeaull, 0x94c98fb389307e39ull}, {0x55555556ull, 0x95c01a37192d9afdull},
    {0x551c979bull, 0x96b6009a32b4322full}, {0x54e42524ull, 0x97ab43ae8a39ae12ull}, {0x54abfd5bull, 0x989fe44f3755e3c6ull},
    {0x54741facull, 0x9993e353a9111392ull}, {0x543c8b85ull, 0x9a87418f8d735b85ull}, {0x54054055ull, 0x9b79ffd71e5300e9ull},
    {0x53ce3d8cull, 0x9c6c1eff17346549ull}, {0x5397829dull, 0x9d5d9fd3d4f69643ull}, {0x53610efcull, 0x9e4e83220aa765baull},
    {0x532ae21dull, 0x9f3ec9bb2811cd97ull}, {0x52f4fb77ull, 0xa02e746802a4463full}, {0x52bf5a82ull, 0xa11d83f19b6c8866ull},
    {0x5289feb6ull, 0xa20bf9258e263c1dull}, {0x5254e78full, 0xa2f9d4c4239fa95aull}, {0x52201489ull, 0xa3e7179218fc35b0ull},
    {0x51eb851full, 0xa4d3c25d25b2706aull}, {0x51b738d2ull, 0xa5bfd5dc6a78fc30ull}, {0x51832f20ull, 0xa6ab52d8e5cbe72aull},
    {0x514f678cull, 0xa7963a094c670aaaull}, {0x511be196ull, 0xa8808c36325e5cd9ull}, {0x50e89cc3ull, 0xa96a4a15b5567d12ull},
    {0x50b59898ull, 0xaa5374621948f221ull}, {0x5082d49aull, 0xab3c0bd9cc082e08ull}, {0x50505051ull, 0xac2411319d00db4aull},
    {0x501e0b45ull, 0xad0b852269bfb459ull}, {0x4fec04ffull, 0xadf268648252570dull}, {0x4fba3d0bull, 0xaed8bba65a685e16ull},
    {0x4f88b2f4ull, 0xafbe7f9ef4795315ull}, {0x4f576647ull, 0xb0a3b4fffc768c51ull}, {0x4f265692ull, 0xb1885c7a58b7c821ull},
    {0x4ef58365ull, 0xb26c76b9714e17e8ull}, {0x4ec4ec4full, 0xb3500471274705abull}, {0x4e9490e2ull, 0xb433064b1961ca4eull},
    {0x4e6470b1ull, 0xb5157cefe80a11c4ull}, {0x4e348b4eull, 0xb5f769109be94337ull}, {0x4e04e04full, 0xb6d8cb4f0c0271f9ull},
    {0x4dd56f48ull, 0xb7b9a45a1f733071ull}, {0x4da637d0ull, 0xb899f4d62510101aull}, {0x4d77397full, 0xb979bd66340c4dc6ull},
    {0x4d4873edull, 0xba58feb0e7d0e080ull}, {0x4d19e6b4ull, 0xbb37b956ce3b8a78ull}, {0x4ceb916eull, 0xbc15edfbe7e9e424ull},
    {0x4cbd73b6ull, 0xbcf39d42daeca730ull}, {0x4c8f8d29ull, 0xbdd0c7c81422bee5ull}, {0x4c61dd64ull, 0xbead6e2b58bb7933ull},
    {0x4c346405ull, 0xbf89910af0296040ull}, {0x4c0720acull, 0xc06530febcbd30daull}, {0x4bda12f7ull, 0xc1404eab9b5a569aull},
    {0x4bad3a88ull, 0xc21aeaa63aa65659ull}, {0x4b809702ull, 0xc2f5058190a64773ull}, {0x4b542805ull, 0xc3ce9fe26b69b88dull},
    {0x4b27ed37ull, 0xc4a7ba536489ee66ull}, {0x4afbe63aull, 0xc5805575ce37088full}, {0x4ad012b5ull, 0xc65871d581263025ull},
    {0x4aa4724cull, 0xc73010102c539699ull}, {0x4a7904a8ull, 0xc80730add617b677ull}, {0x4a4dc96full, 0xc8ddd4485a05faceull},
    {0x4a22c04bull, 0xc9b3fb68b72163cdull}, {0x49f7e8e3ull, 0xca89a6a9cc0b3209ull}, {0x49cd42e3ull, 0xcb5ed6907ba7fc7dull},
    {0x49a2cdf4ull, 0xcc338bb38738c641ull}, {0x497889c3ull, 0xcd07c6988baad667ull}, {0x494e75fbull, 0xcddb87d204b1efb8ull},
    {0x4924924aull, 0xceaecfe62c883841ull}, {0x48fade5dull, 0xcf819f6310f4a31dull}, {0x48d159e3ull, 0xd053f6cf6c908503ull},
    {0x48a8048bull, 0xd125d6b4b6a53d5cull}, {0x487ede05ull, 0xd1f73f9a0d0d128cull}, {0x4855e602ull, 0xd2c8320427d324ffull},
    {0x482d1c32ull, 0xd398ae7f88bcbeecull}, {0x48048049ull, 0xd468b586e7753069ull}, {0x47dc11f8ull, 0xd53847a6f3fefdceull},
    {0x47b3d0f2ull, 0xd6076564c2d48768ull}, {0x478bbcedull, 0xd6d60f38887c44b1ull}, {0x4763d59dull, 0xd7a445a74e24dff6ull},
    {0x473c1ab7ull, 0xd8720933828f7ac6ull}, {0x47148bf1ull, 0xd93f5a5ced83605aull}, {0x46ed2902ull, 0xda0c39a0a33c81f8ull},
    {0x46c5f1a0ull, 0xdad8a78367b3d676ull}, {0x469ee585ull, 0xdba4a47798c356edull}, {0x46780468ull, 0xdc703101a62f3276ull},
    {0x46514e03ull, 0xdd3b4d98bb2856c4ull}, {0x462ac20full, 0xde05fabba2afe1f6ull}, {0x46046047ull, 0xded038e104abe478ull},
    {0x45de2865ull, 0xdf9a0887268458f2ull}, {0x45b81a26ull, 0xe0636a1ecabc594bull}, {0x45923544ull, 0xe12c5e2ae176cb79ull},
    {0x456c797eull, 0xe1f4e516262ddfa7ull}, {0x4546e690ull, 0xe2bcff5d7f882fbeull}, {0x45217c39ull, 0xe384ad701e363ed6ull},
    {0x44fc3a35ull, 0xe44befcf72a503cdull}, {0x44d72045ull, 0xe512c6e46e4e8b6full}, {0x44b22e28ull, 0xe5d93324df7defbfull},
    {0x448d639eull, 0xe69f35036614a5bdull}, {0x4468c067ull, 0xe764ccf4ccc404e9ull}, {0x44444445ull, 0xe829fb65389c6e3aull},
    {0x441feef9ull, 0xe8eec0c851556915ull}, {0x43fbc044ull, 0xe9b31d93e27961e6ull}, {0x43d7b7ebull, 0xea77122a164f53ecull},
    {0x43b3d5b0ull, 0xeb3a9eff6d51c677ull}, {0x43901957ull, 0xebfdc47f95d93a94ull}, {0x436c82a3ull, 0xecc0831dbf98801dull},
    {0x43491159ull, 0xed82db4433e90437ull}, {0x4325c53full, 0xee44cd59ba6b8cc3ull}, {0x43029e1bull, 0xef0659c70ef536b2ull},
    {0x42df9bb1ull, 0xefc78101eea017a6ull}, {0x42bcbdc9ull, 0xf088436c01a84037ull}, {0x429a042aull, 0xf148a16e5d2096e8ull},
    {0x42776e9bull, 0xf2089b7404381b71ull}, {0x4254fce5ull, 0xf2c831dec6c9c179ull}, {0x4232aeceull, 0xf38765230b295b64ull},
    {0x42108422ull, 0xf4463595aa56d9a4ull}, {0x41ee7ca7ull, 0xf504a3aed32f849aull}, {0x41cc982aull, 0xf5c2afc16a402568ull},
    {0x41aad672ull, 0xf6805a43c39178cdull}, {0x4189374cull, 0xf73da38c5a209c63ull}, {0x4167ba82ull, 0xf7fa8c044cc52c36ull},
    {0x41465fe0ull, 0xf8b7140b405e5a0eull}, {0x41252731ull, 0xf9733c08463c6213ull}, {0x41041042ull, 0xfa2f0458e10b5ffcull},
    {0x40e31adfull, 0xfaea6d61fc8698c4ull}, {0x40c246d5ull, 0xfba57784950f3041ull}, {0x40a193f2ull, 0xfc60231daa6913bdull},
    {0x40810205ull, 0xfd1a70863274f451ull}, {0x406090daull, 0xfdd46029fe8ed3fcull}, {0x40404041ull, 0xfe8df25fab1fb8fdull},
    {0x40201009ull, 0xff47278533331840ull},
};
// clang-format on

#define GV_X_ZERO_E (-(1 << 20))  // exponent of zero

struct GvX {
  unsigned long long m;
  int e;
  unsigned s;  // 0 or 1
};

// ---- integer helpers (the host versions serve the tests)
#ifdef __CUDA_ARCH__
#define GV_X_FN __device__ __forceinline__
GV_X_FN unsigned long long xi_mulhi(unsigned long long a, unsigned long long b) {
  return __umul64hi(a, b);
}
GV_X_FN unsigned xi_mulhi32(unsigned a, unsigned b) { return __umulhi(a, b); }
GV_X_FN int xi_clz(unsigned long long a) { return __clzll((long long)a); }
GV_X_FN float xi_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
GV_X_FN long long xi_bits(double x) { return __double_as_longlong(x); }
GV_X_FN double xi_double(unsigned long long b) { return __longlong_as_double((long long)b); }
GV_X_FN float xi_u2f(unsigned x) { return __uint2float_rz(x); }
GV_X_FN unsigned xi_f2u(float x) { return __float2uint_rz(x); }
#else
#define GV_X_FN inline
#include <cstring>
GV_X_FN unsigned long long xi_mulhi(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
GV_X_FN unsigned xi_mulhi32(unsigned a, unsigned b) {
  return (unsigned)(((unsigned long long)a * b) >> 32);
}
GV_X_FN int xi_clz(unsigned long long a) { return a ? __builtin_clzll(a) : 64; }
GV_X_FN float xi_rcp(float x) { return 1.0f / x; }
GV_X_FN long long xi_bits(double x) {
  long long b;
  memcpy(&b, &x, 8);
  return b;
}
GV_X_FN double xi_double(unsigned long long b) {
  double x;
  memcpy(&x, &b, 8);
  return x;
}
GV_X_FN float xi_u2f(unsigned x) { return (float)x; }
GV_X_FN unsigned xi_f2u(float x) { return (unsigned)x; }
#endif
// (a b) >> 32 for a 32-bit b
GV_X_FN unsigned long long xi_mul64x32(unsigned long long a, unsigned b) {
  return (unsigned long long)(unsigned)(a >> 32) * b + xi_mulhi32((unsigned)a, b);
}

// ---- conversions
GV_X_FN GvX x_zero() { return GvX{0ull, GV_X_ZERO_E, 0u}; }
// m 2^e for any m, normalised
GV_X_FN GvX x_norm(unsigned long long m, int e, unsigned s = 0u) {
  if (m == 0ull) return x_zero();
  const int lz = xi_clz(m);
  return GvX{m << lz, e - lz, s};
}
// a finite double, exactly
GV_X_FN GvX x_from(double x) {
  const unsigned long long b = (unsigned long long)xi_bits(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  const unsigned long long f = b & 0xFFFFFFFFFFFFFull;
  return x_norm(ef ? f | (1ull << 52) : f, (ef ? ef : 1) - 1075, (unsigned)(b >> 63));
}
// rounded to the nearest double, ties to even; beyond FP64, infinity
GV_X_FN double x_to_double(const GvX& v) {
  const unsigned long long sign = (unsigned long long)v.s << 63;
  if (v.m == 0ull) return xi_double(sign);
  const int nf = v.e + 63 + 1023;  // exponent field of the leading bit
  if (nf > 0 && nf < 0x7FF) {
    // 53 bits and a round bit; a carry runs into the exponent, as it should
    const unsigned long long q = v.m >> 11, rest = v.m & 0x7FFull;
    const unsigned long long up = (rest > 0x400ull || (rest == 0x400ull && (q & 1ull))) ? 1ull : 0ull;
    return xi_double((sign | ((unsigned long long)nf << 52)) + (q & 0xFFFFFFFFFFFFFull) + up);
  }
  if (nf >= 0x7FF) return xi_double(sign | 0x7FF0000000000000ull);
  const int sh = 12 - nf;  // subnormal: units of 2^-1074
  if (sh > 64) return xi_double(sign);
  const unsigned long long q = sh == 64 ? 0ull : v.m >> sh;
  const unsigned long long half = (v.m >> (sh - 1)) & 1ull;
  const unsigned long long rest = v.m & ((1ull << (sh - 1)) - 1ull);
  return xi_double(sign | (q + ((half && (rest || (q & 1ull))) ? 1ull : 0ull)));
}
// a fraction in [0, 1) as GvX; a GvX in [0, 1] as a fraction (truncated; 1, which
// a grid's width or an exponential can round to, is the largest fraction)
GV_X_FN GvX x_from_q64(unsigned long long q) { return x_norm(q, -64); }
GV_X_FN unsigned long long x_to_q64(const GvX& v) {
  const int sh = -64 - v.e;
  if (sh < 0) return ~0ull;
  return sh < 64 ? v.m >> sh : 0ull;
}

// ---- arithmetic (errors: truncations below 2^-62 of the result)
GV_X_FN GvX x_mul(const GvX& a, const GvX& b) {
  unsigned long long m = xi_mulhi(a.m, b.m);
  int e = a.e + b.e + 64;
  if ((long long)m >= 0) {
    m += m;
    --e;
  }
  return GvX{m, e, a.s ^ b.s};
}
GV_X_FN GvX x_sqr(const GvX& a) { return x_mul(a, a); }
GV_X_FN GvX x_neg(GvX a) {
  a.s ^= 1u;
  return a;
}
// a 2^k
GV_X_FN GvX x_scale(GvX a, int k) {
  a.e += k;
  return a;
}
// a + b for two values of the same sign
GV_X_FN GvX x_addp(const GvX& a, const GvX& b) {
  const bool sw = a.e < b.e;
  const unsigned long long hm = sw ? b.m : a.m, lm = sw ? a.m : b.m;
  const int he = sw ? b.e : a.e, d = he - (sw ? a.e : b.e);
  unsigned long long m = hm + (d < 64 ? lm >> d : 0ull);
  int e = he;
  if (m < hm) {
    m = (m >> 1) | (1ull << 63);
    ++e;
  }
  return GvX{m, e, a.s};
}
GV_X_FN GvX x_add(const GvX& a, const GvX& b) {
  const bool sw = a.e < b.e || (a.e == b.e && a.m < b.m);
  const unsigned long long hm = sw ? b.m : a.m, lm = sw ? a.m : b.m;
  const int he = sw ? b.e : a.e, d = he - (sw ? a.e : b.e);
  const unsigned s = sw ? b.s : a.s;
  const unsigned long long t = d < 64 ? lm >> d : 0ull;
  if (a.s == b.s) {
    unsigned long long m = hm + t;
    int e = he;
    if (m < hm) {
      m = (m >> 1) | (1ull << 63);
      ++e;
    }
    return GvX{m, e, s};
  }
  return x_norm(hm - t, he, s);
}
GV_X_FN GvX x_sub(const GvX& a, const GvX& b) { return x_add(a, x_neg(b)); }

// 1/x for x != 0: rho = 2^64/m in (1, 2] from the FP32 approximation (22
// bits, Q30) by two Newton-Raphson steps rho + rho (1 - mu rho), mu = m 2^-64;
// the residual 1 - mu rho is the negated low word of the product.
GV_X_FN GvX x_rcp(const GvX& x) {
  const unsigned mh = (unsigned)(x.m >> 32), ml = (unsigned)x.m;
  const unsigned y0 = xi_f2u(xi_rcp(xi_u2f(mh)) * 0x1p62f);  // Q30 of 2^32/mh
  const unsigned long long t0 =
      (((unsigned long long)mh * y0) << 2) + (((unsigned long long)ml * y0) >> 30);
  const long long e0 = -(long long)t0;  // Q64
  const unsigned long long y1 =
      ((unsigned long long)y0 << 32) + (unsigned long long)(((long long)y0 * (e0 >> 12)) >> 20);  // Q62
  const unsigned long long t1 = (xi_mulhi(x.m, y1) << 2) | ((x.m * y1) >> 62);
  const long long e1 = -(long long)t1;
  unsigned long long y2 = y1 + (unsigned long long)(((long long)(y1 >> 32) * e1) >> 32);
  y2 = y2 >> 63 ? ~0ull : y2 << 1;  // x a power of two: 2 to the last place
  return GvX{y2, -127 - x.e, x.s};
}

// 2^t with t = -(m 2^e) (neg) or m 2^e, m not necessarily normalised and e < 0.
GV_X_FN GvX x_exp2(unsigned long long m, int e, bool neg) {
  if (e > -44) {  // |t| >= 2^20 unless m is small
    if (m == 0ull) return GvX{1ull << 63, -63, 0u};
    const int lz = xi_clz(m);
    if (64 - lz + e > 20) return neg ? x_zero() : GvX{1ull << 63, 1 << 18, 0u};
    m <<= lz;
    e -= lz;
  }
  const int r = -e;  // 44 <= r
  int k = r < 64 ? (int)(m >> r) : 0;
  unsigned long long f = r <= 64 ? (r == 64 ? m : m << (64 - r)) : (r < 128 ? m >> (r - 64) : 0ull);
  if (neg) {
    k = -k;
    if (f) {
      --k;
      f = 0ull - f;
    }
  }
#ifdef __CUDA_ARCH__
  const unsigned long long T = __ldg(gv_x_exp2_tab + (f >> 56));
#else
  const unsigned long long T = gv_x_exp2_tab[f >> 56];
#endif
  // y = (fraction below 2^-8) ln 2 as Q64, below 2^-8.5; e^y - 1 by Taylor
  const unsigned long long y = xi_mulhi(f << 8, 0xb17217f7d1cf79abull) >> 8;
  const unsigned y32 = (unsigned)(y >> 32);
  unsigned q = 0x2222222u + xi_mulhi32(y32, 0x5b05b0u);  // 1/120 + y/720
  q = 0xaaaaaaau + xi_mulhi32(y32, q);                   // 1/24 + ..
  const unsigned long long q2 = 0x2aaaaaaaaaaaaaaaull + xi_mul64x32(y, q);  // 1/6 + ..
  const unsigned long long q1 = 0x8000000000000000ull + xi_mulhi(y, q2);   // 1/2 + ..
  const unsigned long long em1 = y + xi_mulhi(y, xi_mulhi(y, q1));
  return GvX{T + xi_mulhi(T, em1), k - 63, 0u};
}
GV_X_FN GvX x_exp2(const GvX& t) { return x_exp2(t.m, t.e, t.s != 0u); }

// log2 x for x > 0.
GV_X_FN GvX x_log2(const GvX& x) {
#ifdef __CUDA_ARCH__
  const ulonglong2 RL = __ldg(gv_x_log2_tab + ((x.m >> 55) & 255));
#else
  const ulonglong2 RL = gv_x_log2_tab[(x.m >> 55) & 255];
#endif
  const unsigned R = (unsigned)RL.x;
  // r = (m 2^-63) (R 2^-31) - 1 in [0, 2^-8), Q64: the product's integer part drops out
  const unsigned long long r = (((x.m >> 32) * R) << 2) + (((x.m & 0xFFFFFFFFull) * R) >> 30);
  const unsigned r32 = (unsigned)(r >> 32);
  // ln(1 + r) = r - r^2 (1/2 - r (1/3 - r (1/4 - r (1/5 - r (1/6 - r/7)))))
  unsigned b = 0x2aaaaaaau - xi_mulhi32(r32, 0x24924924u);
  b = 0x33333333u - xi_mulhi32(r32, b);
  b = 0x40000000u - xi_mulhi32(r32, b);
  const unsigned long long b2 = 0x5555555555555555ull - xi_mul64x32(r, b);
  const unsigned long long b1 = 0x8000000000000000ull - xi_mulhi(r, b2);
  const unsigned long long ln = r - xi_mulhi(r, xi_mulhi(r, b1));
  unsigned long long F = RL.y + (xi_mulhi(ln, 0xb8aa3b295c17f0bbull) << 1);
  if (F < RL.y) F = ~0ull;  // the last place below 1
  // integer part I and fraction F
  const int I = x.e + 63;
  if (I == -1 && F) return x_norm(0ull - F, -64, 1u);  // x in (1/2, 1): -(1 - F)
  if (I == 0) return x_norm(F, -64);
  if (I > 0) return x_addp(x_norm((unsigned long long)I, 0), x_norm(F, -64));
  return x_add(GvX{x_norm((unsigned long long)(-I), 0).m, x_norm((unsigned long long)(-I), 0).e, 1u},
               x_norm(F, -64));
}

// cos and sin of 2 pi p, p a fraction of a turn, in signed Q62.  u = the
// distance to the nearest quarter turn in quarter turns (<= 1/2), z = u^2;
// Taylor series in z with (pi/2)^n/n!, the high terms in 32 bits.
GV_X_FN long long xi_cos_quarter(unsigned long long z) {  // cos(u pi/2), Q62
  const unsigned z32 = (unsigned)(z >> 32);
  unsigned q = 0x48319u - xi_mulhi32(z32, 0x950u);  // Q52
  q = 0x1b6e24fu - xi_mulhi32(z32, q);
  q = 0x7e74e28eu - xi_mulhi32(z32, q);
  unsigned long long c = 0x000069b47ca8812aull - xi_mulhi(z, (unsigned long long)q << 10);
  c = 0x000f0fa83448dd5dull - xi_mulhi(z, c);
  c = 0x0155d3c7e3cbff9full - xi_mulhi(z, c);
  c = 0x103c1f081b5ac3b3ull - xi_mulhi(z, c);
  c = 0x4ef4f326f9177969ull - xi_mulhi(z, c);
  return (long long)(0x4000000000000000ull - xi_mulhi(z, c));
}
GV_X_FN long long xi_sin_quarter(unsigned long long u, unsigned long long z) {  // Q62
  const unsigned z32 = (unsigned)(z >> 32);
  unsigned q = 0x5beb7u - xi_mulhi32(z32, 0xd57u);  // Q49
  q = 0x1e8f435u - xi_mulhi32(z32, q);
  q = 0x78c1d3f8u - xi_mulhi32(z32, q);
  unsigned long long c = 0x0002a0f0690fdcf0ull - xi_mulhi(z, (unsigned long long)q << 13);
  c = 0x004cb4b3398af616ull - xi_mulhi(z, c);
  c = 0x0519af19dd6ab874ull - xi_mulhi(z, c);
  c = 0x295779cc4b7ca57dull - xi_mulhi(z, c);
  c = 0x6487ed5110b4611aull - xi_mulhi(z, c);
  return (long long)xi_mulhi(u, c);
}
struct GvTurn {  // p = quadrant/4 + (-1)^neg u/4
  unsigned quadrant;
  bool neg;
  unsigned long long u, z;
};
GV_X_FN GvTurn xi_turn(unsigned long long p) {
  GvTurn t;
  const unsigned long long c = p + (1ull << 61);
  t.quadrant = (unsigned)(c >> 62);
  const long long d = (long long)(p - (c & 0xC000000000000000ull));  // [-2^61, 2^61)
  t.neg = d < 0;
  t.u = (unsigned long long)(t.neg ? -d : d) << 2;
  t.z = xi_mulhi(t.u, t.u);
  return t;
}
GV_X_FN long long x_cos_turn(unsigned long long p) {
  const GvTurn t = xi_turn(p);
  // both polynomials have one shape: the coefficients are selected, so that
  // the lanes of a warp do not take two paths
  const bool odd = (t.quadrant & 1u) != 0u;
  const unsigned z32 = (unsigned)(t.z >> 32);
  unsigned q = (odd ? 0x5beb7u : 0x48319u) - xi_mulhi32(z32, odd ? 0xd57u : 0x950u);
  q = (odd ? 0x1e8f435u : 0x1b6e24fu) - xi_mulhi32(z32, q);
  q = (odd ? 0x78c1d3f8u : 0x7e74e28eu) - xi_mulhi32(z32, q);
  unsigned long long p4 = (odd ? 0x0002a0f0690fdcf0ull : 0x000069b47ca8812aull) -
                          xi_mulhi(t.z, (unsigned long long)q << (odd ? 13 : 10));
  p4 = (odd ? 0x004cb4b3398af616ull : 0x000f0fa83448dd5dull) - xi_mulhi(t.z, p4);
  p4 = (odd ? 0x0519af19dd6ab874ull : 0x0155d3c7e3cbff9full) - xi_mulhi(t.z, p4);
  p4 = (odd ? 0x295779cc4b7ca57dull : 0x103c1f081b5ac3b3ull) - xi_mulhi(t.z, p4);
  p4 = (odd ? 0x6487ed5110b4611aull : 0x4ef4f326f9177969ull) - xi_mulhi(t.z, p4);
  p4 = xi_mulhi(odd ? t.u : t.z, p4);
  const long long v = (long long)(odd ? p4 : 0x4000000000000000ull - p4);
  // quadrant 0: cos, 1: -sin d, 2: -cos, 3: sin d
  const bool neg = t.quadrant == 0u   ? false
                   : t.quadrant == 1u ? !t.neg
                   : t.quadrant == 2u ? true
                                      : t.neg;
  return neg ? -v : v;
}
GV_X_FN void x_sincos_turn(unsigned long long p, long long* sn, long long* cs) {
  const GvTurn t = xi_turn(p);
  const long long c = xi_cos_quarter(t.z);
  const long long s0 = xi_sin_quarter(t.u, t.z), s = t.neg ? -s0 : s0;
  const bool odd = (t.quadrant & 1u) != 0u;
  const long long a = odd ? c : s, b = odd ? s : c;  // |sin|, |cos| up to signs
  *sn = (t.quadrant & 2u) ? -a : a;
  *cs = (t.quadrant == 1u || t.quadrant == 2u) ? -b : b;
}
// a signed Q62 value as GvX
GV_X_FN GvX x_from_q62(long long v) {
  return x_norm((unsigned long long)(v < 0 ? -v : v), -62, v < 0 ? 1u : 0u);
}
// sqrt of v in [0, 1] (Q62): s0 = mu rsqrt(mu) from the FP32 approximation,
// then two steps s + (mu - s^2) rsqrt(mu) / 2.
GV_X_FN float xi_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}
GV_X_FN long long xi_sqrt_q62(unsigned long long v) {
  if (v == 0ull) return 0;
  const int z = xi_clz(v) & ~1;
  const unsigned long long u = v << z;  // mu = u 2^-64 in [1/4, 1)
  const float f = xi_u2f((unsigned)(u >> 32)) * 0x1p-32f, y = xi_rsqrt(f);
  const float sf = f * y * 0x1p32f;
  const unsigned s0 = sf < 0x1.fffffep31f ? xi_f2u(sf) : 0xFFFFFF00u;  // Q32
  const unsigned yq = xi_f2u(y * 0x1p30f);                             // Q30
  const long long r0 = (long long)(u - (unsigned long long)s0 * s0);   // Q64
  const unsigned long long s1 =
      ((unsigned long long)s0 << 31) + (unsigned long long)(((r0 >> 12) * (long long)yq) >> 20);  // Q63
  // mu - s1^2 in Q126, then its bits from 2^-94 up
  const unsigned long long ph = xi_mulhi(s1, s1), pl = s1 * s1;
  const unsigned long long tl = u << 62, th = u >> 2;
  const unsigned long long dl = tl - pl, dh = th - ph - (tl < pl ? 1ull : 0ull);
  const long long r1 = (long long)((dh << 32) | (dl >> 32));  // Q94
  const unsigned long long s2 = s1 + (unsigned long long)(((r1 >> 20) * (long long)yq) >> 42);
  return (long long)(s2 >> (z / 2));  // sqrt(v 2^62): s2 2^-63 sqrt(2^-z) in Q62 is s2 >> (1 + z/2) << 1
}
// signed Q62 product (truncated towards minus infinity)
GV_X_FN long long xi_mulq62(long long a, long long b) {
#ifdef __CUDA_ARCH__
  return (__mul64hi(a, b) << 2) | (long long)(((unsigned long long)a * (unsigned long long)b) >> 62);
#else
  return (long long)(((__int128)a * b) >> 62);
#endif
}
