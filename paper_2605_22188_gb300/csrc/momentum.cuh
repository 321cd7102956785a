// The FISTA momentum sequence t_1 = 1, t_{k+1} = (1 + sqrt(1 + 4 t_k^2)) / 2 and its
// coefficients c_k = (t_k - 1) / t_{k+1}, rounded as the kernels round them (4 t^2 + 1 with
// one rounding).  A node's state is the number of steps since its last restart while
// the table holds it, so that a step reads two values; computing them is some fifty
// dependent FP64 operations in one lane, each of which holds the SM's FP64 pipe for 16
// cycles (a proximal step of 1024 nodes of p = 200 between its events 17.7 us with them,
// 15.6 without; of 2048 nodes of p = 2000 51.8 and 49.8).  From step
// 256 on the state is t itself.
#pragma once

#include <cuda_runtime.h>

namespace kglm {

constexpr int kMomN = 256;
constexpr double kMomEnd = 0x1.046d79675393fp+7;   // t after kMomN steps
static __device__ const double kMomC[kMomN] = {
    0x0.0p+0, 0x1.2083feffc8abbp-2, 0x1.bc75b6146cc75p-2, 0x1.0fe798589a647p-1,
    0x1.32931b9e07f5cp-1, 0x1.4c3fad9e9d504p-1, 0x1.60131e0c6922ep-1, 0x1.6fdf367993570p-1,
    0x1.7cc512a6ff0b4p-1, 0x1.878222452490bp-1, 0x1.9097f1bf813e7p-1, 0x1.9862390d6e9fap-1,
    0x1.9f23cc02baaf7p-1, 0x1.a50e8d032888ep-1, 0x1.aa4880039b226p-1, 0x1.aeef2371dd852p-1,
    0x1.b319b59da3892p-1, 0x1.b6dac8fda1804p-1, 0x1.ba4163667c055p-1, 0x1.bd59ce0595db7p-1,
    0x1.c02e2e910c723p-1, 0x1.c2c6f9d8e971cp-1, 0x1.c52b4aa6e158ep-1, 0x1.c7612472dfb2ep-1,
    0x1.c96da731bfa1cp-1, 0x1.cb5537fe5326bp-1, 0x1.cd1ba151ba068p-1, 0x1.cec42cc5d4031p-1,
    0x1.d051b7d8eebdfp-1, 0x1.d1c6c4cb78105p-1, 0x1.d325886c1041cp-1, 0x1.d46ff57425279p-1,
    0x1.d5a7c5f20864cp-1, 0x1.d6ce832196529p-1, 0x1.d7e58bff7570cp-1, 0x1.d8ee1ad2ea59dp-1,
    0x1.d9e949dde7c29p-1, 0x1.dad817597610ap-1, 0x1.dbbb68dd1c184p-1, 0x1.dc940e4a19f9fp-1,
    0x1.dd62c44ea8647p-1, 0x1.de283691c223ap-1, 0x1.dee501950dd87p-1, 0x1.df99b45821000p-1,
    0x1.e046d1c66c97bp-1, 0x1.e0ecd1f7968c6p-1, 0x1.e18c2348befe7p-1, 0x1.e2252b5426929p-1,
    0x1.e2b847cbd0254p-1, 0x1.e345cf3b032ebp-1, 0x1.e3ce11b1fdda0p-1, 0x1.e451595ea88ddp-1,
    0x1.e4cfeb14b3dcbp-1, 0x1.e54a06c731debp-1, 0x1.e5bfe7f571dd3p-1, 0x1.e631c60ca6a25p-1,
    0x1.e69fd4bfaaa94p-1, 0x1.e70a4456084fbp-1, 0x1.e77141f345ae0p-1, 0x1.e7d4f7d752d84p-1,
    0x1.e8358d98dd10fp-1, 0x1.e893285a313bbp-1, 0x1.e8edeaf942f2cp-1, 0x1.e945f63b5b9b4p-1,
    0x1.e99b68f4e5297p-1, 0x1.e9ee602db6bbcp-1, 0x1.ea3ef7423d60fp-1, 0x1.ea8d4801d1156p-1,
    0x1.ead96aca7d05bp-1, 0x1.eb2376a27a46bp-1, 0x1.eb6b814f954c2p-1, 0x1.ebb19f6cb0574p-1,
    0x1.ebf5e47d8fbf2p-1, 0x1.ec38630118426p-1, 0x1.ec792c8223628p-1, 0x1.ecb851a70a246p-1,
    0x1.ecf5e24003441p-1, 0x1.ed31ed546f0dbp-1, 0x1.ed6c812f2872fp-1, 0x1.eda5ab69f0ac5p-1,
    0x1.eddd78f808ab3p-1, 0x1.ee13f63009c9fp-1, 0x1.ee492ed50d87cp-1, 0x1.ee7d2e1f32a6cp-1,
    0x1.eeaffec38cb17p-1, 0x1.eee1aafb89c06p-1, 0x1.ef123c8bd9483p-1, 0x1.ef41bccaddc3ep-1,
    0x1.ef7034a6b233ep-1, 0x1.ef9dacaacba30p-1, 0x1.efca2d053e2cbp-1, 0x1.eff5bd8bac638p-1,
    0x1.f02065bfe75a5p-1, 0x1.f04a2cd44516fp-1, 0x1.f07319afb2b4dp-1, 0x1.f09b32f18713ap-1,
    0x1.f0c27ef51a892p-1, 0x1.f0e903d527b1dp-1, 0x1.f10ec76ef92a1p-1, 0x1.f133cf6567abdp-1,
    0x1.f1582123abcb9p-1, 0x1.f17bc1e0064a5p-1, 0x1.f19eb69e41bf5p-1, 0x1.f1c1043210218p-1,
    0x1.f1e2af41468c7p-1, 0x1.f203bc45f96cfp-1, 0x1.f2242f907b1bdp-1, 0x1.f2440d493ec50p-1,
    0x1.f2635972a158ap-1, 0x1.f28217ea9a23bp-1, 0x1.f2a04c6c548f8p-1, 0x1.f2bdfa91b46f3p-1,
    0x1.f2db25d4c625ep-1, 0x1.f2f7d1911bdcbp-1, 0x1.f314010518e8bp-1, 0x1.f32fb7532c6e8p-1,
    0x1.f34af782fc3ddp-1, 0x1.f365c48280d0ap-1, 0x1.f380212713482p-1, 0x1.f39a102e6e34ap-1,
    0x1.f3b3943fa1e80p-1, 0x1.f3ccafebfd05ap-1, 0x1.f3e565afe9f7ap-1, 0x1.f3fdb7f3c1e6fp-1,
    0x1.f415a90c95c93p-1, 0x1.f42d3b3cee0e6p-1, 0x1.f44470b58170ap-1, 0x1.f45b4b95e35f0p-1,
    0x1.f471cded2a75fp-1, 0x1.f487f9ba8f70ep-1, 0x1.f49dd0ee04f9ep-1, 0x1.f4b35568c8b59p-1,
    0x1.f4c888fdede60p-1, 0x1.f4dd6d72e1f7bp-1, 0x1.f4f2047feb479p-1, 0x1.f5064fd0a26eap-1,
    0x1.f51a510466562p-1, 0x1.f52e09aecb5aep-1, 0x1.f5417b5805ba0p-1, 0x1.f554a77d4f862p-1,
    0x1.f5678f914a5a4p-1, 0x1.f57a34fc5cff0p-1, 0x1.f58c991d0d36ep-1, 0x1.f59ebd4855dcbp-1,
    0x1.f5b0a2c9f983bp-1, 0x1.f5c24ae4d1c23p-1, 0x1.f5d3b6d31b4eep-1, 0x1.f5e4e7c6bf16fp-1,
    0x1.f5f5dee998704p-1, 0x1.f6069d5db8897p-1, 0x1.f617243da7390p-1, 0x1.f627749ca1488p-1,
    0x1.f6378f86d45a3p-1, 0x1.f647760198836p-1, 0x1.f657290ba7b60p-1, 0x1.f666a99d5312ap-1,
    0x1.f675f8a8b6390p-1, 0x1.f6851719e8afap-1, 0x1.f69405d72d752p-1, 0x1.f6a2c5c120d1ep-1,
    0x1.f6b157b2e47a8p-1, 0x1.f6bfbc824a191p-1, 0x1.f6cdf4fffc4a5p-1, 0x1.f6dc01f7a6227p-1,
    0x1.f6e9e43019484p-1, 0x1.f6f79c6b72b4ep-1, 0x1.f7052b673e27ap-1, 0x1.f71291dc985bap-1,
    0x1.f71fd0805009bp-1, 0x1.f72ce80305c77p-1, 0x1.f739d9114acabp-1, 0x1.f746a453be9f8p-1,
    0x1.f7534a6f2bdabp-1, 0x1.f75fcc04a3d2ep-1, 0x1.f76c29b1996a2p-1, 0x1.f778640ffaf1ap-1,
    0x1.f7847bb64b2fdp-1, 0x1.f7907137b9932p-1, 0x1.f79c452439969p-1, 0x1.f7a7f80899638p-1,
    0x1.f7b38a6e97b56p-1, 0x1.f7befcdcf907cp-1, 0x1.f7ca4fd79c159p-1, 0x1.f7d583df8dafbp-1,
    0x1.f7e099731bf12p-1, 0x1.f7eb910de8d76p-1, 0x1.f7f66b28fc445p-1, 0x1.f801283ad56f1p-1,
    0x1.f80bc8b77bc8dp-1, 0x1.f8164d108f5c4p-1, 0x1.f820b5b558aa8p-1, 0x1.f82b0312d80a3p-1,
    0x1.f8353593d4905p-1, 0x1.f83f4da0ea827p-1, 0x1.f8494ba09959ep-1, 0x1.f8532ff7515afp-1,
    0x1.f85cfb0780c2dp-1, 0x1.f866ad31a0919p-1, 0x1.f87046d440f23p-1, 0x1.f879c84c15457p-1,
    0x1.f88331f3ffd0ep-1, 0x1.f88c84251d17bp-1, 0x1.f895bf36ceddep-1, 0x1.f89ee37ec6d9fp-1,
    0x1.f8a7f15111178p-1, 0x1.f8b0e9001e0e3p-1, 0x1.f8b9cadccc6dbp-1, 0x1.f8c2973672a34p-1,
    0x1.f8cb4e5ae8199p-1, 0x1.f8d3f0968e36ep-1, 0x1.f8dc7e3459194p-1, 0x1.f8e4f77dd8155p-1,
    0x1.f8ed5cbb3df86p-1, 0x1.f8f5ae3369103p-1, 0x1.f8fdec2beaf97p-1, 0x1.f90616e91038ap-1,
    0x1.f90e2eade79c9p-1, 0x1.f91633bc496f0p-1, 0x1.f91e2654de71dp-1, 0x1.f92606b726adcp-1,
    0x1.f92dd52180114p-1, 0x1.f93591d12ce2ap-1, 0x1.f93d3d025a063p-1, 0x1.f944d6f0251a1p-1,
    0x1.f94c5fd4a268ep-1, 0x1.f953d7e8e2b46p-1, 0x1.f95b3f64f8d95p-1, 0x1.f962967fff4e6p-1,
    0x1.f969dd701d7dfp-1, 0x1.f971146a8cfd0p-1, 0x1.f9783ba39e9ffp-1, 0x1.f97f534ebf6ddp-1,
    0x1.f9865b9e7d736p-1, 0x1.f98d54c48c775p-1, 0x1.f9943ef1ca8fbp-1, 0x1.f99b1a564499fp-1,
    0x1.f9a1e7213a965p-1, 0x1.f9a8a58123e7ep-1, 0x1.f9af55a3b3791p-1, 0x1.f9b5f7b5dbc62p-1,
    0x1.f9bc8be3d2cebp-1, 0x1.f9c3125915ed7p-1, 0x1.f9c98b406d996p-1, 0x1.f9cff6c3f10e2p-1,
    0x1.f9d6550d09dedp-1, 0x1.f9dca64477725p-1, 0x1.f9e2ea92526a1p-1, 0x1.f9e9221e0ff45p-1,
    0x1.f9ef4d0e8509fp-1, 0x1.f9f56b89e9990p-1, 0x1.f9fb7db5db9b3p-1, 0x1.fa0183b7621abp-1,
    0x1.fa077db2f024ap-1, 0x1.fa0d6bcc67a9bp-1, 0x1.fa134e271c4d9p-1, 0x1.fa1924e5d6260p-1};
static __device__ const float kMomCf[kMomN] = {
    0x0.0p+0f, 0x1.2083fe0000000p-2f, 0x1.bc75b60000000p-2f, 0x1.0fe7980000000p-1f,
    0x1.32931c0000000p-1f, 0x1.4c3fae0000000p-1f, 0x1.60131e0000000p-1f, 0x1.6fdf360000000p-1f,
    0x1.7cc5120000000p-1f, 0x1.8782220000000p-1f, 0x1.9097f20000000p-1f, 0x1.98623a0000000p-1f,
    0x1.9f23cc0000000p-1f, 0x1.a50e8e0000000p-1f, 0x1.aa48800000000p-1f, 0x1.aeef240000000p-1f,
    0x1.b319b60000000p-1f, 0x1.b6dac80000000p-1f, 0x1.ba41640000000p-1f, 0x1.bd59ce0000000p-1f,
    0x1.c02e2e0000000p-1f, 0x1.c2c6fa0000000p-1f, 0x1.c52b4a0000000p-1f, 0x1.c761240000000p-1f,
    0x1.c96da80000000p-1f, 0x1.cb55380000000p-1f, 0x1.cd1ba20000000p-1f, 0x1.cec42c0000000p-1f,
    0x1.d051b80000000p-1f, 0x1.d1c6c40000000p-1f, 0x1.d325880000000p-1f, 0x1.d46ff60000000p-1f,
    0x1.d5a7c60000000p-1f, 0x1.d6ce840000000p-1f, 0x1.d7e58c0000000p-1f, 0x1.d8ee1a0000000p-1f,
    0x1.d9e94a0000000p-1f, 0x1.dad8180000000p-1f, 0x1.dbbb680000000p-1f, 0x1.dc940e0000000p-1f,
    0x1.dd62c40000000p-1f, 0x1.de28360000000p-1f, 0x1.dee5020000000p-1f, 0x1.df99b40000000p-1f,
    0x1.e046d20000000p-1f, 0x1.e0ecd20000000p-1f, 0x1.e18c240000000p-1f, 0x1.e2252c0000000p-1f,
    0x1.e2b8480000000p-1f, 0x1.e345d00000000p-1f, 0x1.e3ce120000000p-1f, 0x1.e4515a0000000p-1f,
    0x1.e4cfec0000000p-1f, 0x1.e54a060000000p-1f, 0x1.e5bfe80000000p-1f, 0x1.e631c60000000p-1f,
    0x1.e69fd40000000p-1f, 0x1.e70a440000000p-1f, 0x1.e771420000000p-1f, 0x1.e7d4f80000000p-1f,
    0x1.e8358e0000000p-1f, 0x1.e893280000000p-1f, 0x1.e8edea0000000p-1f, 0x1.e945f60000000p-1f,
    0x1.e99b680000000p-1f, 0x1.e9ee600000000p-1f, 0x1.ea3ef80000000p-1f, 0x1.ea8d480000000p-1f,
    0x1.ead96a0000000p-1f, 0x1.eb23760000000p-1f, 0x1.eb6b820000000p-1f, 0x1.ebb1a00000000p-1f,
    0x1.ebf5e40000000p-1f, 0x1.ec38640000000p-1f, 0x1.ec792c0000000p-1f, 0x1.ecb8520000000p-1f,
    0x1.ecf5e20000000p-1f, 0x1.ed31ee0000000p-1f, 0x1.ed6c820000000p-1f, 0x1.eda5ac0000000p-1f,
    0x1.eddd780000000p-1f, 0x1.ee13f60000000p-1f, 0x1.ee492e0000000p-1f, 0x1.ee7d2e0000000p-1f,
    0x1.eeaffe0000000p-1f, 0x1.eee1aa0000000p-1f, 0x1.ef123c0000000p-1f, 0x1.ef41bc0000000p-1f,
    0x1.ef70340000000p-1f, 0x1.ef9dac0000000p-1f, 0x1.efca2e0000000p-1f, 0x1.eff5be0000000p-1f,
    0x1.f020660000000p-1f, 0x1.f04a2c0000000p-1f, 0x1.f0731a0000000p-1f, 0x1.f09b320000000p-1f,
    0x1.f0c27e0000000p-1f, 0x1.f0e9040000000p-1f, 0x1.f10ec80000000p-1f, 0x1.f133d00000000p-1f,
    0x1.f158220000000p-1f, 0x1.f17bc20000000p-1f, 0x1.f19eb60000000p-1f, 0x1.f1c1040000000p-1f,
    0x1.f1e2b00000000p-1f, 0x1.f203bc0000000p-1f, 0x1.f224300000000p-1f, 0x1.f2440e0000000p-1f,
    0x1.f2635a0000000p-1f, 0x1.f282180000000p-1f, 0x1.f2a04c0000000p-1f, 0x1.f2bdfa0000000p-1f,
    0x1.f2db260000000p-1f, 0x1.f2f7d20000000p-1f, 0x1.f314020000000p-1f, 0x1.f32fb80000000p-1f,
    0x1.f34af80000000p-1f, 0x1.f365c40000000p-1f, 0x1.f380220000000p-1f, 0x1.f39a100000000p-1f,
    0x1.f3b3940000000p-1f, 0x1.f3ccb00000000p-1f, 0x1.f3e5660000000p-1f, 0x1.f3fdb80000000p-1f,
    0x1.f415aa0000000p-1f, 0x1.f42d3c0000000p-1f, 0x1.f444700000000p-1f, 0x1.f45b4c0000000p-1f,
    0x1.f471ce0000000p-1f, 0x1.f487fa0000000p-1f, 0x1.f49dd00000000p-1f, 0x1.f4b3560000000p-1f,
    0x1.f4c8880000000p-1f, 0x1.f4dd6e0000000p-1f, 0x1.f4f2040000000p-1f, 0x1.f506500000000p-1f,
    0x1.f51a520000000p-1f, 0x1.f52e0a0000000p-1f, 0x1.f5417c0000000p-1f, 0x1.f554a80000000p-1f,
    0x1.f567900000000p-1f, 0x1.f57a340000000p-1f, 0x1.f58c9a0000000p-1f, 0x1.f59ebe0000000p-1f,
    0x1.f5b0a20000000p-1f, 0x1.f5c24a0000000p-1f, 0x1.f5d3b60000000p-1f, 0x1.f5e4e80000000p-1f,
    0x1.f5f5de0000000p-1f, 0x1.f6069e0000000p-1f, 0x1.f617240000000p-1f, 0x1.f627740000000p-1f,
    0x1.f637900000000p-1f, 0x1.f647760000000p-1f, 0x1.f6572a0000000p-1f, 0x1.f666aa0000000p-1f,
    0x1.f675f80000000p-1f, 0x1.f685180000000p-1f, 0x1.f694060000000p-1f, 0x1.f6a2c60000000p-1f,
    0x1.f6b1580000000p-1f, 0x1.f6bfbc0000000p-1f, 0x1.f6cdf40000000p-1f, 0x1.f6dc020000000p-1f,
    0x1.f6e9e40000000p-1f, 0x1.f6f79c0000000p-1f, 0x1.f7052c0000000p-1f, 0x1.f712920000000p-1f,
    0x1.f71fd00000000p-1f, 0x1.f72ce80000000p-1f, 0x1.f739da0000000p-1f, 0x1.f746a40000000p-1f,
    0x1.f7534a0000000p-1f, 0x1.f75fcc0000000p-1f, 0x1.f76c2a0000000p-1f, 0x1.f778640000000p-1f,
    0x1.f7847c0000000p-1f, 0x1.f790720000000p-1f, 0x1.f79c460000000p-1f, 0x1.f7a7f80000000p-1f,
    0x1.f7b38a0000000p-1f, 0x1.f7befc0000000p-1f, 0x1.f7ca500000000p-1f, 0x1.f7d5840000000p-1f,
    0x1.f7e09a0000000p-1f, 0x1.f7eb920000000p-1f, 0x1.f7f66c0000000p-1f, 0x1.f801280000000p-1f,
    0x1.f80bc80000000p-1f, 0x1.f8164e0000000p-1f, 0x1.f820b60000000p-1f, 0x1.f82b040000000p-1f,
    0x1.f835360000000p-1f, 0x1.f83f4e0000000p-1f, 0x1.f8494c0000000p-1f, 0x1.f853300000000p-1f,
    0x1.f85cfc0000000p-1f, 0x1.f866ae0000000p-1f, 0x1.f870460000000p-1f, 0x1.f879c80000000p-1f,
    0x1.f883320000000p-1f, 0x1.f88c840000000p-1f, 0x1.f895c00000000p-1f, 0x1.f89ee40000000p-1f,
    0x1.f8a7f20000000p-1f, 0x1.f8b0ea0000000p-1f, 0x1.f8b9ca0000000p-1f, 0x1.f8c2980000000p-1f,
    0x1.f8cb4e0000000p-1f, 0x1.f8d3f00000000p-1f, 0x1.f8dc7e0000000p-1f, 0x1.f8e4f80000000p-1f,
    0x1.f8ed5c0000000p-1f, 0x1.f8f5ae0000000p-1f, 0x1.f8fdec0000000p-1f, 0x1.f906160000000p-1f,
    0x1.f90e2e0000000p-1f, 0x1.f916340000000p-1f, 0x1.f91e260000000p-1f, 0x1.f926060000000p-1f,
    0x1.f92dd60000000p-1f, 0x1.f935920000000p-1f, 0x1.f93d3e0000000p-1f, 0x1.f944d60000000p-1f,
    0x1.f94c600000000p-1f, 0x1.f953d80000000p-1f, 0x1.f95b400000000p-1f, 0x1.f962960000000p-1f,
    0x1.f969de0000000p-1f, 0x1.f971140000000p-1f, 0x1.f9783c0000000p-1f, 0x1.f97f540000000p-1f,
    0x1.f9865c0000000p-1f, 0x1.f98d540000000p-1f, 0x1.f9943e0000000p-1f, 0x1.f99b1a0000000p-1f,
    0x1.f9a1e80000000p-1f, 0x1.f9a8a60000000p-1f, 0x1.f9af560000000p-1f, 0x1.f9b5f80000000p-1f,
    0x1.f9bc8c0000000p-1f, 0x1.f9c3120000000p-1f, 0x1.f9c98c0000000p-1f, 0x1.f9cff60000000p-1f,
    0x1.f9d6560000000p-1f, 0x1.f9dca60000000p-1f, 0x1.f9e2ea0000000p-1f, 0x1.f9e9220000000p-1f,
    0x1.f9ef4e0000000p-1f, 0x1.f9f56c0000000p-1f, 0x1.f9fb7e0000000p-1f, 0x1.fa01840000000p-1f,
    0x1.fa077e0000000p-1f, 0x1.fa0d6c0000000p-1f, 0x1.fa134e0000000p-1f, 0x1.fa19240000000p-1f};

// The state: sign bit set and the step count in the low word, or t (positive).
__device__ __forceinline__ double mom_start() { return -0.0; }
// The state after a step from `state` without a restart, and the step's coefficient.
__device__ __forceinline__ double mom_next(double state, double& c) {
    if (__double2hiint(state) < 0) {
        const int i = __double2loint(state);
        c = kMomC[i];
        return i + 1 < kMomN ? __hiloint2double((int)0x80000000, i + 1) : kMomEnd;
    }
    const double t = 0.5 * (1.0 + sqrt(1.0 + 4.0 * state * state));
    c = (state - 1.0) / t;
    return t;
}
__device__ __forceinline__ double mom_next(double state, float& c) {
    if (__double2hiint(state) < 0) {
        const int i = __double2loint(state);
        c = kMomCf[i];
        return i + 1 < kMomN ? __hiloint2double((int)0x80000000, i + 1) : kMomEnd;
    }
    double cd;
    const double t = mom_next(state, cd);
    c = (float)cd;
    return t;
}

}  // namespace kglm
