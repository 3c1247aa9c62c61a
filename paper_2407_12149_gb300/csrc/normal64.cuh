// normal64.cuh -- FP64 Box-Muller pairs from integer uniforms.
//
// FP64 issues at 1/64 of the FP32 rate on this GPU, so the sampler's FP64 normals are bound by
// the count of FP64 instructions.  A uniform here is (k + 1/2) 2^-b with an integer k, which
// lets integer instructions do the argument reductions and the conversions:
//  - -2 ln u: table-driven (P. T. P. Tang, "Table-driven implementation of the logarithm
//    function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): u = 2^e z, z in
//    [0.6875, 1.375), z inv_i = 1 + r with |r| < 2^-7.4 and the Taylor series of log(1 + r); the
//    cell next to 1 has inv = 1, so a small logarithm keeps its relative accuracy.  Cell and exponent
//    come from the high word less 0x3fe60000, its top mantissa bits and an arithmetic shift, as in
//    the log of Arm's Optimized Routines (table and polynomial are not that one's);
//  - its square root: Newton's iteration from the hardware reciprocal square root;
//  - sine and cosine of 2 pi u: the nearest odd multiple of 2 pi / 256 from a table, Taylor
//    series of the remainder, angle addition.
// 38 FP64 instructions a pair (14 + 6 + 2 + 16 below) instead of about 70 (log, sqrt, sincospi and
// the integer conversions).  Error relative to the radius against extended precision over 10^6 draws: rms
// 5.8e-17 (library functions 5.9e-17), largest 3.4e-16 (3.0e-16); 53-bit pairs rms 6.0e-17 and 3.7e-16
// (18e-17: their angle was rounded before the call).  tests/test_normal64_host.py bounds it by five
// roundings at the ends of every cell, next to 0 and 1, at ties and at the carry to u = 1.
// Measured (GB300): 31^2 FP64 chain, 8 cycles 584 -> 418 us; 1023^2 FP64, 2 cycles 1883 -> 1470 us.
#pragma once
#include <cuda_runtime.h>

namespace mgmc {
namespace n64 {

struct LogCell {
    double inv;      // 1 / c to 10 bits
    double hi, lo;   // -2 ln c
};
__device__ const LogCell kLog[128] = {
    {0x1.7340000000000p+0, 0x1.7c9e7703f8cfap-1, 0x1.55747742b9ed3p-55},
    {0x1.7140000000000p+0, 0x1.77166c744025ap-1, 0x1.99f82a5539353p-55},
    {0x1.6f40000000000p+0, 0x1.7186b11381193p-1, 0x1.3899df49cac22p-55},
    {0x1.6d00000000000p+0, 0x1.6b3bb2235943ep-1, -0x1.da856ccd987b3p-55},
    {0x1.6b00000000000p+0, 0x1.659b57303e1f3p-1, -0x1.f893d41c411f1p-55},
    {0x1.6900000000000p+0, 0x1.5ff3070a793d4p-1, -0x1.bc60efafc6f6ep-56},
    {0x1.6700000000000p+0, 0x1.5a42ab0f4cfe2p-1, -0x1.8ebcb7dee9a3dp-55},
    {0x1.6540000000000p+0, 0x1.5541aec91bfa0p-1, -0x1.6aadc72eeb980p-55},
    {0x1.6340000000000p+0, 0x1.4f81fe4763d00p-1, 0x1.84de5807b96b5p-55},
    {0x1.6140000000000p+0, 0x1.49b9feb7c176bp-1, 0x1.c58ab60d731b6p-59},
    {0x1.5f80000000000p+0, 0x1.44a41b463c47cp-1, -0x1.d70c8309edcfcp-55},
    {0x1.5d80000000000p+0, 0x1.3ecc460ef5f50p-1, -0x1.4313e09807affp-57},
    {0x1.5bc0000000000p+0, 0x1.39a8619f4518fp-1, -0x1.ae6c8cab0b631p-57},
    {0x1.59c0000000000p+0, 0x1.33c05f128dda9p-1, -0x1.06380e1a7d303p-56},
    {0x1.5800000000000p+0, 0x1.2e8e2bae11d31p-1, -0x1.8f4cdb95ebdf9p-55},
    {0x1.5640000000000p+0, 0x1.29552f81ff523p-1, 0x1.301771c407dbfp-55},
    {0x1.5480000000000p+0, 0x1.241558bfd1404p-1, -0x1.9bae06a5c872dp-64},
    {0x1.52c0000000000p+0, 0x1.1ece95528ae7bp-1, 0x1.84f64b5c47f86p-57},
    {0x1.5100000000000p+0, 0x1.1980d2dd4236fp-1, 0x1.9d3d1b0e4d147p-55},
    {0x1.4f40000000000p+0, 0x1.142bfeb9a0474p-1, -0x1.9e7a4a75619eep-55},
    {0x1.4d80000000000p+0, 0x1.0ed005f657da4p-1, 0x1.c56bd2abfe82ap-55},
    {0x1.4bc0000000000p+0, 0x1.096cd555917e6p-1, 0x1.8d20550a30eeep-55},
    {0x1.4a40000000000p+0, 0x1.04c8de1841e02p-1, -0x1.ae944b3ae19cfp-55},
    {0x1.4880000000000p+0, 0x1.feb0233e607ccp-2, 0x1.6e32d5e8c707fp-56},
    {0x1.46c0000000000p+0, 0x1.f3bfa934d6768p-2, -0x1.aad908df8942ep-57},
    {0x1.4540000000000p+0, 0x1.ea5349e23ac0ep-2, -0x1.b2ce30cd2d061p-57},
    {0x1.43c0000000000p+0, 0x1.e0dbc3d92aac9p-2, 0x1.9f8294df883d6p-58},
    {0x1.4200000000000p+0, 0x1.d5c216b4fbb91p-2, 0x1.6e443597e4d40p-56},
    {0x1.4080000000000p+0, 0x1.cc320c0176502p-2, 0x1.039a653793a85p-56},
    {0x1.3f00000000000p+0, 0x1.c2968558c18c1p-2, -0x1.73dee38a3fb6bp-56},
    {0x1.3d40000000000p+0, 0x1.b7526a22e4703p-2, 0x1.bf2e78548fd89p-56},
    {0x1.3bc0000000000p+0, 0x1.ad9da1f8273bfp-2, -0x1.6f9007e0a0d70p-56},
    {0x1.3a40000000000p+0, 0x1.a3dd04b93865fp-2, 0x1.a1366e2c5a7aap-56},
    {0x1.38c0000000000p+0, 0x1.9a10756988593p-2, -0x1.59dbd32f67a3ap-56},
    {0x1.3740000000000p+0, 0x1.9037d6a1804c3p-2, 0x1.ea57c1c8d979fp-56},
    {0x1.35c0000000000p+0, 0x1.86530a8c70cc6p-2, -0x1.3cd2c57073be9p-57},
    {0x1.3480000000000p+0, 0x1.7e0afd630c274p-2, -0x1.83e270efcc373p-57},
    {0x1.3300000000000p+0, 0x1.740f8f54037a5p-2, -0x1.b264062a84cdbp-57},
    {0x1.3180000000000p+0, 0x1.6a079d0f7aad2p-2, -0x1.eedcbac2a7f18p-61},
    {0x1.3000000000000p+0, 0x1.5ff3070a793d4p-2, -0x1.bc60efafc6f6ep-57},
    {0x1.2ec0000000000p+0, 0x1.5782cb309162ep-2, -0x1.8d45e51106d5ep-57},
    {0x1.2d40000000000p+0, 0x1.4d56b5798ec03p-2, -0x1.ffa95a6aaa4edp-57},
    {0x1.2c00000000000p+0, 0x1.44d2b6ccb7d1ep-2, 0x1.9f4f6543e1f88p-56},
    {0x1.2a80000000000p+0, 0x1.3a8eb2d31a376p-2, -0x1.220a8abf098f4p-59},
    {0x1.2940000000000p+0, 0x1.31f693eb19966p-2, 0x1.b234b8d209720p-57},
    {0x1.27c0000000000p+0, 0x1.279a300ab4f7ap-2, 0x1.95991a883feffp-58},
    {0x1.2680000000000p+0, 0x1.1eed90e2dc2c3p-2, -0x1.4e47b44db8540p-56},
    {0x1.2540000000000p+0, 0x1.16377fb124192p-2, -0x1.e540be89c1eaap-58},
    {0x1.2400000000000p+0, 0x1.0d77e7cd08e59p-2, 0x1.9a5dc5e9030acp-56},
    {0x1.22c0000000000p+0, 0x1.04aeb449f66bfp-2, -0x1.6f9a332ca3851p-56},
    {0x1.2140000000000p+0, 0x1.f42dba3a22cedp-3, 0x1.2334824fcc6ebp-57},
    {0x1.2000000000000p+0, 0x1.e27076e2af2e6p-3, -0x1.61578001e0162p-59},
    {0x1.1ec0000000000p+0, 0x1.d09f72b4c4824p-3, 0x1.80006a9c6606cp-57},
    {0x1.1d80000000000p+0, 0x1.beba818146765p-3, -0x1.e2db7c7d5a130p-57},
    {0x1.1c40000000000p+0, 0x1.acc17684332acp-3, 0x1.f17d2016d0e25p-58},
    {0x1.1b00000000000p+0, 0x1.9ab42462033adp-3, -0x1.2099e1c184e8ep-58},
    {0x1.1a00000000000p+0, 0x1.8c345d6319b21p-3, -0x1.4a697ab3424a9p-60},
    {0x1.18c0000000000p+0, 0x1.7a0216f649e12p-3, 0x1.32861063fdf57p-57},
    {0x1.1780000000000p+0, 0x1.67bb0726ec0fcp-3, -0x1.b692c214ddbecp-57},
    {0x1.1640000000000p+0, 0x1.555efe40b50b5p-3, -0x1.a1cde5c772a1ap-57},
    {0x1.1500000000000p+0, 0x1.42edcbea646f0p-3, 0x1.ddd4f935996c9p-58},
    {0x1.1400000000000p+0, 0x1.341d7961bd1d1p-3, -0x1.b599f227becbbp-57},
    {0x1.12c0000000000p+0, 0x1.2185b3b75a1cep-3, 0x1.d81c3373f1357p-57},
    {0x1.11c0000000000p+0, 0x1.129644402e2acp-3, 0x1.122b956232089p-57},
    {0x1.1080000000000p+0, 0x1.ffae9119b9303p-4, 0x1.ba13162a9c446p-59},
    {0x1.0f40000000000p+0, 0x1.da0478be39253p-4, -0x1.c270480fd528ep-59},
    {0x1.0e40000000000p+0, 0x1.bbc2bfc44f417p-4, 0x1.e5bafa0943c21p-59},
    {0x1.0d40000000000p+0, 0x1.9d644fdffa279p-4, 0x1.0539a473b598bp-59},
    {0x1.0c00000000000p+0, 0x1.77458f632dcfcp-4, 0x1.18d3ca87b9296p-58},
    {0x1.0b00000000000p+0, 0x1.58a5bafc8e4d5p-4, -0x1.ce55c2b4e2b72p-58},
    {0x1.09c0000000000p+0, 0x1.32348c7001697p-4, -0x1.237a70db06b41p-59},
    {0x1.08c0000000000p+0, 0x1.13523785971f3p-4, -0x1.876e3f4b360c5p-58},
    {0x1.07c0000000000p+0, 0x1.e8a3ee30cdcacp-5, 0x1.7086b1c00b395p-62},
    {0x1.06c0000000000p+0, 0x1.aa6721ee835aap-5, -0x1.4a3a50b6c5621p-60},
    {0x1.0580000000000p+0, 0x1.5c45a51b8d389p-5, -0x1.b10b6c3ec21b4p-59},
    {0x1.0480000000000p+0, 0x1.1d7f7eb9eebe7p-5, -0x1.d41fe63d2dbf9p-60},
    {0x1.0380000000000p+0, 0x1.bcf712c74384cp-6, -0x1.f6842688f499ap-61},
    {0x1.0280000000000p+0, 0x1.3e7295d25a7d9p-6, -0x1.ff29a11443a06p-64},
    {0x1.0180000000000p+0, 0x1.7ee11ebd82e94p-7, -0x1.61e96e2fc5d90p-61},
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0},
    {0x1.fe00000000000p-1, -0x1.0080559588b35p-7, -0x1.f96638cf63677p-61},
    {0x1.fa00000000000p-1, -0x1.82448a388a2aap-6, -0x1.04b16137f09a0p-61},
    {0x1.f600000000000p-1, -0x1.432a925980cc1p-5, 0x1.8cdaf39004192p-59},
    {0x1.f280000000000p-1, -0x1.b5cc258b718e6p-5, -0x1.1b8afbfe81965p-61},
    {0x1.ee80000000000p-1, -0x1.1ce5a62bc353ap-4, 0x1.c39390333b61cp-58},
    {0x1.eb00000000000p-1, -0x1.5715c4c03ceefp-4, 0x1.bbf88ec501b56p-60},
    {0x1.e780000000000p-1, -0x1.91b073efd7314p-4, -0x1.d60449ab527bfp-60},
    {0x1.e380000000000p-1, -0x1.d52ed6405d86fp-4, -0x1.16aeb2214c8c0p-58},
    {0x1.e000000000000p-1, -0x1.08598b59e3a07p-3, 0x1.dd7009902bf32p-57},
    {0x1.dc80000000000p-1, -0x1.26536c3d8c369p-3, -0x1.d604be2dd16f0p-57},
    {0x1.d900000000000p-1, -0x1.4485e03dbdfadp-3, -0x1.1ba349aadbc6ep-57},
    {0x1.d600000000000p-1, -0x1.5e95a4d9791cbp-3, -0x1.f38745c5c450ap-57},
    {0x1.d280000000000p-1, -0x1.7d33687c293c9p-3, 0x1.cf063e63e7075p-57},
    {0x1.cf00000000000p-1, -0x1.9c0c32d4d2548p-3, -0x1.fb0be3ccc1532p-58},
    {0x1.cc00000000000p-1, -0x1.b6ac88dad5b1cp-3, 0x1.0057eed1ca59fp-58},
    {0x1.c880000000000p-1, -0x1.d5f55659210e2p-3, -0x1.ce60c2a34a8fbp-58},
    {0x1.c580000000000p-1, -0x1.f0f70cdd992e3p-3, -0x1.f6c272c1dca71p-59},
    {0x1.c280000000000p-1, -0x1.06135354d4b18p-2, -0x1.18a0d03ba5397p-57},
    {0x1.bf80000000000p-1, -0x1.13c2605c398c3p-2, 0x1.fdd94f6508b88p-56},
    {0x1.bc80000000000p-1, -0x1.2188fd9807263p-2, 0x1.e7f50c701268fp-59},
    {0x1.b980000000000p-1, -0x1.2f677cbbc0a96p-2, 0x1.9fbd3e17e5527p-56},
    {0x1.b680000000000p-1, -0x1.3d5e3126bc27fp-2, -0x1.97c284b6258aap-56},
    {0x1.b380000000000p-1, -0x1.4b6d6fefe22a4p-2, -0x1.767ab73ca8d5ep-56},
    {0x1.b080000000000p-1, -0x1.59958ff1d52f1p-2, -0x1.f4d12c6bf5a87p-56},
    {0x1.ad80000000000p-1, -0x1.67d6e9d785771p-2, 0x1.10614e0da5fb8p-56},
    {0x1.ab00000000000p-1, -0x1.73cb9074fd14dp-2, 0x1.521a000b4cf01p-56},
    {0x1.a800000000000p-1, -0x1.823c16551a3c2p-2, 0x1.1232ce70be781p-56},
    {0x1.a580000000000p-1, -0x1.8e588ebac2dbfp-2, 0x1.46a9a5dd7ff12p-56},
    {0x1.a300000000000p-1, -0x1.9a8778debaa38p-2, -0x1.f47dfd871f87fp-56},
    {0x1.a000000000000p-1, -0x1.a93ed3c8ad9e3p-2, -0x1.bcafa9de97203p-56},
    {0x1.9d80000000000p-1, -0x1.b5971a213acdbp-2, 0x1.e2f8aadc42f8fp-56},
    {0x1.9b00000000000p-1, -0x1.c2028ab17f9b4p-2, -0x1.f11aa3853a5f1p-56},
    {0x1.9880000000000p-1, -0x1.ce816157f1988p-2, 0x1.5744132a297b0p-57},
    {0x1.9600000000000p-1, -0x1.db13db0d48940p-2, -0x1.aa11d49f96cb9p-57},
    {0x1.9380000000000p-1, -0x1.e7ba35eb77e2ap-2, -0x1.11dc86c9b7564p-58},
    {0x1.9100000000000p-1, -0x1.f474b134df229p-2, 0x1.27c77ded76aadp-57},
    {0x1.8e80000000000p-1, -0x1.00a1c6adda473p-1, -0x1.8d688b9e17a8ap-55},
    {0x1.8c00000000000p-1, -0x1.07138604d5862p-1, -0x1.cdb16ed4e9138p-55},
    {0x1.8980000000000p-1, -0x1.0d8fb813eb1efp-1, 0x1.cdde2b0172bd5p-55},
    {0x1.8780000000000p-1, -0x1.12c77cd00713bp-1, -0x1.4a4508fbcba26p-56},
    {0x1.8500000000000p-1, -0x1.1956d3b9bc2fap-1, -0x1.7b9d68d50a15dp-55},
    {0x1.8280000000000p-1, -0x1.1ff0fe7cf47a7p-1, -0x1.5b513ff0c1450p-55},
    {0x1.8080000000000p-1, -0x1.25410494e56c7p-1, -0x1.7ac0ef77f252ap-55},
    {0x1.7e00000000000p-1, -0x1.2bef07cdc9354p-1, 0x1.82dad7fd86088p-55},
    {0x1.7c00000000000p-1, -0x1.314f1e1d35ce4p-1, 0x1.3d69909e5c3dcp-55},
    {0x1.7980000000000p-1, -0x1.3811728564cb2p-1, 0x1.e493a0702b236p-56},
    {0x1.7780000000000p-1, -0x1.3d81fb5946dbap-1, -0x1.c1eab1642e36dp-55},
    {0x1.7580000000000p-1, -0x1.42f9f3ff62642p-1, 0x1.bbf082ccabbaep-55},
};
// -2 e ln 2, e = 0, -1, ..
__device__ const double kExp[56] = {
    0x0.0p+0,
    0x1.62e42fefa39efp+0,
    0x1.62e42fefa39efp+1,
    0x1.0a2b23f3bab73p+2,
    0x1.62e42fefa39efp+2,
    0x1.bb9d3beb8c86bp+2,
    0x1.0a2b23f3bab73p+3,
    0x1.3687a9f1af2b1p+3,
    0x1.62e42fefa39efp+3,
    0x1.8f40b5ed9812dp+3,
    0x1.bb9d3beb8c86bp+3,
    0x1.e7f9c1e980fa9p+3,
    0x1.0a2b23f3bab73p+4,
    0x1.205966f2b4f12p+4,
    0x1.3687a9f1af2b1p+4,
    0x1.4cb5ecf0a9650p+4,
    0x1.62e42fefa39efp+4,
    0x1.791272ee9dd8ep+4,
    0x1.8f40b5ed9812dp+4,
    0x1.a56ef8ec924ccp+4,
    0x1.bb9d3beb8c86bp+4,
    0x1.d1cb7eea86c0ap+4,
    0x1.e7f9c1e980fa9p+4,
    0x1.fe2804e87b348p+4,
    0x1.0a2b23f3bab73p+5,
    0x1.1542457337d43p+5,
    0x1.205966f2b4f12p+5,
    0x1.2b708872320e2p+5,
    0x1.3687a9f1af2b1p+5,
    0x1.419ecb712c481p+5,
    0x1.4cb5ecf0a9650p+5,
    0x1.57cd0e7026820p+5,
    0x1.62e42fefa39efp+5,
    0x1.6dfb516f20bbfp+5,
    0x1.791272ee9dd8ep+5,
    0x1.8429946e1af5ep+5,
    0x1.8f40b5ed9812dp+5,
    0x1.9a57d76d152fdp+5,
    0x1.a56ef8ec924ccp+5,
    0x1.b0861a6c0f69cp+5,
    0x1.bb9d3beb8c86bp+5,
    0x1.c6b45d6b09a3ap+5,
    0x1.d1cb7eea86c0ap+5,
    0x1.dce2a06a03dd9p+5,
    0x1.e7f9c1e980fa9p+5,
    0x1.f310e368fe178p+5,
    0x1.fe2804e87b348p+5,
    0x1.049f9333fc28cp+6,
    0x1.0a2b23f3bab73p+6,
    0x1.0fb6b4b37945bp+6,
    0x1.1542457337d43p+6,
    0x1.1acdd632f662bp+6,
    0x1.205966f2b4f12p+6,
    0x1.25e4f7b2737fap+6,
    0x1.2b708872320e2p+6,
    0x1.30fc1931f09cap+6,
};
// cos and sin of 2 pi (2 k + 1) / 256: leading and trailing parts
struct TrigCell {
    double2 hi, lo;
};
__device__ const TrigCell kTrig[128] = {
    {{0x1.ffd886084cd0dp-1, 0x1.92155f7a3667ep-6}, {-0x1.1354d4556e4cbp-55, -0x1.b1d63091a0130p-64}},
    {{0x1.fe9cdad01883ap-1, 0x1.2d52092ce19f6p-4}, {0x1.521ecd0c67e35p-57, -0x1.9a088a8bf6b2cp-59}},
    {{0x1.fc26470e19fd3p-1, 0x1.f564e56a9730ep-4}, {0x1.1ec8668ecaceep-55, 0x1.a2704729ae56dp-59}},
    {{0x1.f8764fa714ba9p-1, 0x1.5e214448b3fc6p-3}, {0x1.ab256778ffcb6p-56, 0x1.531ff779ddac6p-57}},
    {{0x1.f38f3ac64e589p-1, 0x1.c0b826a7e4f63p-3}, {-0x1.d7bafb51f72e6p-56, -0x1.af1439e521935p-62}},
    {{0x1.ed740e7684963p-1, 0x1.111d262b1f677p-2}, {0x1.e82c791f59cc2p-56, 0x1.824c20ab7aa9ap-56}},
    {{0x1.e6288ec48e112p-1, 0x1.4135c94176601p-2}, {-0x1.16b56f2847754p-57, 0x1.0c97c4afa2518p-56}},
    {{0x1.ddb13b6ccc23cp-1, 0x1.7088530fa459fp-2}, {0x1.83c37c6107db3p-55, -0x1.44b19e0864c5dp-56}},
    {{0x1.d4134d14dc93ap-1, 0x1.9ef7943a8ed8ap-2}, {-0x1.4ef5295d25af2p-55, 0x1.6da81290bdbabp-57}},
    {{0x1.c954b213411f5p-1, 0x1.cc66e9931c45ep-2}, {-0x1.2fb761e946603p-58, 0x1.6850e59c37f8fp-58}},
    {{0x1.bd7c0ac6f952ap-1, 0x1.f8ba4dbf89abap-2}, {-0x1.825a732ac700ap-55, -0x1.2ec1fc1b776b8p-60}},
    {{0x1.b090a58150200p-1, 0x1.11eb3541b4b23p-1}, {-0x1.926da300ffccep-55, -0x1.ef23b69abe4f1p-55}},
    {{0x1.a29a7a0462782p-1, 0x1.26d054cdd12dfp-1}, {-0x1.128bb015df175p-56, -0x1.5da743ef3770cp-55}},
    {{0x1.93a22499263fbp-1, 0x1.3affa292050b9p-1}, {0x1.3d419a920df0bp-55, 0x1.e3e25e3954964p-56}},
    {{0x1.83b0e0bff976ep-1, 0x1.4e6cabbe3e5e9p-1}, {-0x1.6f420f8ea3475p-56, 0x1.3c293edceb327p-57}},
    {{0x1.72d0837efff96p-1, 0x1.610b7551d2cdfp-1}, {0x1.0d4ef0f1d915cp-55, -0x1.251b352ff2a37p-56}},
    {{0x1.610b7551d2cdfp-1, 0x1.72d0837efff96p-1}, {-0x1.251b352ff2a37p-56, 0x1.0d4ef0f1d915cp-55}},
    {{0x1.4e6cabbe3e5e9p-1, 0x1.83b0e0bff976ep-1}, {0x1.3c293edceb327p-57, -0x1.6f420f8ea3475p-56}},
    {{0x1.3affa292050b9p-1, 0x1.93a22499263fbp-1}, {0x1.e3e25e3954964p-56, 0x1.3d419a920df0bp-55}},
    {{0x1.26d054cdd12dfp-1, 0x1.a29a7a0462782p-1}, {-0x1.5da743ef3770cp-55, -0x1.128bb015df175p-56}},
    {{0x1.11eb3541b4b23p-1, 0x1.b090a58150200p-1}, {-0x1.ef23b69abe4f1p-55, -0x1.926da300ffccep-55}},
    {{0x1.f8ba4dbf89abap-2, 0x1.bd7c0ac6f952ap-1}, {-0x1.2ec1fc1b776b8p-60, -0x1.825a732ac700ap-55}},
    {{0x1.cc66e9931c45ep-2, 0x1.c954b213411f5p-1}, {0x1.6850e59c37f8fp-58, -0x1.2fb761e946603p-58}},
    {{0x1.9ef7943a8ed8ap-2, 0x1.d4134d14dc93ap-1}, {0x1.6da81290bdbabp-57, -0x1.4ef5295d25af2p-55}},
    {{0x1.7088530fa459fp-2, 0x1.ddb13b6ccc23cp-1}, {-0x1.44b19e0864c5dp-56, 0x1.83c37c6107db3p-55}},
    {{0x1.4135c94176601p-2, 0x1.e6288ec48e112p-1}, {0x1.0c97c4afa2518p-56, -0x1.16b56f2847754p-57}},
    {{0x1.111d262b1f677p-2, 0x1.ed740e7684963p-1}, {0x1.824c20ab7aa9ap-56, 0x1.e82c791f59cc2p-56}},
    {{0x1.c0b826a7e4f63p-3, 0x1.f38f3ac64e589p-1}, {-0x1.af1439e521935p-62, -0x1.d7bafb51f72e6p-56}},
    {{0x1.5e214448b3fc6p-3, 0x1.f8764fa714ba9p-1}, {0x1.531ff779ddac6p-57, 0x1.ab256778ffcb6p-56}},
    {{0x1.f564e56a9730ep-4, 0x1.fc26470e19fd3p-1}, {0x1.a2704729ae56dp-59, 0x1.1ec8668ecaceep-55}},
    {{0x1.2d52092ce19f6p-4, 0x1.fe9cdad01883ap-1}, {-0x1.9a088a8bf6b2cp-59, 0x1.521ecd0c67e35p-57}},
    {{0x1.92155f7a3667ep-6, 0x1.ffd886084cd0dp-1}, {-0x1.b1d63091a0130p-64, -0x1.1354d4556e4cbp-55}},
    {{-0x1.92155f7a3667ep-6, 0x1.ffd886084cd0dp-1}, {0x1.b1d63091a0130p-64, -0x1.1354d4556e4cbp-55}},
    {{-0x1.2d52092ce19f6p-4, 0x1.fe9cdad01883ap-1}, {0x1.9a088a8bf6b2cp-59, 0x1.521ecd0c67e35p-57}},
    {{-0x1.f564e56a9730ep-4, 0x1.fc26470e19fd3p-1}, {-0x1.a2704729ae56dp-59, 0x1.1ec8668ecaceep-55}},
    {{-0x1.5e214448b3fc6p-3, 0x1.f8764fa714ba9p-1}, {-0x1.531ff779ddac6p-57, 0x1.ab256778ffcb6p-56}},
    {{-0x1.c0b826a7e4f63p-3, 0x1.f38f3ac64e589p-1}, {0x1.af1439e521935p-62, -0x1.d7bafb51f72e6p-56}},
    {{-0x1.111d262b1f677p-2, 0x1.ed740e7684963p-1}, {-0x1.824c20ab7aa9ap-56, 0x1.e82c791f59cc2p-56}},
    {{-0x1.4135c94176601p-2, 0x1.e6288ec48e112p-1}, {-0x1.0c97c4afa2518p-56, -0x1.16b56f2847754p-57}},
    {{-0x1.7088530fa459fp-2, 0x1.ddb13b6ccc23cp-1}, {0x1.44b19e0864c5dp-56, 0x1.83c37c6107db3p-55}},
    {{-0x1.9ef7943a8ed8ap-2, 0x1.d4134d14dc93ap-1}, {-0x1.6da81290bdbabp-57, -0x1.4ef5295d25af2p-55}},
    {{-0x1.cc66e9931c45ep-2, 0x1.c954b213411f5p-1}, {-0x1.6850e59c37f8fp-58, -0x1.2fb761e946603p-58}},
    {{-0x1.f8ba4dbf89abap-2, 0x1.bd7c0ac6f952ap-1}, {0x1.2ec1fc1b776b8p-60, -0x1.825a732ac700ap-55}},
    {{-0x1.11eb3541b4b23p-1, 0x1.b090a58150200p-1}, {0x1.ef23b69abe4f1p-55, -0x1.926da300ffccep-55}},
    {{-0x1.26d054cdd12dfp-1, 0x1.a29a7a0462782p-1}, {0x1.5da743ef3770cp-55, -0x1.128bb015df175p-56}},
    {{-0x1.3affa292050b9p-1, 0x1.93a22499263fbp-1}, {-0x1.e3e25e3954964p-56, 0x1.3d419a920df0bp-55}},
    {{-0x1.4e6cabbe3e5e9p-1, 0x1.83b0e0bff976ep-1}, {-0x1.3c293edceb327p-57, -0x1.6f420f8ea3475p-56}},
    {{-0x1.610b7551d2cdfp-1, 0x1.72d0837efff96p-1}, {0x1.251b352ff2a37p-56, 0x1.0d4ef0f1d915cp-55}},
    {{-0x1.72d0837efff96p-1, 0x1.610b7551d2cdfp-1}, {-0x1.0d4ef0f1d915cp-55, -0x1.251b352ff2a37p-56}},
    {{-0x1.83b0e0bff976ep-1, 0x1.4e6cabbe3e5e9p-1}, {0x1.6f420f8ea3475p-56, 0x1.3c293edceb327p-57}},
    {{-0x1.93a22499263fbp-1, 0x1.3affa292050b9p-1}, {-0x1.3d419a920df0bp-55, 0x1.e3e25e3954964p-56}},
    {{-0x1.a29a7a0462782p-1, 0x1.26d054cdd12dfp-1}, {0x1.128bb015df175p-56, -0x1.5da743ef3770cp-55}},
    {{-0x1.b090a58150200p-1, 0x1.11eb3541b4b23p-1}, {0x1.926da300ffccep-55, -0x1.ef23b69abe4f1p-55}},
    {{-0x1.bd7c0ac6f952ap-1, 0x1.f8ba4dbf89abap-2}, {0x1.825a732ac700ap-55, -0x1.2ec1fc1b776b8p-60}},
    {{-0x1.c954b213411f5p-1, 0x1.cc66e9931c45ep-2}, {0x1.2fb761e946603p-58, 0x1.6850e59c37f8fp-58}},
    {{-0x1.d4134d14dc93ap-1, 0x1.9ef7943a8ed8ap-2}, {0x1.4ef5295d25af2p-55, 0x1.6da81290bdbabp-57}},
    {{-0x1.ddb13b6ccc23cp-1, 0x1.7088530fa459fp-2}, {-0x1.83c37c6107db3p-55, -0x1.44b19e0864c5dp-56}},
    {{-0x1.e6288ec48e112p-1, 0x1.4135c94176601p-2}, {0x1.16b56f2847754p-57, 0x1.0c97c4afa2518p-56}},
    {{-0x1.ed740e7684963p-1, 0x1.111d262b1f677p-2}, {-0x1.e82c791f59cc2p-56, 0x1.824c20ab7aa9ap-56}},
    {{-0x1.f38f3ac64e589p-1, 0x1.c0b826a7e4f63p-3}, {0x1.d7bafb51f72e6p-56, -0x1.af1439e521935p-62}},
    {{-0x1.f8764fa714ba9p-1, 0x1.5e214448b3fc6p-3}, {-0x1.ab256778ffcb6p-56, 0x1.531ff779ddac6p-57}},
    {{-0x1.fc26470e19fd3p-1, 0x1.f564e56a9730ep-4}, {-0x1.1ec8668ecaceep-55, 0x1.a2704729ae56dp-59}},
    {{-0x1.fe9cdad01883ap-1, 0x1.2d52092ce19f6p-4}, {-0x1.521ecd0c67e35p-57, -0x1.9a088a8bf6b2cp-59}},
    {{-0x1.ffd886084cd0dp-1, 0x1.92155f7a3667ep-6}, {0x1.1354d4556e4cbp-55, -0x1.b1d63091a0130p-64}},
    {{-0x1.ffd886084cd0dp-1, -0x1.92155f7a3667ep-6}, {0x1.1354d4556e4cbp-55, 0x1.b1d63091a0130p-64}},
    {{-0x1.fe9cdad01883ap-1, -0x1.2d52092ce19f6p-4}, {-0x1.521ecd0c67e35p-57, 0x1.9a088a8bf6b2cp-59}},
    {{-0x1.fc26470e19fd3p-1, -0x1.f564e56a9730ep-4}, {-0x1.1ec8668ecaceep-55, -0x1.a2704729ae56dp-59}},
    {{-0x1.f8764fa714ba9p-1, -0x1.5e214448b3fc6p-3}, {-0x1.ab256778ffcb6p-56, -0x1.531ff779ddac6p-57}},
    {{-0x1.f38f3ac64e589p-1, -0x1.c0b826a7e4f63p-3}, {0x1.d7bafb51f72e6p-56, 0x1.af1439e521935p-62}},
    {{-0x1.ed740e7684963p-1, -0x1.111d262b1f677p-2}, {-0x1.e82c791f59cc2p-56, -0x1.824c20ab7aa9ap-56}},
    {{-0x1.e6288ec48e112p-1, -0x1.4135c94176601p-2}, {0x1.16b56f2847754p-57, -0x1.0c97c4afa2518p-56}},
    {{-0x1.ddb13b6ccc23cp-1, -0x1.7088530fa459fp-2}, {-0x1.83c37c6107db3p-55, 0x1.44b19e0864c5dp-56}},
    {{-0x1.d4134d14dc93ap-1, -0x1.9ef7943a8ed8ap-2}, {0x1.4ef5295d25af2p-55, -0x1.6da81290bdbabp-57}},
    {{-0x1.c954b213411f5p-1, -0x1.cc66e9931c45ep-2}, {0x1.2fb761e946603p-58, -0x1.6850e59c37f8fp-58}},
    {{-0x1.bd7c0ac6f952ap-1, -0x1.f8ba4dbf89abap-2}, {0x1.825a732ac700ap-55, 0x1.2ec1fc1b776b8p-60}},
    {{-0x1.b090a58150200p-1, -0x1.11eb3541b4b23p-1}, {0x1.926da300ffccep-55, 0x1.ef23b69abe4f1p-55}},
    {{-0x1.a29a7a0462782p-1, -0x1.26d054cdd12dfp-1}, {0x1.128bb015df175p-56, 0x1.5da743ef3770cp-55}},
    {{-0x1.93a22499263fbp-1, -0x1.3affa292050b9p-1}, {-0x1.3d419a920df0bp-55, -0x1.e3e25e3954964p-56}},
    {{-0x1.83b0e0bff976ep-1, -0x1.4e6cabbe3e5e9p-1}, {0x1.6f420f8ea3475p-56, -0x1.3c293edceb327p-57}},
    {{-0x1.72d0837efff96p-1, -0x1.610b7551d2cdfp-1}, {-0x1.0d4ef0f1d915cp-55, 0x1.251b352ff2a37p-56}},
    {{-0x1.610b7551d2cdfp-1, -0x1.72d0837efff96p-1}, {0x1.251b352ff2a37p-56, -0x1.0d4ef0f1d915cp-55}},
    {{-0x1.4e6cabbe3e5e9p-1, -0x1.83b0e0bff976ep-1}, {-0x1.3c293edceb327p-57, 0x1.6f420f8ea3475p-56}},
    {{-0x1.3affa292050b9p-1, -0x1.93a22499263fbp-1}, {-0x1.e3e25e3954964p-56, -0x1.3d419a920df0bp-55}},
    {{-0x1.26d054cdd12dfp-1, -0x1.a29a7a0462782p-1}, {0x1.5da743ef3770cp-55, 0x1.128bb015df175p-56}},
    {{-0x1.11eb3541b4b23p-1, -0x1.b090a58150200p-1}, {0x1.ef23b69abe4f1p-55, 0x1.926da300ffccep-55}},
    {{-0x1.f8ba4dbf89abap-2, -0x1.bd7c0ac6f952ap-1}, {0x1.2ec1fc1b776b8p-60, 0x1.825a732ac700ap-55}},
    {{-0x1.cc66e9931c45ep-2, -0x1.c954b213411f5p-1}, {-0x1.6850e59c37f8fp-58, 0x1.2fb761e946603p-58}},
    {{-0x1.9ef7943a8ed8ap-2, -0x1.d4134d14dc93ap-1}, {-0x1.6da81290bdbabp-57, 0x1.4ef5295d25af2p-55}},
    {{-0x1.7088530fa459fp-2, -0x1.ddb13b6ccc23cp-1}, {0x1.44b19e0864c5dp-56, -0x1.83c37c6107db3p-55}},
    {{-0x1.4135c94176601p-2, -0x1.e6288ec48e112p-1}, {-0x1.0c97c4afa2518p-56, 0x1.16b56f2847754p-57}},
    {{-0x1.111d262b1f677p-2, -0x1.ed740e7684963p-1}, {-0x1.824c20ab7aa9ap-56, -0x1.e82c791f59cc2p-56}},
    {{-0x1.c0b826a7e4f63p-3, -0x1.f38f3ac64e589p-1}, {0x1.af1439e521935p-62, 0x1.d7bafb51f72e6p-56}},
    {{-0x1.5e214448b3fc6p-3, -0x1.f8764fa714ba9p-1}, {-0x1.531ff779ddac6p-57, -0x1.ab256778ffcb6p-56}},
    {{-0x1.f564e56a9730ep-4, -0x1.fc26470e19fd3p-1}, {-0x1.a2704729ae56dp-59, -0x1.1ec8668ecaceep-55}},
    {{-0x1.2d52092ce19f6p-4, -0x1.fe9cdad01883ap-1}, {0x1.9a088a8bf6b2cp-59, -0x1.521ecd0c67e35p-57}},
    {{-0x1.92155f7a3667ep-6, -0x1.ffd886084cd0dp-1}, {0x1.b1d63091a0130p-64, 0x1.1354d4556e4cbp-55}},
    {{0x1.92155f7a3667ep-6, -0x1.ffd886084cd0dp-1}, {-0x1.b1d63091a0130p-64, 0x1.1354d4556e4cbp-55}},
    {{0x1.2d52092ce19f6p-4, -0x1.fe9cdad01883ap-1}, {-0x1.9a088a8bf6b2cp-59, -0x1.521ecd0c67e35p-57}},
    {{0x1.f564e56a9730ep-4, -0x1.fc26470e19fd3p-1}, {0x1.a2704729ae56dp-59, -0x1.1ec8668ecaceep-55}},
    {{0x1.5e214448b3fc6p-3, -0x1.f8764fa714ba9p-1}, {0x1.531ff779ddac6p-57, -0x1.ab256778ffcb6p-56}},
    {{0x1.c0b826a7e4f63p-3, -0x1.f38f3ac64e589p-1}, {-0x1.af1439e521935p-62, 0x1.d7bafb51f72e6p-56}},
    {{0x1.111d262b1f677p-2, -0x1.ed740e7684963p-1}, {0x1.824c20ab7aa9ap-56, -0x1.e82c791f59cc2p-56}},
    {{0x1.4135c94176601p-2, -0x1.e6288ec48e112p-1}, {0x1.0c97c4afa2518p-56, 0x1.16b56f2847754p-57}},
    {{0x1.7088530fa459fp-2, -0x1.ddb13b6ccc23cp-1}, {-0x1.44b19e0864c5dp-56, -0x1.83c37c6107db3p-55}},
    {{0x1.9ef7943a8ed8ap-2, -0x1.d4134d14dc93ap-1}, {0x1.6da81290bdbabp-57, 0x1.4ef5295d25af2p-55}},
    {{0x1.cc66e9931c45ep-2, -0x1.c954b213411f5p-1}, {0x1.6850e59c37f8fp-58, 0x1.2fb761e946603p-58}},
    {{0x1.f8ba4dbf89abap-2, -0x1.bd7c0ac6f952ap-1}, {-0x1.2ec1fc1b776b8p-60, 0x1.825a732ac700ap-55}},
    {{0x1.11eb3541b4b23p-1, -0x1.b090a58150200p-1}, {-0x1.ef23b69abe4f1p-55, 0x1.926da300ffccep-55}},
    {{0x1.26d054cdd12dfp-1, -0x1.a29a7a0462782p-1}, {-0x1.5da743ef3770cp-55, 0x1.128bb015df175p-56}},
    {{0x1.3affa292050b9p-1, -0x1.93a22499263fbp-1}, {0x1.e3e25e3954964p-56, -0x1.3d419a920df0bp-55}},
    {{0x1.4e6cabbe3e5e9p-1, -0x1.83b0e0bff976ep-1}, {0x1.3c293edceb327p-57, 0x1.6f420f8ea3475p-56}},
    {{0x1.610b7551d2cdfp-1, -0x1.72d0837efff96p-1}, {-0x1.251b352ff2a37p-56, -0x1.0d4ef0f1d915cp-55}},
    {{0x1.72d0837efff96p-1, -0x1.610b7551d2cdfp-1}, {0x1.0d4ef0f1d915cp-55, 0x1.251b352ff2a37p-56}},
    {{0x1.83b0e0bff976ep-1, -0x1.4e6cabbe3e5e9p-1}, {-0x1.6f420f8ea3475p-56, -0x1.3c293edceb327p-57}},
    {{0x1.93a22499263fbp-1, -0x1.3affa292050b9p-1}, {0x1.3d419a920df0bp-55, -0x1.e3e25e3954964p-56}},
    {{0x1.a29a7a0462782p-1, -0x1.26d054cdd12dfp-1}, {-0x1.128bb015df175p-56, 0x1.5da743ef3770cp-55}},
    {{0x1.b090a58150200p-1, -0x1.11eb3541b4b23p-1}, {-0x1.926da300ffccep-55, 0x1.ef23b69abe4f1p-55}},
    {{0x1.bd7c0ac6f952ap-1, -0x1.f8ba4dbf89abap-2}, {-0x1.825a732ac700ap-55, 0x1.2ec1fc1b776b8p-60}},
    {{0x1.c954b213411f5p-1, -0x1.cc66e9931c45ep-2}, {-0x1.2fb761e946603p-58, -0x1.6850e59c37f8fp-58}},
    {{0x1.d4134d14dc93ap-1, -0x1.9ef7943a8ed8ap-2}, {-0x1.4ef5295d25af2p-55, -0x1.6da81290bdbabp-57}},
    {{0x1.ddb13b6ccc23cp-1, -0x1.7088530fa459fp-2}, {0x1.83c37c6107db3p-55, 0x1.44b19e0864c5dp-56}},
    {{0x1.e6288ec48e112p-1, -0x1.4135c94176601p-2}, {-0x1.16b56f2847754p-57, -0x1.0c97c4afa2518p-56}},
    {{0x1.ed740e7684963p-1, -0x1.111d262b1f677p-2}, {0x1.e82c791f59cc2p-56, -0x1.824c20ab7aa9ap-56}},
    {{0x1.f38f3ac64e589p-1, -0x1.c0b826a7e4f63p-3}, {-0x1.d7bafb51f72e6p-56, 0x1.af1439e521935p-62}},
    {{0x1.f8764fa714ba9p-1, -0x1.5e214448b3fc6p-3}, {0x1.ab256778ffcb6p-56, -0x1.531ff779ddac6p-57}},
    {{0x1.fc26470e19fd3p-1, -0x1.f564e56a9730ep-4}, {0x1.1ec8668ecaceep-55, -0x1.a2704729ae56dp-59}},
    {{0x1.fe9cdad01883ap-1, -0x1.2d52092ce19f6p-4}, {0x1.521ecd0c67e35p-57, 0x1.9a088a8bf6b2cp-59}},
    {{0x1.ffd886084cd0dp-1, -0x1.92155f7a3667ep-6}, {-0x1.1354d4556e4cbp-55, 0x1.b1d63091a0130p-64}},
};

__device__ __forceinline__ double from_words(unsigned hi, unsigned lo) { return __hiloint2double((int)hi, (int)lo); }

// -2 ln u of a double 2^-60 < u <= 1 given by its words, as t + rest (the rounding of the last sum)
__device__ __forceinline__ double minus2log(unsigned hi, unsigned lo, double& rest)
{
    const unsigned t = hi - 0x3fe60000u;
    const LogCell* c = &kLog[(t >> 13) & 127u];
    const int e = (int)t >> 20;   // <= 0
    const double z = from_words(hi - ((unsigned)e << 20), lo);
    const double inv = __ldg(&c->inv), ch = __ldg(&c->hi), cl = __ldg(&c->lo), ke = __ldg(&kExp[-e]);
    const double r = fma(z, inv, -1.0);
    double p = fma(-2.0 / 7.0, r, 1.0 / 3.0);
    p = fma(p, r, -2.0 / 5.0);
    p = fma(p, r, 0.5);
    p = fma(p, r, -2.0 / 3.0);
    p = fma(p, r, 1.0);
    const double s = fma(-2.0, r, ke + ch);
    p = fma(r * r, p, cl);
    const double t2 = s + p;
    rest = (s - t2) + p;
    return t2;
}

// sqrt(t + rest) of t >= 0 (0 below 2^-1000)
__device__ __forceinline__ double newton_sqrt(double t, double rest)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(t));
    const int yh = __double2hiint(y);
    // y / 2 by its exponent; t = 0 (y infinite) gives 0
    const double h = from_words((unsigned)yh - 0x100000u, (unsigned)__double2loint(y));
    double g = t * y;
    g = fma(fma(-g, g, t), h, g);
    g = fma(fma(-g, g, t) + rest, h, g);
    return __double2hiint(t) < 0x01700000 ? 0.0 : g;
}

// z0 = r cos(phi), z1 = r sin(phi), phi = 2 pi (2 k + 1) / 256 + delta
__device__ __forceinline__ void rotate(double r, unsigned k, double delta, double& z0, double& z1)
{
    const double2 cs = __ldg(&kTrig[k].hi), cl = __ldg(&kTrig[k].lo);
    const double q = delta * delta;
    const double sp = fma(fma(-1.0 / 5040.0, q, 1.0 / 120.0), q, -1.0 / 6.0);
    const double cp = fma(fma(-1.0 / 720.0, q, 1.0 / 24.0), q, -0.5);
    const double s = fma(delta * q, sp, delta), c = q * cp;
    z0 = r * (cs.x + fma(-cs.y, s, fma(cs.x, c, cl.x)));
    z1 = r * (cs.y + fma(cs.x, s, fma(cs.y, c, cl.y)));
}

// the pair of the 32-bit uniforms u = (w + 1/2) 2^-32
__device__ __forceinline__ void pair32(unsigned wa, unsigned wb, double& z0, double& z1)
{
    // 2 wa + 1 (33 bits) normalised by shifts: u exactly
    const int p = 32 - __clz((int)wa);   // position of the leading one of 2 wa + 1
    const unsigned long long m = (2ull * wa + 1ull) << (52 - p);
    const unsigned hi = ((unsigned)(m >> 32) & 0xfffffu) | ((unsigned)(1023 - 33 + p) << 20);
    double rest;
    const double t = minus2log(hi, (unsigned)m, rest), r = newton_sqrt(t, rest);
    // odd integer 2 (wb mod 2^25) + 1 - 2^25 in units of 2 pi 2^-33, converted by an exponent trick
    const unsigned odd = 2u * (wb & 0x1ffffffu) + 1u;
    const double delta = (from_words(0x43300000u, odd) - 4503599660924928.0) * (6.283185307179586476925 * 0x1p-33);
    rotate(r, wb >> 25, delta, z0, z1);
}

// the pair of the 53-bit uniforms u = (k + 1/2) 2^-53, k the top 53 bits of two words; u
// rounded to 53 bits (ties to even)
__device__ __forceinline__ void pair53(const uint4 w, double& z0, double& z1)
{
    const unsigned long long k1 = (((unsigned long long)w.x << 32) | w.y) >> 11;
    const unsigned long long k2 = (((unsigned long long)w.z << 32) | w.w) >> 11;
    // 2 k1 + 1 has 54 bits at most; with 54 its last bit is a tie
    unsigned long long m = 2ull * k1 + 1ull;
    int p = 63 - __clzll((long long)m);
    if (p == 53) {
        m = k1 + (k1 & 1ull);      // in units of 2: 53 bits, or 2^53
        p = (m >> 53) ? 54 : 53;
        m = p == 54 ? 1ull << 52 : m;
    } else {
        m <<= 52 - p;
    }
    const unsigned hi = ((unsigned)(m >> 32) & 0xfffffu) | ((unsigned)(1023 - 54 + p) << 20);
    double rest;
    const double t = minus2log(hi, (unsigned)m, rest), r = newton_sqrt(t, rest);
    // odd integer 2 (k2 mod 2^46) + 1 - 2^46 in units of 2 pi 2^-54
    const unsigned long long odd = 0x4330000000000000ull + 2ull * (k2 & 0x3fffffffffffull) + 1ull;
    const double delta = (__longlong_as_double((long long)odd) - 4573968371548160.0) * (6.283185307179586476925 * 0x1p-54);
    rotate(r, (unsigned)(k2 >> 46), delta, z0, z1);
}

}  // namespace n64
}  // namespace mgmc
