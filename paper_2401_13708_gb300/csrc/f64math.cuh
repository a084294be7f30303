// f64math.cuh -- the float64 functions of the pair terms with few operations on
// the float64 pipe, which runs two lanes a cycle per SM on this GPU (a float64
// operation of a warp costs as much as 64 float32 ones): sqrt and its
// reciprocal from one reciprocal-square-root seed, a reciprocal from its seed,
// log(1 + g) by table.  Seeds come from the special-function unit
// (rsqrt.approx / rcp.approx.ftz.f64), everything that only moves bits or
// needs few digits runs on integers or float32.  Compiles for the host too
// (with seeds of the same accuracy), so that a host program can check it.
#pragma once

#include "bits.cuh"

namespace hts {

#ifdef __CUDA_ARCH__
#define HTS_TABLE static __device__ const
#else
#define HTS_TABLE static const
#endif

// log(1 + g) by Tang's table-driven method (P. T. P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic",
// ACM TOMS 16(4), 1990) with accurate tables (S. Gal and B. Bachelis, "An
// accurate elementary mathematical library for the IEEE floating point
// standard", ACM TOMS 17(1), 1991): entry j holds a float64 r_j near
// 1 / (1 + j / 128) chosen so that -log r_j is a multiple of 2^-46 to within
// 2^-65, and that multiple.
struct __align__(16) LogEntry {
    double r, t;
};
HTS_TABLE LogEntry kLogTable[128] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.fc07ef1c55a1fp-1, 0x1.fe032969e0000p-8},
    {0x1.f81f83e5d993ap-1, 0x1.fc0a0db382000p-7}, {0x1.f44655e6340c7p-1, 0x1.7b92334a33000p-6},
    {0x1.f07c19372919bp-1, 0x1.f82a70cb38000p-6}, {0x1.ecc077a02cc14p-1, 0x1.39e8b6d904000p-5},
    {0x1.e9131791b816bp-1, 0x1.7745c49a62800p-5}, {0x1.e573a52b31edfp-1, 0x1.b42e53d8ad800p-5},
    {0x1.e1e1df70e5c05p-1, 0x1.f0a33581d4800p-5}, {0x1.de5d68d0f2021p-1, 0x1.16539d6d1fc00p-4},
    {0x1.dae60d5604a8ap-1, 0x1.341d465bd5400p-4}, {0x1.d77b68c955a05p-1, 0x1.51b0559b49c00p-4},
    {0x1.d41d489c5e6a6p-1, 0x1.6f0ced561d000p-4}, {0x1.d0cb53fa9c46ap-1, 0x1.8c34895298c00p-4},
    {0x1.cd856948d6cc9p-1, 0x1.a926cd3e3b000p-4}, {0x1.ca4b2ec6a3b7cp-1, 0x1.c5e556e665400p-4},
    {0x1.c71c750f2664ap-1, 0x1.e270595a55c00p-4}, {0x1.c3f8ef15737efp-1, 0x1.fec91c6b58000p-4},
    {0x1.c0e06fcbd1b42p-1, 0x1.0d77e9bb1c200p-3}, {0x1.bdd2b1f79cc07p-1, 0x1.1b72cbc97ea00p-3},
    {0x1.bacf955ec101dp-1, 0x1.29551cabc2c00p-3}, {0x1.b7d6c393e8e7dp-1, 0x1.371fc35934800p-3},
    {0x1.b4e81be325ef7p-1, 0x1.44d2b413f6000p-3}, {0x1.b20367c91c41fp-1, 0x1.526e4c7d1e000p-3},
    {0x1.af2872521dd63p-1, 0x1.5ff2e8046bc00p-3}, {0x1.ac5705da482dcp-1, 0x1.6d60ea75f4200p-3},
    {0x1.a98ef201f9835p-1, 0x1.7ab8a3778ce00p-3}, {0x1.a6d01e09e8daep-1, 0x1.87f9f4d20cc00p-3},
    {0x1.a41a47dde714bp-1, 0x1.95258b757f200p-3}, {0x1.a16d40786cef9p-1, 0x1.a23bbdaf54e00p-3},
    {0x1.9ec8ef3cd1a97p-1, 0x1.af3c77abc1000p-3}, {0x1.9c2d1b43007cap-1, 0x1.bc2847cdeea00p-3},
    {0x1.999995298cf36p-1, 0x1.c8ff92a9e9000p-3}, {0x1.970e5442661c0p-1, 0x1.d5c1fec6ea200p-3},
    {0x1.948b120d7e30bp-1, 0x1.e2706b7e60600p-3}, {0x1.920fb2c3476e2p-1, 0x1.ef0ae62b11c00p-3},
    {0x1.8f9c17483d017p-1, 0x1.fb918f83ab400p-3}, {0x1.8d3016bc8aa77p-1, 0x1.04025ead37900p-2},
    {0x1.8acb93d358ec6p-1, 0x1.0a3246bb0a700p-2}, {0x1.886e632734bc7p-1, 0x1.1058b4e097200p-2},
    {0x1.86185b7439c96p-1, 0x1.1675daa9a2d00p-2}, {0x1.83c974379c76fp-1, 0x1.1c899533c0800p-2},
    {0x1.8181849ff4f69p-1, 0x1.2294177414f00p-2}, {0x1.7f4059e77f25fp-1, 0x1.2895b10760d00p-2},
    {0x1.7d05f887f2376p-1, 0x1.2e8e1fc0b6f00p-2}, {0x1.7ad21ce900e76p-1, 0x1.347de383b1700p-2},
    {0x1.78a4cca0245ecp-1, 0x1.3a64b90331900p-2}, {0x1.767dca5d04cb8p-1, 0x1.4043131211700p-2},
    {0x1.745d1bcf25515p-1, 0x1.4618afa81f600p-2}, {0x1.724283431571fp-1, 0x1.4be60651f0500p-2},
    {0x1.702e009762d96p-1, 0x1.51aae6cdd4b00p-2}, {0x1.6e1f753d2b79ep-1, 0x1.5767758d40100p-2},
    {0x1.6c16be8de5d43p-1, 0x1.5d1be4066a400p-2}, {0x1.6a13c792050cap-1, 0x1.62c83ec2a6500p-2},
    {0x1.68167eb21ac5cp-1, 0x1.686c899f35300p-2}, {0x1.661ec56ded17bp-1, 0x1.6e08ee1c68300p-2},
    {0x1.642c836fd3d54p-1, 0x1.739d858a3c000p-2}, {0x1.623fac5aca517p-1, 0x1.792a47c763c00p-2},
    {0x1.605817fdc5136p-1, 0x1.7eaf7dfea6400p-2}, {0x1.5e75be284b0c9p-1, 0x1.842d16042d700p-2},
    {0x1.5c98872f957bap-1, 0x1.89a32b504d200p-2}, {0x1.5ac0585e3975bp-1, 0x1.8f11e37d24800p-2},
    {0x1.58ed22509ce27p-1, 0x1.947943e2bfb00p-2}, {0x1.571ed717d51ddp-1, 0x1.99d94e265e100p-2},
    {0x1.555552cb4f340p-1, 0x1.9f32466a0bf00p-2}, {0x1.539094e37cc49p-1, 0x1.a484081057700p-2},
    {0x1.51d07eb473e72p-1, 0x1.a9cec996a1300p-2}, {0x1.501502c5e5e0ep-1, 0x1.af128eb17f200p-2},
    {0x1.4e5e07c6ad5d9p-1, 0x1.b44f7fec56100p-2}, {0x1.4cab856386ac7p-1, 0x1.b98592d2d6900p-2},
    {0x1.4afd6a026a935p-1, 0x1.beb4d9e2f8000p-2}, {0x1.495399b57d0ffp-1, 0x1.c3dd888c8a100p-2},
    {0x1.47ae17883e845p-1, 0x1.c8ff72efe6500p-2}, {0x1.460cbda815c07p-1, 0x1.ce1aed147af00p-2},
    {0x1.446f88e903c4fp-1, 0x1.d32fdfc09ae00p-2}, {0x1.42d6639786878p-1, 0x1.d83e6e7404400p-2},
    {0x1.4141420479d13p-1, 0x1.dd469dddd8000p-2}, {0x1.3fb015dc58252p-1, 0x1.e2487ba1fc700p-2},
    {0x1.3e22cd059be07p-1, 0x1.e74422335ac00p-2}, {0x1.3c9956d9fed0dp-1, 0x1.ec39a83b54b00p-2},
    {0x1.3b13b4f55ee2dp-1, 0x1.f128e9dd7c200p-2}, {0x1.3991c2b1010bep-1, 0x1.f6123fdcfb200p-2},
    {0x1.38137c699f07ap-1, 0x1.faf598bcfd800p-2}, {0x1.3698de2bb87cbp-1, 0x1.ffd2e40d5b100p-2},
    {0x1.3521cd6e4340ep-1, 0x1.02552e1bbdb00p-1}, {0x1.33ae4620c377cp-1, 0x1.04bdf9280d280p-1},
    {0x1.323e3150c2969p-1, 0x1.0723eb4ec8a80p-1}, {0x1.30d19294aedc9p-1, 0x1.0986f0bfb5a00p-1},
    {0x1.2f684f320e473p-1, 0x1.0be7289dda980p-1}, {0x1.2e025bdabe15bp-1, 0x1.0e4498a446880p-1},
    {0x1.2c9fb20c44c01p-1, 0x1.109f3ea5efb80p-1}, {0x1.2b404bd8f29aap-1, 0x1.12f717940fe80p-1},
    {0x1.29e41372dd296p-1, 0x1.154c3bc1e1400p-1}, {0x1.288afe1660462p-1, 0x1.179eb10ae7680p-1},
    {0x1.273509878515ep-1, 0x1.19ee6ebf71c80p-1}, {0x1.25e2258216a0cp-1, 0x1.1c3b849e70580p-1},
    {0x1.24924b0869290p-1, 0x1.1e85f2984c080p-1}, {0x1.2345659a06874p-1, 0x1.20cdd0806b400p-1},
    {0x1.21fb762b72cb5p-1, 0x1.231310d735480p-1}, {0x1.20b46d2a5abf2p-1, 0x1.2555c35072980p-1},
    {0x1.1f704654365bdp-1, 0x1.2795e3e29a400p-1}, {0x1.1e2eefa844ebcp-1, 0x1.29d387291fc80p-1},
    {0x1.1cf06dcf95186p-1, 0x1.2c0e998349080p-1}, {0x1.1bb4a6250af2dp-1, 0x1.2e473f9766680p-1},
    {0x1.1a7b97d68ae04p-1, 0x1.307d700015580p-1}, {0x1.19453a2431abdp-1, 0x1.32b12fbb3f700p-1},
    {0x1.18118240c5bd7p-1, 0x1.34e287bb64a00p-1}, {0x1.16e065f3d53a6p-1, 0x1.37118026cb080p-1},
    {0x1.15b1e3f4c9809p-1, 0x1.393e10ea0f200p-1}, {0x1.1485f452d6c6fp-1, 0x1.3b683e3e9e200p-1},
    {0x1.135c7cf6219c2p-1, 0x1.3d902e4d6f000p-1}, {0x1.12358a58ec8efp-1, 0x1.3fb5bffb0d500p-1},
    {0x1.111114e8b1910p-1, 0x1.41d8f7501a480p-1}, {0x1.0feeff5ee1877p-1, 0x1.43fa015ef8480p-1},
    {0x1.0ecf56b72cda0p-1, 0x1.4618bc2f75200p-1}, {0x1.0db208c28140bp-1, 0x1.4835407d67300p-1},
    {0x1.0c9712104b236p-1, 0x1.4a4f8b6bf4b80p-1}, {0x1.0b7e6a94f54c1p-1, 0x1.4c67a2fbb1700p-1},
    {0x1.0a680cb1e0436p-1, 0x1.4e7d88b59ac80p-1}, {0x1.0953f2625be72p-1, 0x1.50913f0649300p-1},
    {0x1.084211c765612p-1, 0x1.52a2cff367f00p-1}, {0x1.07325ffce5f6bp-1, 0x1.54b247bfa1f00p-1},
    {0x1.0624dc7207409p-1, 0x1.56bf9ecc89100p-1}, {0x1.05197f06d348dp-1, 0x1.58cadc4575480p-1},
    {0x1.0410403274e14p-1, 0x1.5ad4066003d80p-1}, {0x1.03091aa2e3006p-1, 0x1.5cdb1f20ccc80p-1},
    {0x1.020407e144382p-1, 0x1.5ee02aef3e080p-1}, {0x1.01010105fed9ap-1, 0x1.60e32f3a86d80p-1},
};
// k log 2: its multiple of 2^-46 and the rest
HTS_TABLE LogEntry kLn2Table[128] = {
    {0x0.0p+0, 0x0.0p+0}, {0x1.62e42fefa3980p-1, 0x1.bcd5e4f1d9cc0p-47},
    {0x1.62e42fefa39c0p+0, 0x1.79abc9e3b3980p-47}, {0x1.0a2b23f3bab60p+1, 0x1.3681aed58d640p-47},
    {0x1.62e42fefa39e0p+1, 0x1.e6af278ece601p-48}, {0x1.bb9d3beb8c860p+1, 0x1.605af17281f81p-48},
    {0x1.0a2b23f3bab70p+2, 0x1.b40d76ac6b203p-49}, {0x1.3687a9f1af2b0p+2, 0x1.4eca14e7a4a07p-50},
    {0x1.62e42fefa39e0p+2, 0x1.e6af278ece601p-47}, {0x1.8f40b5ed98120p+2, 0x1.a3850c80a82c1p-47},
    {0x1.bb9d3beb8c860p+2, 0x1.605af17281f81p-47}, {0x1.e7f9c1e980fa0p+2, 0x1.1d30d6645bc41p-47},
    {0x1.0a2b23f3bab70p+3, 0x1.b40d76ac6b203p-48}, {0x1.205966f2b4f10p+3, 0x1.2db940901eb83p-48},
    {0x1.3687a9f1af2b0p+3, 0x1.4eca14e7a4a07p-49}, {0x1.4cb5ecf0a9650p+3, 0x1.0886a2bc2f41ep-51},
    {0x1.62e42fefa39e8p+3, 0x1.cd5e4f1d9cc02p-47}, {0x1.791272ee9dd88p+3, 0x1.8a34340f768c2p-47},
    {0x1.8f40b5ed98128p+3, 0x1.470a190150582p-47}, {0x1.a56ef8ec924c8p+3, 0x1.03dffdf32a242p-47},
    {0x1.bb9d3beb8c868p+3, 0x1.816bc5ca07e05p-48}, {0x1.d1cb7eea86c08p+3, 0x1.f62f1f5b76f0ap-49},
    {0x1.e7f9c1e980fa8p+3, 0x1.d30d6645bc416p-50}, {0x1.fe2804e87b340p+3, 0x1.f73791ba91543p-47},
    {0x1.0a2b23f3bab70p+4, 0x1.b40d76ac6b203p-47}, {0x1.1542457337d40p+4, 0x1.70e35b9e44ec3p-47},
    {0x1.205966f2b4f10p+4, 0x1.2db940901eb83p-47}, {0x1.2b708872320e0p+4, 0x1.d51e4b03f1087p-48},
    {0x1.3687a9f1af2b0p+4, 0x1.4eca14e7a4a07p-48}, {0x1.419ecb712c480p+4, 0x1.90ebbd96b070ep-49},
    {0x1.4cb5ecf0a9650p+4, 0x1.0886a2bc2f41ep-50}, {0x1.57cd0e702681cp+4, 0x1.dde6b9495fb44p-47},
    {0x1.62e42fefa39ecp+4, 0x1.9abc9e3b39804p-47}, {0x1.6dfb516f20bbcp+4, 0x1.5792832d134c4p-47},
    {0x1.791272ee9dd8cp+4, 0x1.1468681eed184p-47}, {0x1.8429946e1af5cp+4, 0x1.a27c9a218dc89p-48},
    {0x1.8f40b5ed9812cp+4, 0x1.1c28640541609p-48}, {0x1.9a57d76d152fcp+4, 0x1.2ba85bd1e9f12p-49},
    {0x1.a56ef8ec924ccp+4, 0x1.effef9951212cp-53}, {0x1.b0861a6c0f698p+4, 0x1.c495e0d82e145p-47},
    {0x1.bb9d3beb8c868p+4, 0x1.816bc5ca07e05p-47}, {0x1.c6b45d6b09a38p+4, 0x1.3e41aabbe1ac5p-47},
    {0x1.d1cb7eea86c08p+4, 0x1.f62f1f5b76f0ap-48}, {0x1.dce2a06a03dd8p+4, 0x1.6fdae93f2a88bp-48},
    {0x1.e7f9c1e980fa8p+4, 0x1.d30d6645bc416p-49}, {0x1.f310e368fe178p+4, 0x1.8cc9f41a46e2cp-50},
    {0x1.fe2804e87b344p+4, 0x1.ee6f237522a86p-47}, {0x1.049f9333fc28ap+5, 0x1.ab450866fc746p-47},
    {0x1.0a2b23f3bab72p+5, 0x1.681aed58d6406p-47}, {0x1.0fb6b4b37945ap+5, 0x1.24f0d24ab00c6p-47},
    {0x1.1542457337d42p+5, 0x1.c38d6e7913b0cp-48}, {0x1.1acdd632f662ap+5, 0x1.3d39385cc748dp-48},
    {0x1.205966f2b4f12p+5, 0x1.6dca0480f5c1ap-49}, {0x1.25e4f7b2737fap+5, 0x1.8486612173c69p-51},
    {0x1.2b708872320e0p+5, 0x1.d51e4b03f1087p-47}, {0x1.30fc1931f09c8p+5, 0x1.91f42ff5cad47p-47},
    {0x1.3687a9f1af2b0p+5, 0x1.4eca14e7a4a07p-47}, {0x1.3c133ab16db98p+5, 0x1.0b9ff9d97e6c7p-47},
    {0x1.419ecb712c480p+5, 0x1.90ebbd96b070ep-48}, {0x1.472a5c30ead68p+5, 0x1.0a97877a6408fp-48},
    {0x1.4cb5ecf0a9650p+5, 0x1.0886a2bc2f41ep-49}, {0x1.52417db067f36p+5, 0x1.fef78da0e59c8p-47},
    {0x1.57cd0e702681ep+5, 0x1.bbcd7292bf688p-47}, {0x1.5d589f2fe5106p+5, 0x1.78a3578499348p-47},
    {0x1.62e42fefa39eep+5, 0x1.35793c7673008p-47}, {0x1.686fc0af622d6p+5, 0x1.e49e42d099990p-48},
    {0x1.6dfb516f20bbep+5, 0x1.5e4a0cb44d310p-48}, {0x1.7386e22edf4a6p+5, 0x1.afebad3001921p-49},
    {0x1.791272ee9dd8ep+5, 0x1.468681eed1843p-50}, {0x1.7e9e03ae5c674p+5, 0x1.e5a6b52fb3fc9p-47},
    {0x1.8429946e1af5cp+5, 0x1.a27c9a218dc89p-47}, {0x1.89b5252dd9844p+5, 0x1.5f527f1367949p-47},
    {0x1.8f40b5ed9812cp+5, 0x1.1c28640541609p-47}, {0x1.94cc46ad56a14p+5, 0x1.b1fc91ee36592p-48},
    {0x1.9a57d76d152fcp+5, 0x1.2ba85bd1e9f12p-48}, {0x1.9fe3682cd3be4p+5, 0x1.4aa84b6b3b125p-49},
    {0x1.a56ef8ec924ccp+5, 0x1.effef9951212cp-52}, {0x1.aafa89ac50db2p+5, 0x1.cc55dcbe825cap-47},
    {0x1.b0861a6c0f69ap+5, 0x1.892bc1b05c28ap-47}, {0x1.b611ab2bcdf82p+5, 0x1.4601a6a235f4ap-47},
    {0x1.bb9d3beb8c86ap+5, 0x1.02d78b940fc0ap-47}, {0x1.c128ccab4b152p+5, 0x1.7f5ae10bd3194p-48},
    {0x1.c6b45d6b09a3ap+5, 0x1.f20d55df0d628p-49}, {0x1.cc3fee2ac8322p+5, 0x1.cac9d34ce9252p-50},
    {0x1.d1cb7eea86c08p+5, 0x1.f62f1f5b76f0ap-47}, {0x1.d7570faa454f0p+5, 0x1.b305044d50bcap-47},
    {0x1.dce2a06a03dd8p+5, 0x1.6fdae93f2a88bp-47}, {0x1.e26e3129c26c0p+5, 0x1.2cb0ce310454bp-47},
    {0x1.e7f9c1e980fa8p+5, 0x1.d30d6645bc416p-48}, {0x1.ed8552a93f890p+5, 0x1.4cb930296fd96p-48},
    {0x1.f310e368fe178p+5, 0x1.8cc9f41a46e2cp-49}, {0x1.f89c7428bca60p+5, 0x1.00430fc35c25ap-50},
    {0x1.fe2804e87b346p+5, 0x1.dcde46ea4550bp-47}, {0x1.01d9cad41ce17p+6, 0x1.99b42bdc1f1cbp-47},
    {0x1.049f9333fc28bp+6, 0x1.568a10cdf8e8cp-47}, {0x1.07655b93db6ffp+6, 0x1.135ff5bfd2b4cp-47},
    {0x1.0a2b23f3bab73p+6, 0x1.a06bb56359018p-48}, {0x1.0cf0ec5399fe7p+6, 0x1.1a177f470c998p-48},
    {0x1.0fb6b4b37945bp+6, 0x1.2786925580630p-49}, {0x1.127c7d13588cfp+6, 0x1.ade261ce7930ep-53},
    {0x1.1542457337d42p+6, 0x1.c38d6e7913b0cp-47}, {0x1.18080dd3171b6p+6, 0x1.8063536aed7ccp-47},
    {0x1.1acdd632f662ap+6, 0x1.3d39385cc748dp-47}, {0x1.1d939e92d5a9ep+6, 0x1.f41e3a9d42299p-48},
    {0x1.205966f2b4f12p+6, 0x1.6dca0480f5c1ap-48}, {0x1.231f2f5294386p+6, 0x1.ceeb9cc952b34p-49},
    {0x1.25e4f7b2737fap+6, 0x1.8486612173c69p-50}, {0x1.28aac01252c6dp+6, 0x1.ed66b1160844dp-47},
    {0x1.2b708872320e1p+6, 0x1.aa3c9607e210dp-47}, {0x1.2e3650d211555p+6, 0x1.67127af9bbdcdp-47},
    {0x1.30fc1931f09c9p+6, 0x1.23e85feb95a8ep-47}, {0x1.33c1e191cfe3dp+6, 0x1.c17c89badee9bp-48},
    {0x1.3687a9f1af2b1p+6, 0x1.3b28539e9281cp-48}, {0x1.394d72518e725p+6, 0x1.69a83b048c338p-49},
    {0x1.3c133ab16db99p+6, 0x1.73ff3b2fcd8e1p-51}, {0x1.3ed903114d00cp+6, 0x1.d415d8a4d6a4ep-47},
    {0x1.419ecb712c480p+6, 0x1.90ebbd96b070ep-47}, {0x1.446493d10b8f4p+6, 0x1.4dc1a2888a3cep-47},
    {0x1.472a5c30ead68p+6, 0x1.0a97877a6408fp-47}, {0x1.49f02490ca1dcp+6, 0x1.8edad8d87ba9dp-48},
    {0x1.4cb5ecf0a9650p+6, 0x1.0886a2bc2f41ep-48}, {0x1.4f7bb55088ac4p+6, 0x1.0464d93fc5b3cp-49},
    {0x1.52417db067f37p+6, 0x1.fdef1b41cb38fp-47}, {0x1.55074610473abp+6, 0x1.bac50033a504fp-47},
    {0x1.57cd0e702681fp+6, 0x1.779ae5257ed0fp-47}, {0x1.5a92d6d005c93p+6, 0x1.3470ca17589cfp-47},
    {0x1.5d589f2fe5107p+6, 0x1.e28d5e1264d1fp-48}, {0x1.601e678fc457bp+6, 0x1.5c3927f61869fp-48},
};

__host__ __device__ __forceinline__ double rsqrt_seed(double x)  // 1 / sqrt(x) to about 2^-20
{
#ifdef __CUDA_ARCH__
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
#else
    return double_of(bits_of(1.0 / sqrt(x)) & 0xFFFFFFFF00000000ull);
#endif
}

__host__ __device__ __forceinline__ double rcp_seed(double x)  // 1 / x to about 2^-20
{
#ifdef __CUDA_ARCH__
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
#else
    return double_of(bits_of(1.0 / x) & 0xFFFFFFFF00000000ull);
#endif
}

// t = sqrt(x) and rs = 1 / sqrt(x) for a normal x > 0, within about one unit in
// the last place each: with h = x y0 and e = 1 - h y0 for the seed y0,
// 1 / sqrt(1 - e) = 1 + e / 2 + 3 e^2 / 8 + O(e^3), e ~ 2^-20 (7 operations).
__host__ __device__ __forceinline__ void sqrt_rsqrt(double x, double &t, double &rs)
{
    const double y0 = rsqrt_seed(x);
    const double h = x * y0;
    const double e = fma(-h, y0, 1.0);
    const double p = fma(0.375, e, 0.5);
    rs = fma(y0 * e, p, y0);
    t = fma(h * e, p, h);
}

// 1 / x for a normal x whose reciprocal is normal: w0 (1 + e + e^2), e = 1 - x w0
// (3 operations).
__host__ __device__ __forceinline__ double reciprocal(double x)
{
    const double w0 = rcp_seed(x);
    const double e = fma(-x, w0, 1.0);
    return fma(w0, fma(e, e, e), w0);
}

// log(1 + m), |m| < 2^-7.99 (5 operations): m + m^2 (-1/2 + m (1/3 + m (-1/4 +
// m q))), q = 1/5 - m / 6 + m^2 / 7 in float32 (it is worth 2^-32 of the
// result; the next term of the series 2^-59).
__host__ __device__ __forceinline__ double log1p_series(double m)
{
    const unsigned mh = (unsigned)(bits_of(m) >> 32), ma = mh & 0x7FFFFFFFu;
    // m as float32 from the top 20 bits of its significand (0 below 2^-123)
    const float mf = ma < (900u << 20) ? 0.0f : float_of((mh & 0x80000000u) | ((ma << 3) - (896u << 23)));
    const float q = fmaf(mf, fmaf(mf, 1.0f / 7.0f, -1.0f / 6.0f), 0.2f);
    const unsigned qb = bits_of(q);
    const double qd = double_of(((unsigned long long)((qb >> 3) + (896u << 20)) << 32) | (unsigned long long)(qb << 29));
    double c = fma(m, qd, -0.25);
    c = fma(m, c, 1.0 / 3.0);
    c = fma(m, c, -0.5);
    return fma(m * m, c, m);
}

// log(1 + g), g >= 0 (11 operations).  z = 1 + g = 2^k v with v rounded to a
// 1 + j / 128 below 2, m = v r_j - 1 with |m| < 2^-7.99: log z = k log 2 -
// log r_j + log(1 + m); the first two have an exact sum.  Where k = 0, m =
// g r + (r - 1) instead, so that small g keeps its digits (r = 1 below
// g = 2^-8: m = g).
__host__ __device__ __forceinline__ double log1p_pos(double g)
{
    const double z = 1.0 + g;
    const unsigned long long zb = bits_of(z);
    const unsigned zr = (unsigned)(zb >> 32) + 0x1000u;  // rounded to 7 bits
    const int k = (int)((zr >> 20) - 1023u) & 127;       // (z < 2^127; masked: the tables are never left)
    const int j = (int)((zr & 0xFFFFFu) >> 13);
#ifdef __CUDA_ARCH__
    const double2 tab = __ldg(reinterpret_cast<const double2 *>(kLogTable) + j);
    const double2 kl = __ldg(reinterpret_cast<const double2 *>(kLn2Table) + k);
    const double r = tab.x, tt = tab.y, kh = kl.x, klo = kl.y;
#else
    const double r = kLogTable[j].r, tt = kLogTable[j].t, kh = kLn2Table[k].r, klo = kLn2Table[k].t;
#endif
    const double a = k == 0 ? g : double_of(zb - ((unsigned long long)(unsigned)k << 52));
    const double b = k == 0 ? r - 1.0 : -1.0;
    const double m = fma(a, r, b);
    return (tt + kh) + (log1p_series(m) + klo);
}

// log x, x > 0 normal (8 operations; library outside 2^-127 .. 2^127).
__host__ __device__ __forceinline__ double log_pos(double x)
{
    const unsigned long long xb = bits_of(x);
    const unsigned xr = (unsigned)(xb >> 32) + 0x1000u;
    const int k = (int)(xr >> 20) - 1023;
    if (k < -127 || k > 127) return log(x);
    const int j = (int)((xr & 0xFFFFFu) >> 13), ka = k < 0 ? -k : k;
#ifdef __CUDA_ARCH__
    const double2 tab = __ldg(reinterpret_cast<const double2 *>(kLogTable) + j);
    const double2 kl = __ldg(reinterpret_cast<const double2 *>(kLn2Table) + ka);
    const double r = tab.x, tt = tab.y, kh = kl.x, klo = kl.y;
#else
    const double r = kLogTable[j].r, tt = kLogTable[j].t, kh = kLn2Table[ka].r, klo = kLn2Table[ka].t;
#endif
    const double m = fma(double_of(xb - ((unsigned long long)(long long)k << 52)), r, -1.0);
    const double lp = log1p_series(m);
    return k < 0 ? (tt - kh) + (lp - klo) : (tt + kh) + (lp + klo);
}

#undef HTS_TABLE

}  // namespace hts
