// fp64_math.cuh -- log2, reciprocal and exp2 in FP64 for the rates of Eq. 1.
//
// GB300 issues one FP64 instruction in the time of about 64 FP32 ones (2
// lanes per clock and SM), so these are written for the fewest of them, by
// the table method of P. T. P. Tang ("Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989;
// "... of the logarithm function ...", ACM TOMS 16, 1990): a table entry picked
// by the leading bits, and a short polynomial in what is left.  Exponents,
// table indices, comparisons and conversions are integer and FP32 work.
//   log2_rcp_f64   9 FP64 instructions for log2 E and 3 for 1/E
//   exp2_f64       8
// against some 25, 10 and 15 of log2(), a division and exp2().  Errors (measured over
// 2^-20..2^60 and -1000..1000, against 113-bit arithmetic): log2 0.69 ulp of
// max(|log2 E|, 1), 1/E 0.50 ulp, exp2 1.03 ulp.
// The tables are nearest doubles of 40-digit values; the polynomials
// interpolate at Chebyshev nodes.
#pragma once

#include <cstdint>

namespace ion {

// log2(1 + r) / r for |r| <= 1/257, lowest degree first (error of the product below 2^-55)
constexpr double kLog1 = 0x1.71547652b82fep+0, kLog2 = -0x1.71547652924f5p-1,
                 kLog3 = 0x1.ec709dc35f513p-2, kLog4 = -0x1.7155a7b607d21p-2,
                 kLog5 = 0x1.2777cad1d781ep-2;
// (2^r - 1) / r for |r| <= 1/512
constexpr double kExp1 = 0x1.62e42fefa39d9p-1, kExp2 = 0x1.ebfbdff82c585p-3,
                 kExp3 = 0x1.c6b0902b5a621p-5, kExp4 = 0x1.3b2ab83eae236p-7;

// Interval j of the mantissa, [1 + j/128, 1 + (j+1)/128): c = 1/(its middle),
// and -log2 c = hi + lo, hi a multiple of 2^-12 (so that exponent + hi is
// exact in FP32).
struct LogRow {
  double c, lo;
};
static __device__ const LogRow kLogTab[128] = {
    {0x1.fe01fe01fe020p-1, 0x1.388daf558c06bp-17}, {0x1.fa11caa01fa12p-1, -0x1.39dd0ad09fae3p-15},
    {0x1.f6310aca0dbb5p-1, 0x1.363ba850f9bdcp-14}, {0x1.f25f644230ab5p-1, 0x1.a6128d0b44e98p-14},
    {0x1.ee9c7f8458e02p-1, 0x1.6ff0d25464b05p-15}, {0x1.eae807aba01ebp-1, -0x1.8ecf99b58c53fp-14},
    {0x1.e741aa59750e4p-1, -0x1.29207b296fa60p-14}, {0x1.e3a9179dc1a73p-1, 0x1.ee0d80ceee769p-14},
    {0x1.e01e01e01e01ep-1, -0x1.1169475d7eacbp-16}, {0x1.dca01dca01dcap-1, 0x1.11df348494026p-16},
    {0x1.d92f2231e7f8ap-1, -0x1.cb1ca47d29656p-16}, {0x1.d5cac807572b2p-1, 0x1.9a83c2c02929ep-14},
    {0x1.d272ca3fc5b1ap-1, -0x1.8f25bb7ce7abfp-14}, {0x1.cf26e5c44bfc6p-1, -0x1.eb5a7c2cdfe2bp-14},
    {0x1.cbe6d9601cbe7p-1, 0x1.146d9a8a62f7ep-15}, {0x1.c8b265afb8a42p-1, 0x1.d5c83d2e452a2p-14},
    {0x1.c5894d10d4986p-1, 0x1.fb7d64898a747p-14}, {0x1.c26b5392ea01cp-1, 0x1.fec7d05ddfef7p-15},
    {0x1.bf583ee868d8bp-1, -0x1.1a8be56a4a677p-14}, {0x1.bc4fd65883e7bp-1, -0x1.39b9be8f27664p-16},
    {0x1.b951e2b18ff23p-1, -0x1.30e8a06a144d4p-15}, {0x1.b65e2e3beee05p-1, -0x1.f4e1c4791b3e5p-14},
    {0x1.b37484ad806cep-1, -0x1.80389d6fe4abcp-16}, {0x1.b094b31d922a4p-1, 0x1.4ce4823c9a978p-17},
    {0x1.adbe87f94905ep-1, -0x1.5176cbe670fc9p-16}, {0x1.aaf1d2f87ebfdp-1, -0x1.d68aabd572843p-14},
    {0x1.a82e65130e159p-1, -0x1.662513dc07841p-16}, {0x1.a574107688a4ap-1, 0x1.2fb6c4709bb77p-17},
    {0x1.a2c2a87c51ca0p-1, -0x1.53293365ee1ffp-16}, {0x1.a01a01a01a01ap-1, -0x1.c69c94d7ca5f5p-14},
    {0x1.9d79f176b682dp-1, -0x1.62faf11824ed0p-17}, {0x1.9ae24ea5510dap-1, 0x1.f3fb753f12621p-16},
    {0x1.9852f0d8ec0ffp-1, 0x1.c40747db55ba5p-17}, {0x1.95cbb0be377aep-1, -0x1.edc9990e6dba5p-15},
    {0x1.934c67f9b2ce6p-1, 0x1.e36852915b397p-15}, {0x1.90d4f120190d5p-1, 0x1.f5248cd4b831fp-14},
    {0x1.8e6527af1373fp-1, -0x1.e9c8343e7d51dp-14}, {0x1.8bfce8062ff3ap-1, 0x1.57ac51aac45d3p-14},
    {0x1.899c0f601899cp-1, -0x1.0f309e79c7fa3p-16}, {0x1.87427bcc092b9p-1, 0x1.4673b5c37168ep-14},
    {0x1.84f00c2780614p-1, 0x1.f90527409a9a9p-14}, {0x1.82a4a0182a4a0p-1, 0x1.d6759b25dfe53p-14},
    {0x1.8060180601806p-1, 0x1.c28def7de8b09p-15}, {0x1.7e225515a4f1dp-1, -0x1.c8203f37965dcp-15},
    {0x1.7beb3922e017cp-1, 0x1.11b7f10cf28cdp-15}, {0x1.79baa6bb6398bp-1, 0x1.2a6c24cae773dp-14},
    {0x1.77908119ac60dp-1, 0x1.02f6ca47b4a06p-14}, {0x1.756cac201756dp-1, 0x1.4c80bf27c0644p-18},
    {0x1.734f0c541fe8dp-1, -0x1.9dddf9b048396p-14}, {0x1.713786d9c7c09p-1, -0x1.2c2f68d6954f5p-18},
    {0x1.6f26016f26017p-1, 0x1.708fa2b79c3a2p-15}, {0x1.6d1a62681c861p-1, 0x1.8acf798a81799p-15},
    {0x1.6b1490aa31a3dp-1, 0x1.6b902680a153cp-18}, {0x1.691473a88d0c0p-1, -0x1.51b11b3640d44p-14},
    {0x1.6719f3601671ap-1, 0x1.1c67c93ac8928p-15}, {0x1.6524f853b4aa3p-1, 0x1.b869f1c3f86f9p-14},
    {0x1.63356b88ac0dep-1, -0x1.d1156507ddd2ep-14}, {0x1.614b36831ae94p-1, 0x1.f3a73c300cf4dp-14},
    {0x1.5f66434292dfcp-1, 0x1.08892bc00b902p-14}, {0x1.5d867c3ece2a5p-1, -0x1.211c336f787e2p-15},
    {0x1.5babcc647fa91p-1, 0x1.2a3b39774d885p-14}, {0x1.59d61f123ccaap-1, -0x1.c5489254cab0cp-14},
    {0x1.5805601580560p-1, -0x1.5d4e9185f6f6ap-14}, {0x1.56397ba7c52e2p-1, -0x1.9c130dd53fb2bp-14},
    {0x1.54725e6bb82fep-1, 0x1.8026a02700cf1p-14}, {0x1.52aff56a8054bp-1, -0x1.baf2648728ff6p-20},
    {0x1.50f22e111c4c5p-1, 0x1.d064ae0fb3b2bp-14}, {0x1.4f38f62dd4c9bp-1, -0x1.f07f428bdfa24p-15},
    {0x1.4d843bedc2c4cp-1, -0x1.7cdb7a8f76aacp-16}, {0x1.4bd3edda68fe1p-1, -0x1.8b96385a2290ep-16},
    {0x1.4a27fad76014ap-1, -0x1.01b66fbd35f1bp-14}, {0x1.4880522014880p-1, 0x1.c5e5a04b0f37ep-14},
    {0x1.46dce34596066p-1, -0x1.5106da1a8bfeap-19}, {0x1.453d9e2c776cap-1, 0x1.8e8353e67cf46p-14},
    {0x1.43a2730abee4dp-1, -0x1.6d7a370decda8p-14}, {0x1.420b5265e5951p-1, -0x1.fa11e53f4ccabp-15},
    {0x1.40782d10e6566p-1, -0x1.1eb680e5478bap-14}, {0x1.3ee8f42a5af07p-1, -0x1.d115ef7d881c8p-14},
    {0x1.3d5d991aa75c6p-1, 0x1.da80c6c41fec7p-15}, {0x1.3bd60d9232955p-1, -0x1.c4a2399046319p-15},
    {0x1.3a524387ac822p-1, 0x1.8325bdbe206dfp-15}, {0x1.38d22d366088ep-1, 0x1.da44a19b5ae54p-14},
    {0x1.3755bd1c945eep-1, -0x1.96e87473d1d94p-14}, {0x1.35dce5f9f2af8p-1, -0x1.90a5d6749fc73p-14},
    {0x1.34679ace01346p-1, 0x1.ee564c7bdde2ap-14}, {0x1.32f5ced6a1dfap-1, 0x1.cea240187f1ecp-15},
    {0x1.3187758e9ebb6p-1, -0x1.48e97e1d6ef37p-15}, {0x1.301c82ac40260p-1, 0x1.4c40d29bf2a72p-14},
    {0x1.2eb4ea1fed14bp-1, -0x1.45566b911825ap-14}, {0x1.2d50a012d50a0p-1, -0x1.601c2624789b9p-16},
    {0x1.2bef98e5a3711p-1, 0x1.55e2da951b46cp-18}, {0x1.2a91c92f3c105p-1, 0x1.0111eb309295ep-20},
    {0x1.293725bb804a5p-1, -0x1.15db83a3de8d4p-15}, {0x1.27dfa38a1ce4dp-1, -0x1.9654f63a37048p-14},
    {0x1.268b37cd60127p-1, 0x1.c5db68e0b581cp-15}, {0x1.2539d7e9177b2p-1, -0x1.1e0a946366676p-14},
    {0x1.23eb79717605bp-1, 0x1.9f66474ab71c2p-16}, {0x1.22a0122a0122ap-1, 0x1.75adcff6ed5b9p-14},
    {0x1.21579804855e6p-1, -0x1.f37dd9d537ae7p-14}, {0x1.2012012012012p-1, -0x1.d29d03b17694dp-14},
    {0x1.1ecf43c7fb84cp-1, 0x1.d95932267742ep-14}, {0x1.1d8f5672e4abdp-1, 0x1.116a2f25a8d38p-14},
    {0x1.1c522fc1ce059p-1, -0x1.4b4070f761cb5p-17}, {0x1.1b17c67f2bae3p-1, -0x1.d61ee0d335c9dp-14},
    {0x1.19e0119e0119ep-1, 0x1.88221cc248074p-19}, {0x1.18ab083902bdbp-1, 0x1.7eafe46c09af7p-14},
    {0x1.1778a191bd684p-1, -0x1.7ddd7736b2075p-14}, {0x1.1648d50fc3201p-1, -0x1.d0ea66df5c657p-15},
    {0x1.151b9a3fdd5c9p-1, -0x1.80512926a2eb2p-15}, {0x1.13f0e8d344724p-1, -0x1.040be494e45b9p-14},
    {0x1.12c8b89edc0acp-1, -0x1.b336660616083p-14}, {0x1.11a3019a74826p-1, 0x1.333db8a408927p-14},
    {0x1.107fbbe011080p-1, -0x1.3f3259e07f7c2p-16}, {0x1.0f5edfab325a2p-1, 0x1.c48acb8c5386cp-14},
    {0x1.0e40655826011p-1, -0x1.1dbd93565013ap-15}, {0x1.0d24456359e3ap-1, 0x1.6da28bed90aebp-15},
    {0x1.0c0a7868b4171p-1, 0x1.9672e671465afp-14}, {0x1.0af2f722eecb5p-1, -0x1.ef24a116d13a0p-14},
    {0x1.09ddba6af8360p-1, -0x1.d922a355856dep-14}, {0x1.08cabb37565e2p-1, 0x1.d948fdf0ddd22p-14},
    {0x1.07b9f29b8eae2p-1, 0x1.28ebdc7871acbp-14}, {0x1.06ab59c7912fbp-1, 0x1.69117d848d53cp-18},
    {0x1.059eea0727586p-1, -0x1.5cfea0583643ap-14}, {0x1.04949cc1664c5p-1, 0x1.9e05fae11982bp-15},
    {0x1.038c6b78247fcp-1, -0x1.64a621928396bp-14}, {0x1.02864fc7729e9p-1, 0x1.18f3a319fa1a3p-19},
    {0x1.0182436517a37p-1, 0x1.180b8a89c05b7p-14}, {0x1.0080402010080p-1, 0x1.c9e2b7a341bd1p-14},};
static __device__ const float kLogHi[128] = {
    23, 69, 114, 159, 204, 249, 293, 336, 380, 423, 466, 508, 551, 593, 634, 675,
    716, 757, 798, 838, 878, 918, 957, 996, 1035, 1074, 1112, 1150, 1188, 1226, 1263, 1300,
    1337, 1374, 1410, 1446, 1483, 1518, 1554, 1589, 1624, 1659, 1694, 1729, 1763, 1797, 1831, 1865,
    1899, 1932, 1965, 1998, 2031, 2064, 2096, 2128, 2161, 2192, 2224, 2256, 2287, 2319, 2350, 2381,
    2411, 2442, 2472, 2503, 2533, 2563, 2593, 2622, 2652, 2681, 2711, 2740, 2769, 2798, 2826, 2855,
    2883, 2911, 2940, 2968, 2995, 3023, 3051, 3078, 3106, 3133, 3160, 3187, 3214, 3241, 3267, 3294,
    3320, 3346, 3373, 3399, 3424, 3450, 3476, 3502, 3527, 3552, 3578, 3603, 3628, 3653, 3678, 3702,
    3727, 3751, 3776, 3800, 3824, 3849, 3873, 3896, 3920, 3944, 3968, 3991, 4015, 4038, 4061, 4084,};  // in units of 2^-12
// 2^(j/256)
static __device__ const double kExpTab[256] = {
    0x1.0000000000000p+0, 0x1.00b1afa5abcbfp+0, 0x1.0163da9fb3335p+0, 0x1.02168143b0281p+0,
    0x1.02c9a3e778061p+0, 0x1.037d42e11bbccp+0, 0x1.04315e86e7f85p+0, 0x1.04e5f72f654b1p+0,
    0x1.059b0d3158574p+0, 0x1.0650a0e3c1f89p+0, 0x1.0706b29ddf6dep+0, 0x1.07bd42b72a836p+0,
    0x1.0874518759bc8p+0, 0x1.092bdf66607e0p+0, 0x1.09e3ecac6f383p+0, 0x1.0a9c79b1f3919p+0,
    0x1.0b5586cf9890fp+0, 0x1.0c0f145e46c85p+0, 0x1.0cc922b7247f7p+0, 0x1.0d83b23395decp+0,
    0x1.0e3ec32d3d1a2p+0, 0x1.0efa55fdfa9c5p+0, 0x1.0fb66affed31bp+0, 0x1.1073028d7233ep+0,
    0x1.11301d0125b51p+0, 0x1.11edbab5e2ab6p+0, 0x1.12abdc06c31ccp+0, 0x1.136a814f204abp+0,
    0x1.1429aaea92de0p+0, 0x1.14e95934f312ep+0, 0x1.15a98c8a58e51p+0, 0x1.166a45471c3c2p+0,
    0x1.172b83c7d517bp+0, 0x1.17ed48695bbc0p+0, 0x1.18af9388c8deap+0, 0x1.1972658375d2fp+0,
    0x1.1a35beb6fcb75p+0, 0x1.1af99f8138a1cp+0, 0x1.1bbe084045cd4p+0, 0x1.1c82f95281c6bp+0,
    0x1.1d4873168b9aap+0, 0x1.1e0e75eb44027p+0, 0x1.1ed5022fcd91dp+0, 0x1.1f9c18438ce4dp+0,
    0x1.2063b88628cd6p+0, 0x1.212be3578a819p+0, 0x1.21f49917ddc96p+0, 0x1.22bdda27912d1p+0,
    0x1.2387a6e756238p+0, 0x1.2451ffb82140ap+0, 0x1.251ce4fb2a63fp+0, 0x1.25e85711ece75p+0,
    0x1.26b4565e27cddp+0, 0x1.2780e341ddf29p+0, 0x1.284dfe1f56381p+0, 0x1.291ba7591bb70p+0,
    0x1.29e9df51fdee1p+0, 0x1.2ab8a66d10f13p+0, 0x1.2b87fd0dad990p+0, 0x1.2c57e39771b2fp+0,
    0x1.2d285a6e4030bp+0, 0x1.2df961f641589p+0, 0x1.2ecafa93e2f56p+0, 0x1.2f9d24abd886bp+0,
    0x1.306fe0a31b715p+0, 0x1.31432edeeb2fdp+0, 0x1.32170fc4cd831p+0, 0x1.32eb83ba8ea32p+0,
    0x1.33c08b26416ffp+0, 0x1.3496266e3fa2dp+0, 0x1.356c55f929ff1p+0, 0x1.36431a2de883bp+0,
    0x1.371a7373aa9cbp+0, 0x1.37f26231e754ap+0, 0x1.38cae6d05d866p+0, 0x1.39a401b7140efp+0,
    0x1.3a7db34e59ff7p+0, 0x1.3b57fbfec6cf4p+0, 0x1.3c32dc313a8e5p+0, 0x1.3d0e544ede173p+0,
    0x1.3dea64c123422p+0, 0x1.3ec70df1c5175p+0, 0x1.3fa4504ac801cp+0, 0x1.40822c367a024p+0,
    0x1.4160a21f72e2ap+0, 0x1.423fb2709468ap+0, 0x1.431f5d950a897p+0, 0x1.43ffa3f84b9d4p+0,
    0x1.44e086061892dp+0, 0x1.45c2042a7d232p+0, 0x1.46a41ed1d0057p+0, 0x1.4786d668b3237p+0,
    0x1.486a2b5c13cd0p+0, 0x1.494e1e192aed2p+0, 0x1.4a32af0d7d3dep+0, 0x1.4b17dea6db7d7p+0,
    0x1.4bfdad5362a27p+0, 0x1.4ce41b817c114p+0, 0x1.4dcb299fddd0dp+0, 0x1.4eb2d81d8abffp+0,
    0x1.4f9b2769d2ca7p+0, 0x1.508417f4531eep+0, 0x1.516daa2cf6642p+0, 0x1.5257de83f4eefp+0,
    0x1.5342b569d4f82p+0, 0x1.542e2f4f6ad27p+0, 0x1.551a4ca5d920fp+0, 0x1.56070dde910d2p+0,
    0x1.56f4736b527dap+0, 0x1.57e27dbe2c4cfp+0, 0x1.58d12d497c7fdp+0, 0x1.59c0827ff07ccp+0,
    0x1.5ab07dd485429p+0, 0x1.5ba11fba87a03p+0, 0x1.5c9268a5946b7p+0, 0x1.5d84590998b93p+0,
    0x1.5e76f15ad2148p+0, 0x1.5f6a320dceb71p+0, 0x1.605e1b976dc09p+0, 0x1.6152ae6cdf6f4p+0,
    0x1.6247eb03a5585p+0, 0x1.633dd1d1929fdp+0, 0x1.6434634ccc320p+0, 0x1.652b9febc8fb7p+0,
    0x1.6623882552225p+0, 0x1.671c1c70833f6p+0, 0x1.68155d44ca973p+0, 0x1.690f4b19e9538p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6b052fa75173ep+0, 0x1.6c012750bdabfp+0, 0x1.6cfdcddd47645p+0,
    0x1.6dfb23c651a2fp+0, 0x1.6ef9298593ae5p+0, 0x1.6ff7df9519484p+0, 0x1.70f7466f42e87p+0,
    0x1.71f75e8ec5f74p+0, 0x1.72f8286ead08ap+0, 0x1.73f9a48a58174p+0, 0x1.74fbd35d7cbfdp+0,
    0x1.75feb564267c9p+0, 0x1.77024b1ab6e09p+0, 0x1.780694fde5d3fp+0, 0x1.790b938ac1cf6p+0,
    0x1.7a11473eb0187p+0, 0x1.7b17b0976cfdbp+0, 0x1.7c1ed0130c132p+0, 0x1.7d26a62ff86f0p+0,
    0x1.7e2f336cf4e62p+0, 0x1.7f3878491c491p+0, 0x1.80427543e1a12p+0, 0x1.814d2add106d9p+0,
    0x1.82589994cce13p+0, 0x1.8364c1eb941f7p+0, 0x1.8471a4623c7adp+0, 0x1.857f4179f5b21p+0,
    0x1.868d99b4492edp+0, 0x1.879cad931a436p+0, 0x1.88ac7d98a6699p+0, 0x1.89bd0a478580fp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8be05bad61778p+0, 0x1.8cf3216b5448cp+0, 0x1.8e06a5e0866d9p+0,
    0x1.8f1ae99157736p+0, 0x1.902fed0282c8ap+0, 0x1.9145b0b91ffc6p+0, 0x1.925c353aa2fe2p+0,
    0x1.93737b0cdc5e5p+0, 0x1.948b82b5f98e5p+0, 0x1.95a44cbc8520fp+0, 0x1.96bdd9a7670b3p+0,
    0x1.97d829fde4e50p+0, 0x1.98f33e47a22a2p+0, 0x1.9a0f170ca07bap+0, 0x1.9b2bb4d53fe0dp+0,
    0x1.9c49182a3f090p+0, 0x1.9d674194bb8d5p+0, 0x1.9e86319e32323p+0, 0x1.9fa5e8d07f29ep+0,
    0x1.a0c667b5de565p+0, 0x1.a1e7aed8eb8bbp+0, 0x1.a309bec4a2d33p+0, 0x1.a42c980460ad8p+0,
    0x1.a5503b23e255dp+0, 0x1.a674a8af46052p+0, 0x1.a799e1330b358p+0, 0x1.a8bfe53c12e59p+0,
    0x1.a9e6b5579fdbfp+0, 0x1.ab0e521356ebap+0, 0x1.ac36bbfd3f37ap+0, 0x1.ad5ff3a3c2774p+0,
    0x1.ae89f995ad3adp+0, 0x1.afb4ce622f2ffp+0, 0x1.b0e07298db666p+0, 0x1.b20ce6c9a8952p+0,
    0x1.b33a2b84f15fbp+0, 0x1.b468415b749b1p+0, 0x1.b59728de5593ap+0, 0x1.b6c6e29f1c52ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.b928cf22749e4p+0, 0x1.ba5b030a1064ap+0, 0x1.bb8e0b79a6f1fp+0,
    0x1.bcc1e904bc1d2p+0, 0x1.bdf69c3f3a207p+0, 0x1.bf2c25bd71e09p+0, 0x1.c06286141b33dp+0,
    0x1.c199bdd85529cp+0, 0x1.c2d1cd9fa652cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c544778fafb22p+0,
    0x1.c67f12e57d14bp+0, 0x1.c7ba88988c933p+0, 0x1.c8f6d9406e7b5p+0, 0x1.ca3405751c4dbp+0,
    0x1.cb720dcef9069p+0, 0x1.ccb0f2e6d1675p+0, 0x1.cdf0b555dc3fap+0, 0x1.cf3155b5bab74p+0,
    0x1.d072d4a07897cp+0, 0x1.d1b532b08c968p+0, 0x1.d2f87080d89f2p+0, 0x1.d43c8eacaa1d6p+0,
    0x1.d5818dcfba487p+0, 0x1.d6c76e862e6d3p+0, 0x1.d80e316c98398p+0, 0x1.d955d71ff6075p+0,
    0x1.da9e603db3285p+0, 0x1.dbe7cd63a8315p+0, 0x1.dd321f301b460p+0, 0x1.de7d5641c0658p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e11676b197d17p+0, 0x1.e264614f5a129p+0, 0x1.e3b333b16ee12p+0,
    0x1.e502ee78b3ff6p+0, 0x1.e653924676d76p+0, 0x1.e7a51fbc74c83p+0, 0x1.e8f7977cdb740p+0,
    0x1.ea4afa2a490dap+0, 0x1.eb9f4867cca6ep+0, 0x1.ecf482d8e67f1p+0, 0x1.ee4aaa2188510p+0,
    0x1.efa1bee615a27p+0, 0x1.f0f9c1cb6412ap+0, 0x1.f252b376bba97p+0, 0x1.f3ac948dd7274p+0,
    0x1.f50765b6e4540p+0, 0x1.f6632798844f8p+0, 0x1.f7bfdad9cbe14p+0, 0x1.f91d802243c89p+0,
    0x1.fa7c1819e90d8p+0, 0x1.fbdba3692d514p+0, 0x1.fd3c22b8f71f1p+0, 0x1.fe9d96b2a23d9p+0,};

__device__ __forceinline__ int hi_word(double x) { return __double2hiint(x); }
__device__ __forceinline__ int lo_word(double x) { return __double2loint(x); }

// float -> double without the FP64 pipe (normal floats and 0).
__device__ __forceinline__ double f64_of_f32(float x) {
  const uint32_t b = __float_as_uint(x);
  const uint32_t h = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);
  return __hiloint2double((b << 1) ? (int)h : 0, (int)(b << 29));
}

// A double's leading 24 bits as a float, without the FP64 pipe: truncated
// towards 0, its size held within the normal floats (0 becomes about 1e-38).
__device__ __forceinline__ float f32_of_f64(double x) {
  const uint32_t h = (uint32_t)hi_word(x);
  const uint32_t m = min(max(h & 0x7fffffffu, 0x38100000u), 0x47efffffu);
  return __uint_as_float((h & 0x80000000u) | ((m - 0x38000000u) << 3) |
                         ((uint32_t)lo_word(x) >> 29));
}

// Order of two doubles by integer comparison (x, y not NaN; -0 below +0).
__device__ __forceinline__ long long order_f64(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// log2 E of a positive, normal E.
__device__ __forceinline__ double log2_f64(double E) {
  const int h = hi_word(E);
  const int j = (h >> 13) & 127;
  const double m = __hiloint2double((h & 0x000fffff) | 0x3ff00000, lo_word(E));
  const LogRow t = kLogTab[j];
  const double r = fma(m, t.c, -1.0);  // exact up to its own last bit
  // exponent - log2 c's leading part, exact in FP32
  const float ehi = fmaf(kLogHi[j], 1.0f / 4096.0f, (float)((h >> 20) - 1023));
  double p = fma(r, kLog5, kLog4);
  p = fma(p, r, kLog3);
  p = fma(p, r, kLog2);
  p = fma(p, r, kLog1);
  return f64_of_f32(ehi) + fma(p, r, t.lo);
}

// 1/E of a positive, normal E (0 above 2^1020): the FP32 reciprocal of its
// mantissa, one step of the cubic iteration s (1 + d + d^2), d = 1 - m s.
__device__ __forceinline__ double rcp_f64(double E) {
  const int h = hi_word(E), l = lo_word(E);
  const double m = __hiloint2double((h & 0x000fffff) | 0x3ff00000, l);
  const float mf = __uint_as_float(0x3f800000u | ((uint32_t)(h & 0x000fffff) << 3) |
                                   ((uint32_t)l >> 29));
  const double s = f64_of_f32(__fdividef(1.0f, mf));
  const double d = fma(-m, s, 1.0);
  const double q = fma(s, fma(d, d, d), s);
  const int e = (h >> 20) - 1023;
  return e > 1020 ? 0.0 : __hiloint2double(hi_word(q) - (e << 20), lo_word(q));
}

// a / b for a normal b up to 2^1020.
__device__ __forceinline__ double div_f64(double a, double b) {
  const double r = rcp_f64(__longlong_as_double(__double_as_longlong(b) & 0x7fffffffffffffffll));
  return a * __hiloint2double(hi_word(r) ^ (hi_word(b) & (int)0x80000000), lo_word(r));
}

// 2^y; y is clamped to [-1200, 1000] (-1200: 0 after rounding).
__device__ __forceinline__ double exp2_f64(double y) {
  const int yh = hi_word(y);
  if (yh >= 0x408f4000) y = 1000.0;               // 2^1000 at most
  if ((uint32_t)yh > 0xc092c000u) y = -1200.0;    // below -1200
  constexpr double kMagic = 0x1.8p44;             // 8 fractional bits
  const double t = y + kMagic;
  const int n = lo_word(t);
  const double r = y - (t - kMagic);
  double p = fma(r, kExp4, kExp3);
  p = fma(p, r, kExp2);
  p = fma(p, r, kExp1);
  const double T = kExpTab[n & 255];
  const double v = fma(T, p * r, T);
  const int e = n >> 8;
  if (e >= -1021) return __hiloint2double(hi_word(v) + (e << 20), lo_word(v));
  // below the normal range: scaled up by 2^256, then back with one rounding
  return __hiloint2double(hi_word(v) + ((e + 256) << 20), lo_word(v)) * 0x1p-256;
}

// e^z for z <= 0: the product with log2 e rounds once, |z| 2^-53 relative to
// e^z, at most 0.37 2^-53 absolute.
__device__ __forceinline__ double exp_f64(double z) { return exp2_f64(z * 0x1.71547652b82fep+0); }

}  // namespace ion
