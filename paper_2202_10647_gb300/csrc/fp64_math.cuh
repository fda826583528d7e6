// fp64_math.cuh -- log2, reciprocal and exp2 in FP64 for the rates of Eq. 1.
//
// GB300 issues one FP64 instruction in the time of about 64 FP32 ones (2
// lanes per clock and SM), so these are written for the fewest of them, by
// the table method of P. T. P. Tang ("Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989;
// "... of the logarithm function ...", ACM TOMS 16, 1990): a table entry picked
// by the leading bits, and a short polynomial in what is left.  Exponents,
// table indices, comparisons and conversions are integer and FP32 work.
//   log2_f64   1 FP64 instruction
//   rcp_f64, exp2_f64, exp_f64   none
// against some 25, 10 and 15 of log2(), a division and exp2(), and 9, 3 and 8 of the same
// method with the polynomials in FP64: everything else is 64-bit fixed point, 20 to 60
// integer instructions each, whose issue time is that of one FP64 instruction at most.  A
// rate of Eq. 1 keeps the two fused multiply-adds of its exponent.  FP64 step, 33.5M nitrogen
// cells: 2,347 us with the polynomials in FP64, 1,922 so.
// Errors (over 2^-20..2^60 and -1000..1000, against 113-bit arithmetic; the tests restate
// these integer steps and hold them): log2 0.79 ulp of max(|log2 E|, 1), 0.57 below 2;
// 1/E 0.56 ulp; exp2 0.97 ulp; e^z 0.99 ulp down to z = -256 (1.2 to -512, 1.9 below).
// The tables are nearest values of 40-digit ones; the polynomials
// interpolate at Chebyshev nodes.
#pragma once

#include <cstdint>

namespace ion {

// log2(1 + rho/64) 64/rho for rho in [0, 1/2] in units of 2^-51, lowest degree first, every
// other sign a minus (error of the product below 2^-60)
constexpr uint64_t kLog1 = 0xb8aa3b295c17full, kLog2 = 0x171547652b7cull,
                   kLog3 = 0x3d8e13b7caull;
constexpr uint32_t kLog4 = 0xb8aa3580u, kLog5 = 0x24ed7a7u, kLog6 = 0x78ab1u;
// 256 (2^(rho/256) - 1) / rho for rho in [0, 1] in units of 2^-52, lowest degree first (error
// 2^-56.6 of 1)
constexpr uint64_t kExp1 = 0xb17217f7d1cedull, kExp2 = 0x3d7f7bff1b7ull;
constexpr uint32_t kExp3 = 0xe3583fe3u, kExp4 = 0x277045u;
constexpr uint64_t kLog2E = 0xb8aa3b295c17f0bcull;  // log2 e in units of 2^-63

// Interval j of the mantissa, [1 + j/128, 1 + (j+1)/128): c, the reciprocal of its lower end
// rounded up, in units of 2^-31, and -log2 c in units of 2^-57.
struct LogRow {
  unsigned long long log;
  uint32_t c;
};
static __device__ const LogRow kLogTab[128] = {
    {0x000000000000000ull, 0x80000000u}, {0x005bf942d5f6cf7ull, 0x7f01fc08u}, {0x00b73cb3d332c83ull, 0x7e07e07fu},
    {0x0111cd1d01da1bcull, 0x7d11967au}, {0x016bad37532a86aull, 0x7c1f07c2u}, {0x01c4dfab339cee2ull, 0x7b301ecdu},
    {0x021d6713dd3eabfull, 0x7a44c6b0u}, {0x027545fb467f1c1ull, 0x795ceb25u}, {0x02cc7edf2532823ull, 0x78787879u},
    {0x0323142dbd3bc7aull, 0x77975b90u}, {0x037908480b9c281ull, 0x76b981dbu}, {0x03ce5d8223b1685ull, 0x75ded953u},
    {0x04231622d484097ull, 0x75075076u}, {0x04773465b9e19a1ull, 0x7432d63eu}, {0x04caba783d826b9ull, 0x73615a25u},
    {0x051daa7e2b9c9e3ull, 0x7292cc16u}, {0x0570068e67e05a8ull, 0x71c71c72u}, {0x05c1d0b4d9a6306ull, 0x70fe3c08u},
    {0x06130af3a5527ffull, 0x70381c0fu}, {0x0663b74196c10e7ull, 0x6f74ae27u}, {0x06b3d78b055b63bull, 0x6eb3e454u},
    {0x07036db336d8f74ull, 0x6df5b0f8u}, {0x07527b92e4311f0ull, 0x6d3a06d4u}, {0x07a102f9b26bfc9ull, 0x6c80d902u},
    {0x07ef05ae0caa21eull, 0x6bca1af3u}, {0x083c856d731aec6ull, 0x6b15c06cu}, {0x088983ed440326eull, 0x6a63bd82u},
    {0x08d602d8f54b156ull, 0x69b4069cu}, {0x092203d5195e89aull, 0x6906906au}, {0x096d887e1cb4088ull, 0x685b4fe6u},
    {0x09b89266fd487f3ull, 0x67b23a55u}, {0x0a03231d5c74ed0ull, 0x670b453cu}, {0x0a4d3c25a14def5ull, 0x66666667u},
    {0x0a96defdc93d91full, 0x65c393e1u}, {0x0ae00d1cb2e61bcull, 0x6522c3f4u}, {0x0b28c7f1dd2e07bull, 0x6483ed28u},
    {0x0b7110e68c2941full, 0x63e7063fu}, {0x0bb8e95d21ea5a8ull, 0x634c0635u}, {0x0c0052b1658b961ull, 0x62b2e43eu},
    {0x0c474e394a1dd49ull, 0x621b97c3u}, {0x0c8ddd4455d651eull, 0x61861862u}, {0x0cd4011c75d2518ull, 0x60f25debu},
    {0x0d19bb04f339abdull, 0x60606061u}, {0x0d5f0c3c471897eull, 0x5fd017f5u}, {0x0da3f5fb967bfe8ull, 0x5f417d06u},
    {0x0de87974b7303cfull, 0x5eb48824u}, {0x0e2c97d686405eaull, 0x5e293206u}, {0x0e70524906cfa14ull, 0x5d9f7391u},
    {0x0eb3a9efd435315ull, 0x5d1745d2u}, {0x0ef69fe9af2215aull, 0x5c90a1feu}, {0x0f3935508a59535ull, 0x5c0b8171u},
    {0x0f7b6b3919d004full, 0x5b87ddaeu}, {0x0fbd42b3e68e5ecull, 0x5b05b05cu}, {0x0ffebccce71c044ull, 0x5a84f346u},
    {0x103fda8b1733221ull, 0x5a05a05bu}, {0x10809cf21ec7226ull, 0x5987b1aau}, {0x10c105006895934ull, 0x590b2165u},
    {0x110113b0d1388eaull, 0x588fe9ddu}, {0x1140c9fa4e3820dull, 0x58160582u}, {0x118028cf0d9a51full, 0x579d6ee4u},
    {0x11bf311e3698476ull, 0x572620afu}, {0x11fde3d2890e218ull, 0x56b015adu}, {0x123c41d3a0fc191ull, 0x563b48c3u},
    {0x127a4c051f5d8b3ull, 0x55c7b4f2u}, {0x12b80346e325b36ull, 0x55555556u}, {0x12f56875d14735cull, 0x54e42524u},
    {0x13327c6a7522227ull, 0x54741facu}, {0x136f3ffae3ca602ull, 0x54054055u}, {0x13abb3fa7a9ed2dull, 0x5397829du},
    {0x13e7d937650239bull, 0x532ae21du}, {0x1423b07e336d911ull, 0x52bf5a82u}, {0x145f3a988473f53ull, 0x5254e78fu},
    {0x149a784ba4b64e1ull, 0x51eb851fu}, {0x14d56a5b1cb97ceull, 0x51832f20u}, {0x15101186c64bcbaull, 0x511be196u},
    {0x154a6e8c43291e4ull, 0x50b59898u}, {0x1584822633a01b7ull, 0x50505051u}, {0x15be4d0c904a4aeull, 0x4fec04ffu},
    {0x15f7cff3de8f2a6ull, 0x4f88b2f4u}, {0x16310b8f4b16f90ull, 0x4f265692u}, {0x166a008e24e8e0bull, 0x4ec4ec4fu},
    {0x16a2af9dfd01424ull, 0x4e6470b1u}, {0x16db1969e1804e4ull, 0x4e04e04fu}, {0x17133e9ac4a2020ull, 0x4da637d0u},
    {0x174b1fd61cfa1c1ull, 0x4d4873edu}, {0x1782bdbf7cfd3c8ull, 0x4ceb916eu}, {0x17ba18f9028457eull, 0x4c8f8d29u},
    {0x17f132215e052c1ull, 0x4c346405u}, {0x182809d5736b4adull, 0x4bda12f7u}, {0x185ea0b03214c8full, 0x4b809702u},
    {0x1894f74a6c913ddull, 0x4b27ed37u}, {0x18cb0e3ab024c60ull, 0x4ad012b5u}, {0x1900e615bac2f6dull, 0x4a7904a8u},
    {0x19367f6d16e42c8ull, 0x4a22c04bu}, {0x196bdad20f74ff9ull, 0x49cd42e3u}, {0x19a0f8d311755adull, 0x497889c3u},
    {0x19d5d9fcc591071ull, 0x4924924au}, {0x1a0a7ed9ed9210aull, 0x48d159e3u}, {0x1a3ee7f341a1a25ull, 0x487ede05u},
    {0x1a7315cff11797eull, 0x482d1c32u}, {0x1aa708f4de7fdfcull, 0x47dc11f8u}, {0x1adac1e7110f889ull, 0x478bbcedu},
    {0x1b0e41267051ef6ull, 0x473c1ab7u}, {0x1b4187341467904ull, 0x46ed2902u}, {0x1b74948ef3186aeull, 0x469ee585u},
    {0x1ba769b317650aeull, 0x46514e03u}, {0x1bda071c20957c9ull, 0x46046047u}, {0x1c0c6d43d9578b3ull, 0x45b81a26u},
    {0x1c3e9ca2c4c5bbfull, 0x456c797eu}, {0x1c7095ae03c6c7eull, 0x45217c39u}, {0x1ca258dc8dc9d17ull, 0x44d72045u},
    {0x1cd3e6a06cc294bull, 0x448d639eu}, {0x1d053f6ca7138dcull, 0x44444445u}, {0x1d3663b27c4f2c4ull, 0x43fbc044u},
    {0x1d6753dfedaa38dull, 0x43b3d5b0u}, {0x1d981063b7f3100ull, 0x436c82a3u}, {0x1dc899ab374d71aull, 0x4325c53fu},
    {0x1df8f0203dd402full, 0x42df9bb1u}, {0x1e29142dcba412eull, 0x429a042au}, {0x1e59063bd8d9383ull, 0x4254fce5u},
    {0x1e88c6b2b54adb3ull, 0x42108422u}, {0x1eb855f82d4804bull, 0x41cc982au}, {0x1ee7b4718b44139ull, 0x4189374cu},
    {0x1f16e281680bcb4ull, 0x41465fe0u}, {0x1f45e08b1c216c0ull, 0x41041042u}, {0x1f74aef092a1e61ull, 0x40c246d5u},
    {0x1fa34e10c64e9e9ull, 0x40810205u}, {0x1fd1be4bf563f72ull, 0x40404041u}};
// 2^(i/256), in units of 2^-62.
static __device__ const unsigned long long kExpTab[256] = {
    0x4000000000000000ull, 0x402c6be96af2fb58ull, 0x4058f6a7ecccd5b6ull, 0x4085a050ec0a036aull,
    0x40b268f9de0183baull, 0x40df50b846ef302bull, 0x410c57a1b9fe12f6ull, 0x41397dcbd952c4a6ull,
    0x4166c34c5615d0ecull, 0x41942838f07e22a3ull, 0x41c1aca777db771bull, 0x41ef50adcaa0d899ull,
    0x421d1461d66f2023ull, 0x424af7d9981f7e98ull, 0x4278fb2b1bce0d15ull, 0x42a71e6c7ce464afull,
    0x42d561b3e6243d8aull, 0x4303c51791b21550ull, 0x433248adc91fdd02ull, 0x4360ec8ce577ae44ull,
    0x438fb0cb4f468808ull, 0x43be957f7ea712b6ull, 0x43ed9abffb4c6bc9ull, 0x441cc0a35c8cf8eaull,
    0x444c0740496d4294ull, 0x447b6ead78aad636ull, 0x44aaf701b0c72feeull, 0x44daa053c812abd2ull,
    0x450a6abaa4b77ecdull, 0x453a564d3cc4b723ull, 0x456a632296394492ull, 0x459a9151c70f0819ull,
    0x45cae0f1f545eb73ull, 0x45fb521a56ef0042ull, 0x462be4e23237a6efull, 0x465c9960dd74bd4bull,
    0x468d6fadbf2dd4f3ull, 0x46be67e04e28717cull, 0x46ef821011734e6bull, 0x4720be54a071ad01ull,
    0x47521cc5a2e6a9e0ull, 0x47839d7ad1009a90ull, 0x47b5408bf36472e2ull, 0x47e70610e3393241ull,
    0x4818ee218a3358eeull, 0x484af8d5e2a06536ull, 0x487d2645f7725895ull, 0x48af7689e44b44eaull,
    0x48e1e9b9d588e19bull, 0x49147fee085028d6ull, 0x4947393eca98fcd6ull, 0x497a15c47b39d53eull,
    0x49ad159789f37496ull, 0x49e038d0777ca5e0ull, 0x4a137f87d58e025bull, 0x4a46e9d646edbf6aull,
    0x4a7a77d47f7b84b1ull, 0x4aae299b443c4a6bull, 0x4ae1ff436b663ff7ull, 0x4b15f8e5dc6cbab0ull,
    0x4b4a169b900c2d00ull, 0x4b7e587d905625d1ull, 0x4bb2bea4f8bd5847ull, 0x4be7492af621abd6ull,
    0x4c1bf828c6dc54b8ull, 0x4c50cbb7bacbf4cbull, 0x4c85c3f13360c4d5ull, 0x4cbae0eea3a8c63cull,
    0x4cf022c9905bfd32ull, 0x4d25899b8fe8b365ull, 0x4d5b157e4a7fc325ull, 0x4d90c68b7a20eb1eull,
    0x4dc69cdceaa72a9cull, 0x4dfc988c79d52661ull, 0x4e32b9b417619617ull, 0x4e69006dc503ba65ull,
    0x4e9f6cd3967fdba8ull, 0x4ed5feffb1b3d155ull, 0x4f0cb70c4ea39210ull, 0x4f439513b785cc80ull,
    0x4f7a993048d088d7ull, 0x4fb1c37c7145d328ull, 0x4fe91412b2006e83ull, 0x50208b0d9e8090dfull,
    0x50582887dcb8a7e1ull, 0x508fec9c251a267cull, 0x50c7d76542a25b72ull, 0x50ffe8fe12e750c4ull,
    0x513821818624b40cull, 0x5170810a9f48c7cfull, 0x51a907b474015dc9ull, 0x51e1b59a2cc8da3eull,
    0x521a8ad704f3404full, 0x525387864abb4762ull, 0x528cabc35f4f799dull, 0x52c5f7a9b6df5b77ull,
    0x52ff6b54d8a89c75ull, 0x533906e05f045106ull, 0x5372ca67f774358full, 0x53acb60762affaaeull,
    0x53e6c9da74b29ab5ull, 0x542105fd14c7b869ull, 0x545b6a8b3d990704ull, 0x5495f7a0fd3bbb8eull,
    0x54d0ad5a753e077cull, 0x550b8bd3dab49cbdull, 0x5546932976483b15ull, 0x5581c377a44346f0ull,
    0x55bd1cdad49f699cull, 0x55f89f6f8b133af4ull, 0x56344b525f1ff495ull, 0x5670209ffc1f2e82ull,
    0x56ac1f752150a563ull, 0x56e847eea1e80a49ull, 0x57249a29651adc07ull, 0x57611642662e4a33ull,
    0x579dbc56b48521baull, 0x57da8c8373adc331ull, 0x581786e5db7022c2ull, 0x5854ab9b37dbd1e5ull,
    0x5891fac0e95612c8ull, 0x58cf747464a7f584ull, 0x590d18d3330c7f1eull, 0x594ae7faf23eda52ull,
    0x5988e20954889245ull, 0x59c7071c20cfd70cull, 0x5a05575132a5cc20ull, 0x5a43d2c67a54e0c0ull,
    0x5a827999fcef3242ull, 0x5ac14be9d45cf869ull, 0x5b0049d42f6afbb6ull, 0x5b3f737751d915c8ull,
    0x5b7ec8f19468bbc9ull, 0x5bbe4a6164eb92f4ull, 0x5bfdf7e546520f3eull, 0x5c3dd19bd0ba1c1aull,
    0x5c7dd7a3b17dcf75ull, 0x5cbe0a1bab4226dfull, 0x5cfe69229605cef5ull, 0x5d3ef4d75f2ff504ull,
    0x5d7fad59099f22feull, 0x5dc092c6adb825b8ull, 0x5e01a53f7974fd86ull, 0x5e42e4e2b073d935ull,
    0x5e8451cfac061b5full, 0x5ec5ec25db3f6a41ull, 0x5f07b404c304c9f1ull, 0x5f49a98bfe1bc11cull,
    0x5f8bccdb3d398841ull, 0x5fce1e124712437cull, 0x60109d50f86846d8ull, 0x60534ab7441b6546ull,
    0x6096266533384a2bull, 0x60d9307ae507dd9aull, 0x611c69188f1eb339ull, 0x615fd05e7d6c83e4ull,
    0x61a3666d124bb204ull, 0x61e72b64c690d8afull, 0x622b1f66299a6599ull, 0x626f4291e1603dd5ull,
    0x62b39508aa836d6full, 0x62f816eb585de1edull, 0x633cc85ad5122fbdull, 0x6381a978219b628full,
    0x63c6ba6455dcd8aeull, 0x640bfb40a0b22959ull, 0x64516c2e47ff1623ull, 0x64970d4ea8bf8766ull,
    0x64dcdec3371793d1ull, 0x6522e0ad7e639312ull, 0x6569132f21483ba7ull, 0x65af7669d9c2cbe4ull,
    0x65f60a7f79393e2eull, 0x663ccf91e88a8873ull, 0x6683c5c3281ee6e9ull, 0x66caed354ff83222ull,
    0x6712460a8fc24072ull, 0x6759d0652ee352afull, 0x67a18c678c8c8c61ull, 0x67e97a341fca775bull,
    0x683199ed779592caull, 0x6879ebb63ae2edc6ull, 0x68c26fb128b4cd63ull, 0x690b2601182b5e56ull,
    0x69540ec8f895722dull, 0x699d2a2bd181482aull, 0x69e6784cc2cd61bdull, 0x6a2ff94f04b962b0ull,
    0x6a79ad55e7f6fd10ull, 0x6ac39484d5bae8c5ull, 0x6b0daeff4fcde703ull, 0x6b57fce8f09dd17full,
    0x6ba27e656b4eb57aull, 0x6bed33988bcbfab5ull, 0x6c381ca636d99642ull, 0x6c8339b26a25494eull,
    0x6cce8ae13c57ebdbull, 0x6d1a1056dd26c382ull, 0x6d65ca379564e639ull, 0x6db1b8a7c714a92bull,
    0x6dfddbcbed791babull, 0x6e4a33c89d278e49ull, 0x6e96c0c284192610ull, 0x6ee382de69bc7bf8ull,
    0x6f307a412f074892ull, 0x6f7da70fce881bf9ull, 0x6fcb096f5c782210ull, 0x7018a18506ccf314ull,
    0x70666f76154a7089ull, 0x70b47367e994ae92ull, 0x7102ad7fff41e9b4ull, 0x71511de3ebec8913ull,
    0x719fc4b95f452d29ull, 0x71eea2262324cb0cull, 0x723db6501b9ed447ull, 0x728d015d47136b40ull,
    0x72dc8373be41a454ull, 0x732c3cb9b459d38bull, 0x737c2d55770fe711ull, 0x73cc556d6eadce5full,
    0x741cb5281e25ee34ull, 0x746d4cac2325a155ull, 0x74be1c203627c62bull, 0x750f23ab2a87593eull,
    0x75606373ee921c97ull, 0x75b1dba18b9b4c20ull, 0x76038c5b260e5eeeull, 0x765575c7fd81d5a0ull,
    0x76a7980f6cca15c2ull, 0x76f9f358ea0c5249ull, 0x774c87cc06d1812eull, 0x779f559070195e36ull,
    0x77f25ccdee6d7ae6ull, 0x78459dac65f45bb5ull, 0x78991853d684a285ull, 0x78ecccec5bb84661ull,
    0x7940bb9e2cffd89dull, 0x7994e4919db5d74eull, 0x79e947ef1d320d2dull, 0x7a3de5df36dcfeefull,
    0x7a92be8a92436616ull, 0x7ae7d219f329b948ull, 0x7b3d20b6399fc237ull, 0x7b92aa886214411cull,
    0x7be86fb985689ddcull, 0x7c3e7072d904a6ceull, 0x7c94acddaeea5d3aull, 0x7ceb252375c9cf9bull,
    0x7d41d96db915019dull, 0x7d98c9e62113e1faull, 0x7deff6b672f84e24ull, 0x7e47600890f223deull,
    0x7e9f06067a4360baull, 0x7ef6e8da4b544f9aull, 0x7f4f08ae3dc7c426ull, 0x7fa765aca88f6453ull};

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

// The upper 64 bits of a b, at most 2 below (the product of the lower halves is left
// out).
__device__ __forceinline__ uint64_t mul_hi64(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32),
                 bl = (uint32_t)b;
  return (uint64_t)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}
// The same for a of 32 + S bits: cheaper, and at most 2 below too.
template <int S>
__device__ __forceinline__ uint64_t mul_hi_short(uint64_t a, uint32_t bh, uint32_t bl) {
  return (((uint64_t)(uint32_t)a * bh) >> 32) + (uint64_t)(uint32_t)(a >> 32) * bh +
         (__umulhi((uint32_t)(a >> S), bl) >> (32 - S));
}

// log2 E of a positive, normal E: exponent - log2 c + log2(m c), the last two in fixed
// point, rounded to 2^-52 as the fraction of a number in [1, 2].
__device__ __forceinline__ double log2_f64(double E) {
  const uint32_t h = (uint32_t)hi_word(E), l = (uint32_t)lo_word(E);
  const LogRow t = kLogTab[(h >> 13) & 127];
  const uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | l) << 11;
  // m c - 1 = rho/64, m c in units of 2^-62
  const uint64_t mc = (uint64_t)(uint32_t)(m >> 32) * t.c + __umulhi((uint32_t)m, t.c);
  const uint64_t rho = mc << 8;  // the 1 shifted out
  const uint32_t rh = (uint32_t)(rho >> 32), rl = (uint32_t)rho;
  const uint64_t B = kLog3 - __umulhi(kLog4 - __umulhi(kLog5 - __umulhi(kLog6, rh), rh), rh);
  const uint64_t C = kLog2 - mul_hi_short<6>(B, rh, rl);
  const uint64_t q = kLog1 - mul_hi_short<13>(C, rh, rl);
  const uint64_t f = ((t.log + mul_hi64(rho, q) + 16u) >> 5) + 0x3ff0000000000000ull;
  return f64_of_f32((float)((int)(h >> 20) - 1024)) + __longlong_as_double((long long)f);
}

// 1/E of a positive, normal E (0 above 2^1020): the FP32 reciprocal s of its
// mantissa m, and s (1 + d + d^2), d = 1 - m s, in fixed point.
__device__ __forceinline__ double rcp_f64(double E) {
  const uint32_t h = (uint32_t)hi_word(E), l = (uint32_t)lo_word(E);
  const uint32_t sb = __float_as_uint(
      fmaxf(__fdividef(1.0f, __uint_as_float(0x3f800000u | (h & 0xfffffu) << 3 | l >> 29)), 0.5f));
  const uint32_t S = ((sb & 0x7fffffu) | 0x800000u) << ((sb >> 23) - 126u);  // units of 2^-24
  // 1 - m s in units of 2^-76, below 2^-21: its low 64 bits are all of it
  const long long d =
      -(long long)((uint64_t)l * S + ((uint64_t)(((h & 0xfffffu) | 0x100000u) * S) << 32));
  const int dq = (int)(d >> 40);
  const long long t = (d >> 12) + ((uint32_t)(dq * dq) >> 8);  // d + d^2 in units of 2^-64
  const uint64_t q = ((uint64_t)S << 36) + (uint64_t)(((long long)S * (t >> 4)) >> 24);
  const uint64_t M = (q + 64u) >> 7;  // 53 bits, whose leading one adds 1 to the exponent field
  const int e = (int)(h >> 20) - 1023;
  return e > 1020 ? 0.0
                  : __hiloint2double((int)((uint32_t)(M >> 32) + (uint32_t)((1021 - e) << 20)),
                                     (int)(uint32_t)M);
}

// a / b for a normal b up to 2^1020.
__device__ __forceinline__ double div_f64(double a, double b) {
  const double r = rcp_f64(__longlong_as_double(__double_as_longlong(b) & 0x7fffffffffffffffll));
  return a * __hiloint2double(hi_word(r) ^ (hi_word(b) & (int)0x80000000), lo_word(r));
}

// 2^(Y 2^-53) in 64-bit integers, Y two's complement.  Y = n + i/256 + rho/256 (in those
// units): n the exponent, i the table entry T = 2^(i/256), rho in [0, 1) the rest; the result is
// 2^n (T + T p), p = 2^(rho/256) - 1 = rho/256 q(rho), q a cubic in units of 2^-52.
// `tiny`: of an exponent 256 larger, scaled back with one rounding (below the normal range).
__device__ __forceinline__ double exp2_fixed(uint64_t Y, bool tiny) {
  const int yh = (int)(Y >> 32);
  const uint64_t T = kExpTab[(yh >> 13) & 255];
  const uint64_t rho = Y << 19;
  const uint32_t rh = (uint32_t)(rho >> 32), rl = (uint32_t)rho;
  const uint64_t B = kExp2 + __umulhi(kExp3 + __umulhi(kExp4, rh), rh);
  const uint64_t q = kExp1 + mul_hi_short<10>(B, rh, rl);
  const uint64_t p = mul_hi64(rho, q);              // units of 2^-60
  const uint64_t S = T + (mul_hi64(T, p) << 4);     // units of 2^-62
  // rounded to 53 bits, whose leading one adds 1 to the exponent field
  const uint64_t M = (S + 512u) >> 10;
  const double v = __hiloint2double((int)((uint32_t)(M >> 32) + (uint32_t)(((yh >> 21) + 1022) << 20)),
                                    (int)(uint32_t)M);
  return tiny ? v * 0x1p-256 : v;
}

// The upper words of 1000 and of 100, the largest exponents of exp2_f64.
constexpr uint32_t kTop1000 = 0x408f4000u, kTopStep = 0x40590000u;

// 2^y; y is clamped to [-1200, 1000] (-1200: 0 after rounding), or to the number whose
// upper word is Top.
template <uint32_t Top = kTop1000>
__device__ __forceinline__ double exp2_f64(double y) {
  uint32_t h = (uint32_t)hi_word(y), l = (uint32_t)lo_word(y);
  const bool tiny = h >= 0xc08ff000u;  // y <= -1022: below the normal range
  if (tiny) {
    y = (h > 0xc092c000u ? -1200.0 : y) + 256.0;
    h = (uint32_t)hi_word(y);
    l = (uint32_t)lo_word(y);
  }
  if ((int)h >= (int)Top) {
    h = Top;
    l = 0;
  }
  // |y| in units of 2^-53, rounded where it has bits below
  const uint32_t s = 1032u - ((h >> 20) & 0x7ffu);
  uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | l) << 11;
  m = s < 64u ? ((m >> s) + 1u) >> 1 : 0u;
  return exp2_fixed((int)h < 0 ? 0u - m : m, tiny);
}

// e^z for z <= 0: |z| log2 e as a 64-bit product in units of 2^-53 (a product in FP64 would
// round it by |z| 2^-53 of the result, and cost the FP64 pipe an instruction).
__device__ __forceinline__ double exp_f64(double z) {
  const uint32_t h = min((uint32_t)hi_word(z) & 0x7fffffffu, 0x40875000u);  // 0 from -746 on
  const uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | (uint32_t)lo_word(z)) << 11;
  uint64_t P = mul_hi64(m, kLog2E);
  const uint32_t s = 1032u - (h >> 20);  // P is in units of 2^(-53 - s)
  if (s) P = s < 65u ? ((P >> (s - 1u)) + 1u) >> 1 : 0u;
  const bool tiny = P >= 1022ull << 53;
  if (tiny) P -= 256ull << 53;
  return exp2_fixed(0u - P, tiny);
}

}  // namespace ion
