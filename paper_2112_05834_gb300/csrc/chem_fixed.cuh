// Exponentials and logarithms of the rate evaluation in 64-bit fixed point.
//
// One FP64 warp instruction takes 64 cycles of an SM sub-partition on GB300 whatever its
// operands (19 cycles of the SM when all four issue them), a 32 x 32 + 64 bit integer
// multiply-add 4.4 and an integer add or shift 1 (measured with clock loops). The rate
// constants' arguments ln A + b ln T - Theta/T (+ dG/RT) have a known range, so they are
// formed and exponentiated as integers: no FP64 instruction from the temperature to the
// finished double, and 2^-52 absolute error in the argument where a double argument of
// 30 carries 2^-49.
//
// A value v in "Qn" is the 64-bit integer round(v 2^n). Method: table-driven reduction in
// the manner of P. T. P. Tang (ACM TOMS 15(2), 1989 and 16(4), 1990) with Taylor
// polynomials, each power evaluated to the bits it contributes.
#pragma once

#include <cstdint>

namespace chem {

// 2^(j/256) in units of 2^-62
static __device__ const unsigned long long g_fx_exp_tab[256] = {
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
    0x7e9f06067a4360baull, 0x7ef6e8da4b544f9aull, 0x7f4f08ae3dc7c426ull, 0x7fa765aca88f6453ull,
};
// c = 1 / (1 + (j + 1/2) / 256) rounded to 31 fractional bits, and -ln c (of the rounded c) in units of 2^-62
struct FxLog {
  unsigned long long lnc;
  unsigned c, pad;
};
static __device__ const FxLog g_fx_log_tab[256] = {
    {0x001ff802adab10e6ull, 0x7fc01ff0u, 0u}, {0x005fb8477120ba4full, 0x7f411e53u, 0u},
    {0x009f394b156d3ec8ull, 0x7ec31843u, 0u}, {0x00de7b896621c25eull, 0x7e460adau, 0u},
    {0x011d7f7ef9aebe6cull, 0x7dc9f339u, 0u}, {0x015c45a50f8d3889ull, 0x7d4ece90u, 0u},
    {0x019ace758a4c5145ull, 0x7cd49a16u, 0u}, {0x01d91a66c583cc3eull, 0x7c5b5311u, 0u},
    {0x021729ef97ac2ecfull, 0x7be2f6ceu, 0u}, {0x0254fd84295d0e63ull, 0x7b6b82a7u, 0u},
    {0x029295987432238full, 0x7af4f3feu, 0u}, {0x02cff29e1cd7b308ull, 0x7a7f4841u, 0u},
    {0x030d1505ecbed9dcull, 0x7a0a7ce7u, 0u}, {0x0349fd3fc07a469full, 0x79968f70u, 0u},
    {0x0386abb9eec3e59aull, 0x79237d66u, 0u}, {0x03c320e1bbec02b7ull, 0x78b1445cu, 0u},
    {0x03ff5d2237726067ull, 0x783fe1f0u, 0u}, {0x043b60e6d0c9bf83ull, 0x77cf53c6u, 0u},
    {0x04772c9927c65114ull, 0x775f978cu, 0u}, {0x04b2c0a0f7f787b9ull, 0x76f0aafau, 0u},
    {0x04ee1d662cedbb7dull, 0x76828bceu, 0u}, {0x0529434eac6c1004ull, 0x761537d0u, 0u},
    {0x056432bf58070a14ull, 0x75a8acd0u, 0u}, {0x059eec1c88f03ee5ull, 0x753ce8a5u, 0u},
    {0x05d96fc8e9ef84d1ull, 0x74d1e92fu, 0u}, {0x0613be267e4a0a8dull, 0x7467ac55u, 0u},
    {0x064dd7957997b771ull, 0x73fe3007u, 0u}, {0x0687bc75d6473506ull, 0x7395723bu, 0u},
    {0x06c16d26bc10ff92ull, 0x732d70eeu, 0u}, {0x06faea05e359d922ull, 0x72c62a25u, 0u},
    {0x073433701404f854ull, 0x725f9becu, 0u}, {0x076d49c087b649deull, 0x71f9c457u, 0u},
    {0x07a62d528a0519ddull, 0x7194a17fu, 0u}, {0x07dede7fbd1f77b4ull, 0x71303185u, 0u},
    {0x08175da12b9ea570ull, 0x70cc7290u, 0u}, {0x084fab0f3ccce19full, 0x706962cdu, 0u},
    {0x0887c721169cd899ull, 0x70070070u, 0u}, {0x08bfb22c8f53087full, 0x6fa549b4u, 0u},
    {0x08f76c8745a16156ull, 0x6f443cd9u, 0u}, {0x092ef6856fb568e1ull, 0x6ee3d826u, 0u},
    {0x0966507af5392844ull, 0x6e8419e7u, 0u}, {0x099d7abad10727b3ull, 0x6e25006eu, 0u},
    {0x09d475966fd1bafcull, 0x6dc68a14u, 0u}, {0x0a0b415ff87ddff7ull, 0x6d68b535u, 0u},
    {0x0a41de662bb1eea5ull, 0x6d0b8037u, 0u}, {0x0a784cfa31185903ull, 0x6caee980u, 0u},
    {0x0aae8d6a48d6b765ull, 0x6c52ef7fu, 0u}, {0x0ae4a0037ef95c9bull, 0x6bf790a9u, 0u},
    {0x0b1a85149853abd8ull, 0x6b9ccb74u, 0u}, {0x0b503ce8b3d568feull, 0x6b429e60u, 0u},
    {0x0b85c7cbfe153a99ull, 0x6ae907efu, 0u}, {0x0bbb260947d093a5ull, 0x6a9006a9u, 0u},
    {0x0bf057eb2de139e8ull, 0x6a37991au, 0u}, {0x0c255dbadc289c95ull, 0x69dfbdd4u, 0u},
    {0x0c5a37c137712d9full, 0x6988736du, 0u}, {0x0c8ee6463a05ef1bull, 0x6931b880u, 0u},
    {0x0cc3699185c064edull, 0x68db8bacu, 0u}, {0x0cf7c1e922cd19e9ull, 0x6885eb96u, 0u},
    {0x0d2bef93e7e6e672ull, 0x6830d6e5u, 0u}, {0x0d5ff2d7008925c3ull, 0x67dc4c46u, 0u},
    {0x0d93cbf71c9905ddull, 0x67884a6au, 0u}, {0x0dc77b3868861d4dull, 0x6734d006u, 0u},
    {0x0dfb00dd46e270d5ull, 0x66e1dbd5u, 0u}, {0x0e2e5d2a01f21254ull, 0x668f6c92u, 0u},
    {0x0e61905fcbb28121ull, 0x663d8100u, 0u}, {0x0e949ac11119f364ull, 0x65ec17e3u, 0u},
    {0x0ec77c8db20eaefaull, 0x659b3006u, 0u}, {0x0efa36061a9697a1ull, 0x654ac836u, 0u},
    {0x0f2cc76a9d7f1766ull, 0x64fadf43u, 0u}, {0x0f5f30fa293d8576ull, 0x64ab7402u, 0u},
    {0x0f9172f383c82eacull, 0x645c854bu, 0u}, {0x0fc38d93fd682281ull, 0x640e11fbu, 0u},
    {0x0ff58119f703e62eull, 0x63c018f0u, 0u}, {0x10274dc1a9a32f3dull, 0x6372990eu, 0u},
    {0x1058f3c708ebc5e6ull, 0x6325913cu, 0u}, {0x108a73666317af07ull, 0x62d90063u, 0u},
    {0x10bbccdb1124bccbull, 0x628ce570u, 0u}, {0x10ed005f6e7da471ull, 0x62413f54u, 0u},
    {0x111e0e2d77dcb701ull, 0x61f60d03u, 0u}, {0x114ef67f6d285a16ull, 0x61ab4d73u, 0u},
    {0x117fb98dd5495d5dull, 0x6160ff9fu, 0u}, {0x11b05792163b48aeull, 0x61172283u, 0u},
    {0x11e0d0c325d6be3dull, 0x60cdb521u, 0u}, {0x1211255976d60b9eull, 0x6084b67bu, 0u},
    {0x1241558c51540400ull, 0x603c2597u, 0u}, {0x127161911f853d3dull, 0x5ff40180u, 0u},
    {0x12a1499f662bc910ull, 0x5fac4940u, 0u}, {0x12d10dec16458319ull, 0x5f64fbe7u, 0u},
    {0x1300aeacdcb50bd6ull, 0x5f1e1886u, 0u}, {0x13302c161ae58860ull, 0x5ed79e32u, 0u},
    {0x135f865ce5e93e09ull, 0x5e918c01u, 0u}, {0x138ebdb3a09320b0ull, 0x5e4be10fu, 0u},
    {0x13bdd24eb18b6a13ull, 0x5e069c77u, 0u}, {0x13ecc4611d5f4fecull, 0x5dc1bd58u, 0u},
    {0x141b941c7dcbee5cull, 0x5d7d42d5u, 0u}, {0x144a41b467c47b8aull, 0x5d392c10u, 0u},
    {0x1478cd599d73d914ull, 0x5cf57831u, 0u}, {0x14a7373cc3799773ull, 0x5cb22662u, 0u},
    {0x14d57f8fbfa27f25ull, 0x5c6f35cdu, 0u}, {0x1503a682f31cb2e7ull, 0x5c2ca5a0u, 0u},
    {0x1531ac4531a77e0full, 0x5bea750du, 0u}, {0x155f9107e93ee19cull, 0x5ba8a344u, 0u},
    {0x158d54f827c2f23full, 0x5b672f7du, 0u}, {0x15baf846f51b1946ull, 0x5b2618ecu, 0u},
    {0x15e87b20eb5549f4ull, 0x5ae55ecdu, 0u}, {0x1615ddb47e813c7dull, 0x5aa5005bu, 0u},
    {0x1643203095c7bf81ull, 0x5a64fcd2u, 0u}, {0x167042c0477e30a5ull, 0x5a255375u, 0u},
    {0x169d45929d762c6full, 0x59e60383u, 0u}, {0x16ca28d2c5c98568ull, 0x59a70c42u, 0u},
    {0x16f6ecadbc62920bull, 0x59686cf7u, 0u}, {0x1723914eb7c0e0ebull, 0x592a24ebu, 0u},
    {0x175016e0907a6206ull, 0x58ec3369u, 0u}, {0x177c7d8fe7791410ull, 0x58ae97bbu, 0u},
    {0x17a8c586d1f5441full, 0x58715130u, 0u}, {0x17d4eeefb4ec6dfdull, 0x58345f18u, 0u},
    {0x1800f9f3cf14caf4ull, 0x57f7c0c6u, 0u}, {0x182ce6be1d4d9cdaull, 0x57bb758cu, 0u},
    {0x1858b576fa8c42aeull, 0x577f7cc1u, 0u}, {0x188466487ac623faull, 0x5743d5bbu, 0u},
    {0x18aff95ac1177fe9ull, 0x57087fd4u, 0u}, {0x18db6ed570272ca8ull, 0x56cd7a68u, 0u},
    {0x1906c6e1ddc7539full, 0x5692c4d2u, 0u}, {0x193201a7619336a2ull, 0x56585e71u, 0u},
    {0x195d1f4d868a0a20ull, 0x561e46a5u, 0u}, {0x19881ffb4aa6f00dull, 0x55e47cd0u, 0u},
    {0x19b303d71ab61f1dull, 0x55ab0056u, 0u}, {0x19ddcb084da7419cull, 0x5571d09bu, 0u},
    {0x1a0875b4e49d170cull, 0x5538ed06u, 0u}, {0x1a33040244fa6373ull, 0x55005500u, 0u},
    {0x1a5d7615f56c3714ull, 0x54c807f3u, 0u}, {0x1a87cc165df1991eull, 0x54900549u, 0u},
    {0x1ab20627bfa09faaull, 0x54584c70u, 0u}, {0x1adc246f3668ff2bull, 0x5420dcd6u, 0u},
    {0x1b06271070141b56ull, 0x53e9b5ecu, 0u}, {0x1b300e30b482a342ull, 0x53b2d722u, 0u},
    {0x1b59d9f3d7e7c263ull, 0x537c3febu, 0u}, {0x1b838a7cf8c1efdfull, 0x5345efbcu, 0u},
    {0x1bad1fef40d16572ull, 0x530fe60bu, 0u}, {0x1bd69a6ea90c4717ull, 0x52da224eu, 0u},
    {0x1bfffa1ce150844dull, 0x52a4a3ffu, 0u}, {0x1c293f1def937bebull, 0x526f6a96u, 0u},
    {0x1c526992c2cf6b08ull, 0x523a7590u, 0u}, {0x1c7b799e9d6eaf82ull, 0x5205c468u, 0u},
    {0x1ca46f626974e684ull, 0x51d1569du, 0u}, {0x1ccd4b009ae5ef30ull, 0x519d2badu, 0u},
    {0x1cf60c9944aad984ull, 0x5169431au, 0u}, {0x1d1eb44ec9b4c962ull, 0x51359c64u, 0u},
    {0x1d4742405addd58bull, 0x51023710u, 0u}, {0x1d6fb6904107ea1dull, 0x50cf12a0u, 0u},
    {0x1d98115e5679b635ull, 0x509c2e9au, 0u}, {0x1dc052c994f9abffull, 0x50698a86u, 0u},
    {0x1de87af342671a80ull, 0x503725eau, 0u}, {0x1e1089fa29d1683full, 0x50050050u, 0u},
    {0x1e387ffdc70d75c6ull, 0x4fd31942u, 0u}, {0x1e605d1d79892eefull, 0x4fa1704bu, 0u},
    {0x1e882178825d51b1ull, 0x4f7004f7u, 0u}, {0x1eafcd2d339d7127ull, 0x4f3ed6d4u, 0u},
    {0x1ed76059bb263b51ull, 0x4f0de571u, 0u}, {0x1efedb1c20aa0802ull, 0x4edd305eu, 0u},
    {0x1f263d93e43bb759ull, 0x4eacb72au, 0u}, {0x1f4d87dd1cd7e5efull, 0x4e7c7969u, 0u},
    {0x1f74ba16f66c7cdfull, 0x4e4c76acu, 0u}, {0x1f9bd45dfd9ea3b4ull, 0x4e1cae88u, 0u},
    {0x1fc2d6cf5f4f1a14ull, 0x4ded2092u, 0u}, {0x1fe9c188165cff14ull, 0x4dbdcc60u, 0u},
    {0x201094a4e9a70bd2ull, 0x4d8eb189u, 0u}, {0x203750433dcb470bull, 0x4d5fcfa4u, 0u},
    {0x205df47e98e5372aull, 0x4d31264bu, 0u}, {0x2084817319ca9843ull, 0x4d02b518u, 0u},
    {0x20aaf73ca3469b5bull, 0x4cd47ba6u, 0u}, {0x20d155f7afd3b435ull, 0x4ca67990u, 0u},
    {0x20f79dbfa593fadfull, 0x4c78ae73u, 0u}, {0x211dceaed1c8260dull, 0x4c4b19eeu, 0u},
    {0x2143e8e29885234aull, 0x4c1dbb9du, 0u}, {0x2169ec73e6e851eeull, 0x4bf09322u, 0u},
    {0x218fd97ebeca65adull, 0x4bc3a01cu, 0u}, {0x21b5b01d2a30f58bull, 0x4b96e22du, 0u},
    {0x21db7069bffebbeaull, 0x4b6a58f7u, 0u}, {0x22011a7ecaa28c3cull, 0x4b3e041du, 0u},
    {0x2226ae7646050308ull, 0x4b11e343u, 0u}, {0x224c2c6ab834f493ull, 0x4ae5f60du, 0u},
    {0x22719474a0129eb8ull, 0x4aba3c22u, 0u}, {0x2296e6aeb8f9a227ull, 0x4a8eb527u, 0u},
    {0x22bc23328f29c762ull, 0x4a6360c3u, 0u}, {0x22e14a187b2e939full, 0x4a383e9fu, 0u},
    {0x23065b7957c5b1b1ull, 0x4a0d4e64u, 0u}, {0x232b576e82443311ull, 0x49e28fbbu, 0u},
    {0x23503e10fcbaacf3ull, 0x49b8024eu, 0u}, {0x23750f796bd83572ull, 0x498da5c8u, 0u},
    {0x2399cbbf358c449aull, 0x496379d6u, 0u}, {0x23be72fb1ba77d2bull, 0x49397e24u, 0u},
    {0x23e305457e3b60d8ull, 0x490fb25fu, 0u}, {0x240782b578b8f3b1ull, 0x48e61636u, 0u},
    {0x242beb63810e5259ull, 0x48bca957u, 0u}, {0x24503f66c5433ea0ull, 0x48936b72u, 0u},
    {0x24747ed6eb54a606ull, 0x486a5c37u, 0u}, {0x2498a9ca4c0f25a3ull, 0x48417b58u, 0u},
    {0x24bcc0597b688edcull, 0x4818c885u, 0u}, {0x24e0c29adb18703full, 0x47f04371u, 0u},
    {0x2504b0a45befa5ddull, 0x47c7ebd0u, 0u}, {0x25288a8e29eef462ull, 0x479fc154u, 0u},
    {0x254c506d521cb226ull, 0x4777c3b3u, 0u}, {0x257002591b598155ull, 0x474ff2a1u, 0u},
    {0x2593a06772b41e58ull, 0x47284dd4u, 0u}, {0x25b72aaeb43c458dull, 0x4700d502u, 0u},
    {0x25daa143dcd4b352ull, 0x46d987e3u, 0u}, {0x25fe043d3cc4415eull, 0x46b2662eu, 0u},
    {0x262153b0aa062452ull, 0x468b6f9bu, 0u}, {0x26448fb466d94c71ull, 0x4664a3e2u, 0u},
    {0x2667b85c664eec48ull, 0x463e02beu, 0u}, {0x268acdbdec18281full, 0x46178be9u, 0u},
    {0x26adcfeea512f0f1ull, 0x45f13f1du, 0u}, {0x26d0bf03bcd60d9eull, 0x45cb1c15u, 0u},
    {0x26f39b11db7c550eull, 0x45a5228du, 0u}, {0x2716642d236f1be4ull, 0x457f5242u, 0u},
    {0x27391a6b07afd854ull, 0x4559aaf0u, 0u}, {0x275bbddf8860febbull, 0x45342c55u, 0u},
    {0x277e4e9e1b4e1967ull, 0x450ed630u, 0u}, {0x27a0ccbc72f31e2aull, 0x44e9a83eu, 0u},
    {0x27c3384cee43040eull, 0x44c4a240u, 0u}, {0x27e59165162d9ba2ull, 0x449fc3f4u, 0u},
    {0x2807d8171aa4ac45ull, 0x447b0d1cu, 0u}, {0x282a0c78572058b6ull, 0x44567d77u, 0u},
    {0x284c2e9bb8e2cd4full, 0x443214c7u, 0u}, {0x286e3e93993b3a17ull, 0x440dd2cfu, 0u},
    {0x28903c748f081b02ull, 0x43e9b750u, 0u}, {0x28b22851acf8d082ull, 0x43c5c20du, 0u},
    {0x28d4023d6f0e8aa3ull, 0x43a1f2cau, 0u}, {0x28f5ca4aab1c88ceull, 0x437e494bu, 0u},
    {0x2917808c9107b056ull, 0x435ac554u, 0u}, {0x29392515b7457be8ull, 0x433766aau, 0u},
    {0x295ab7f90cda45dcull, 0x43142d12u, 0u}, {0x297c3948e4d6ef87ull, 0x42f11852u, 0u},
    {0x299da917e955e776ull, 0x42ce2830u, 0u}, {0x29bf077730379095ull, 0x42ab5c74u, 0u},
    {0x29e0547a0f5e0c30ull, 0x4288b4e4u, 0u}, {0x2a01903246e868b9ull, 0x42663148u, 0u},
    {0x2a22bab1eaed3739ull, 0x4243d168u, 0u}, {0x2a43d4097434893aull, 0x4221950eu, 0u},
    {0x2a64dc4c94b15910ull, 0x41ff7c01u, 0u}, {0x2a85d38b71fa5e4aull, 0x41dd860cu, 0u},
    {0x2aa6b9d87302500aull, 0x41bbb2f8u, 0u}, {0x2ac78f445e4f9713ull, 0x419a0290u, 0u},
    {0x2ae853e049b37142ull, 0x4178749fu, 0u}, {0x2b0907be95408820ull, 0x415708efu, 0u},
    {0x2b29aaef0100fc52ull, 0x4135bf4du, 0u}, {0x2b4a3d83906be771ull, 0x41149784u, 0u},
    {0x2b6abf8c9e9a560dull, 0x40f39161u, 0u}, {0x2b8b311ad2fbbb5aull, 0x40d2acb1u, 0u},
    {0x2bab923f2189e03bull, 0x40b1e941u, 0u}, {0x2bcbe309cd3c4f27ull, 0x409146dfu, 0u},
    {0x2bec238b63fb3e80ull, 0x4070c559u, 0u}, {0x2c0c53d3c011fae4ull, 0x4050647eu, 0u},
    {0x2c2c73f503a0d2eaull, 0x4030241bu, 0u}, {0x2c4c83fd9f4e85e2ull, 0x40100401u, 0u},
};

// High 64 bits of a b for a signed and b unsigned: a in Qm and b in Qn give Q(m + n - 64).
__device__ __forceinline__ long long fx_mul(long long a, unsigned long long b) {
  return (long long)(__umul64hi((unsigned long long)a, b) - ((unsigned long long)(a >> 63) & b));
}

// a + b and a - b modulo the format: partial sums may leave it when the whole sum does not.
__device__ __forceinline__ long long fx_add(long long a, long long b) {
  return (long long)((unsigned long long)a + (unsigned long long)b);
}
__device__ __forceinline__ long long fx_sub(long long a, long long b) {
  return (long long)((unsigned long long)a - (unsigned long long)b);
}

// A positive double's significand (2^52 .. 2^53) shifted left by its exponent plus sh,
// i.e. the value in Q(52 + sh); the caller's range makes the shift count 0 .. 11.
__device__ __forceinline__ unsigned long long fx_scale(double x, int sh) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return ((b & 0xfffffffffffffull) | 0x10000000000000ull) << (((int)(b >> 52) - 1023 + sh) & 63);
}

// exp(x) of x in Q52, as a double; results outside the normal numbers are taken as about
// the smallest or the largest of them.
// x = N ln2/256 + r with |r| <= ln2/512 (1 + 2^-8), exp(x) = 2^(N/256) (1 + r + r^2/2 +
// r^3/6 + r^4/24 + r^5/120); r and the bracket in Q62, r^2 from the two halves of r, the
// cubic tail (below 2^-31) from 32-bit factors. Error before the final rounding below
// 2^-58 relative.
// tab: g_fx_exp_tab or a copy of it in shared memory.
__device__ __forceinline__ double fx_exp(long long x, const unsigned long long* tab) {
  constexpr int kInvL = 1549082005;                           // 256/ln2, Q22
  constexpr unsigned long long kL = 0x2c5c85fdf473deull;      // ln2/256, Q62, rounded down
  constexpr unsigned kLlo = 1794275565u;                      // the rest, Q94
  constexpr int kLo = -742798459, kHi = 744254700;  // -708.388, 709.777 in Q20
  x = (long long)min(max((int)(x >> 32), kLo), kHi) << 32 | (unsigned)x;
  const int N = ((int)(((long long)(int)(x >> 32) * kInvL) >> 32) + 512) >> 10;
  const long long r = (long long)(((unsigned long long)x << 10) - (unsigned long long)(long long)N * kL) -
                      (((long long)N * (long long)kLlo) >> 32);
  const int rh = (int)(r >> 22);               // Q40
  const int rl = (int)((unsigned)r & 0x3fffffu);
  const long long sq = (long long)rh * rh;     // Q80
  const int r2 = (int)(sq >> 32);              // Q48
  const int r3 = (int)(((long long)r2 * rh) >> 29);  // Q59
  // (1/6)(1 + r/4 + r^2/20), Q32
  const int u = 715827883 + __mulhi(rh, 699051) + (r2 >> 23);
  const long long em1 = r + (sq >> 19) + (((long long)rh * rl) >> 40) + (((long long)r3 * u) >> 29);
  const unsigned long long t = tab[N & 255];
  const int th = (int)(t >> 32), tl = (int)((unsigned)t >> 1);
  const int eh = (int)(em1 >> 22), el = (int)((unsigned)em1 & 0x3fffffu);
  long long v = (long long)t + (((long long)eh * th) >> 8) + (((long long)eh * tl) >> 39) + (((long long)el * th) >> 30);
  int e = (N >> 8) + 1022;
  if (!(v >> 62)) {  // below 1: the interval around j = 0 reaches under a power of two
    v <<= 1;
    --e;
  }
  return __longlong_as_double(((long long)e << 52) + ((v + 512) >> 10));
}

// ln x of a positive normal double in Q52 or Q58 (|ln x| must fit): x = 2^e m,
// z = m c - 1 with c = 1/(1 + (j + 1/2)/256) to 31 bits, |z| < 2^-9, and ln x = e ln2 -
// ln c + z - z^2/2 + z^3 (1/3 - z/4 + z^2/5 - z^3/6). Error below 2^-51 (Q52), 2^-56 (Q58).
// Out of line: it is called once or twice per rate evaluation.
static __device__ __noinline__ long long fx_log(double x, int Q) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) - 1023;
  const int j = (int)(b >> 44) & 255;
  const FxLog t = g_fx_log_tab[j];
  const unsigned mh = ((unsigned)(b >> 32) & 0xfffffu) | 0x100000u, ml = (unsigned)b;
  const long long z = (long long)(((unsigned long long)mh * t.c << 11) + (((unsigned long long)ml * t.c) >> 21) -
                                  (1ull << 62));
  const int zh = (int)(z >> 22);  // Q40
  const int zl = (int)((unsigned)z & 0x3fffffu);
  const long long sq = (long long)zh * zh;           // Q80
  const int z2 = (int)(sq >> 32);                    // Q48
  const int z3 = (int)(((long long)z2 * zh) >> 30);  // Q58
  // 1/3 - z/4 + z^2/5 - z^3/6, Q32
  const int u = 1431655765 - (zh >> 10) + (__mulhi(z2, 858993459) >> 16) - (z3 >> 29);
  const long long f = (long long)t.lnc + z - (sq >> 19) - (((long long)zh * zl) >> 40) + (((long long)z3 * u) >> 28);
  const long long ln2 = Q == 52 ? 0xb17217f7d1cf7ll : 0x2c5c85fdf473de6ll;
  const long long ln2_lo = Q == 52 ? 2596052539ll : 2938605262ll;  // ln2 Q(Q + 32) - ln2 2^32
  return e * ln2 + ((e * ln2_lo) >> 32) + (f >> (62 - Q));
}

// Double to Q52, truncated; |x| >= 1024 and infinities saturate beyond +-1024 (NaN too).
__device__ __forceinline__ long long fx_from_double(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffu) - 1023;
  const long long m = (long long)((b & 0xfffffffffffffull) | 0x10000000000000ull);
  const long long v = e >= 0 ? m << min(e, 10) : m >> min(-e, 63);
  return (long long)b < 0 ? -v : v;
}

// Q52 to double, rounded to nearest (ties up).
__device__ __forceinline__ double fx_to_double(long long v) {
  const unsigned long long s = (unsigned long long)v & 0x8000000000000000ull;
  unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
  const int lz = __clzll((long long)a);
  a <<= lz & 63;  // leading bit at 63
  const unsigned long long bits = ((unsigned long long)(1023 + 11 - lz - 1) << 52) + (((a >> 10) + 1) >> 1);
  return v == 0 ? 0.0 : __longlong_as_double((long long)(bits | s));
}

}  // namespace chem
