// Generated by gen_fixed_tables.py; do not edit.
#pragma once
// 2^(j / 256) times 2^62, j = 0 .. 255
#define CHEM_FX_EXP2_VALUES \
    0x4000000000000000ull, 0x402c6be96af2fb58ull, 0x4058f6a7ecccd5b6ull, 0x4085a050ec0a036aull, \
    0x40b268f9de0183baull, 0x40df50b846ef302bull, 0x410c57a1b9fe12f6ull, 0x41397dcbd952c4a6ull, \
    0x4166c34c5615d0ecull, 0x41942838f07e22a3ull, 0x41c1aca777db771bull, 0x41ef50adcaa0d899ull, \
    0x421d1461d66f2023ull, 0x424af7d9981f7e98ull, 0x4278fb2b1bce0d15ull, 0x42a71e6c7ce464afull, \
    0x42d561b3e6243d8aull, 0x4303c51791b21550ull, 0x433248adc91fdd02ull, 0x4360ec8ce577ae44ull, \
    0x438fb0cb4f468808ull, 0x43be957f7ea712b6ull, 0x43ed9abffb4c6bc9ull, 0x441cc0a35c8cf8eaull, \
    0x444c0740496d4294ull, 0x447b6ead78aad636ull, 0x44aaf701b0c72feeull, 0x44daa053c812abd2ull, \
    0x450a6abaa4b77ecdull, 0x453a564d3cc4b723ull, 0x456a632296394492ull, 0x459a9151c70f0819ull, \
    0x45cae0f1f545eb73ull, 0x45fb521a56ef0042ull, 0x462be4e23237a6efull, 0x465c9960dd74bd4bull, \
    0x468d6fadbf2dd4f3ull, 0x46be67e04e28717cull, 0x46ef821011734e6bull, 0x4720be54a071ad01ull, \
    0x47521cc5a2e6a9e0ull, 0x47839d7ad1009a90ull, 0x47b5408bf36472e2ull, 0x47e70610e3393241ull, \
    0x4818ee218a3358eeull, 0x484af8d5e2a06536ull, 0x487d2645f7725895ull, 0x48af7689e44b44eaull, \
    0x48e1e9b9d588e19bull, 0x49147fee085028d6ull, 0x4947393eca98fcd6ull, 0x497a15c47b39d53eull, \
    0x49ad159789f37496ull, 0x49e038d0777ca5e0ull, 0x4a137f87d58e025bull, 0x4a46e9d646edbf6aull, \
    0x4a7a77d47f7b84b1ull, 0x4aae299b443c4a6bull, 0x4ae1ff436b663ff7ull, 0x4b15f8e5dc6cbab0ull, \
    0x4b4a169b900c2d00ull, 0x4b7e587d905625d1ull, 0x4bb2bea4f8bd5847ull, 0x4be7492af621abd6ull, \
    0x4c1bf828c6dc54b8ull, 0x4c50cbb7bacbf4cbull, 0x4c85c3f13360c4d5ull, 0x4cbae0eea3a8c63cull, \
    0x4cf022c9905bfd32ull, 0x4d25899b8fe8b365ull, 0x4d5b157e4a7fc325ull, 0x4d90c68b7a20eb1eull, \
    0x4dc69cdceaa72a9cull, 0x4dfc988c79d52661ull, 0x4e32b9b417619617ull, 0x4e69006dc503ba65ull, \
    0x4e9f6cd3967fdba8ull, 0x4ed5feffb1b3d155ull, 0x4f0cb70c4ea39210ull, 0x4f439513b785cc80ull, \
    0x4f7a993048d088d7ull, 0x4fb1c37c7145d328ull, 0x4fe91412b2006e83ull, 0x50208b0d9e8090dfull, \
    0x50582887dcb8a7e1ull, 0x508fec9c251a267cull, 0x50c7d76542a25b72ull, 0x50ffe8fe12e750c4ull, \
    0x513821818624b40cull, 0x5170810a9f48c7cfull, 0x51a907b474015dc9ull, 0x51e1b59a2cc8da3eull, \
    0x521a8ad704f3404full, 0x525387864abb4762ull, 0x528cabc35f4f799dull, 0x52c5f7a9b6df5b77ull, \
    0x52ff6b54d8a89c75ull, 0x533906e05f045106ull, 0x5372ca67f774358full, 0x53acb60762affaaeull, \
    0x53e6c9da74b29ab5ull, 0x542105fd14c7b869ull, 0x545b6a8b3d990704ull, 0x5495f7a0fd3bbb8eull, \
    0x54d0ad5a753e077cull, 0x550b8bd3dab49cbdull, 0x5546932976483b15ull, 0x5581c377a44346f0ull, \
    0x55bd1cdad49f699cull, 0x55f89f6f8b133af4ull, 0x56344b525f1ff495ull, 0x5670209ffc1f2e82ull, \
    0x56ac1f752150a563ull, 0x56e847eea1e80a49ull, 0x57249a29651adc07ull, 0x57611642662e4a33ull, \
    0x579dbc56b48521baull, 0x57da8c8373adc331ull, 0x581786e5db7022c2ull, 0x5854ab9b37dbd1e5ull, \
    0x5891fac0e95612c8ull, 0x58cf747464a7f584ull, 0x590d18d3330c7f1eull, 0x594ae7faf23eda52ull, \
    0x5988e20954889245ull, 0x59c7071c20cfd70cull, 0x5a05575132a5cc20ull, 0x5a43d2c67a54e0c0ull, \
    0x5a827999fcef3242ull, 0x5ac14be9d45cf869ull, 0x5b0049d42f6afbb6ull, 0x5b3f737751d915c8ull, \
    0x5b7ec8f19468bbc9ull, 0x5bbe4a6164eb92f4ull, 0x5bfdf7e546520f3eull, 0x5c3dd19bd0ba1c1aull, \
    0x5c7dd7a3b17dcf75ull, 0x5cbe0a1bab4226dfull, 0x5cfe69229605cef5ull, 0x5d3ef4d75f2ff504ull, \
    0x5d7fad59099f22feull, 0x5dc092c6adb825b8ull, 0x5e01a53f7974fd86ull, 0x5e42e4e2b073d935ull, \
    0x5e8451cfac061b5full, 0x5ec5ec25db3f6a41ull, 0x5f07b404c304c9f1ull, 0x5f49a98bfe1bc11cull, \
    0x5f8bccdb3d398841ull, 0x5fce1e124712437cull, 0x60109d50f86846d8ull, 0x60534ab7441b6546ull, \
    0x6096266533384a2bull, 0x60d9307ae507dd9aull, 0x611c69188f1eb339ull, 0x615fd05e7d6c83e4ull, \
    0x61a3666d124bb204ull, 0x61e72b64c690d8afull, 0x622b1f66299a6599ull, 0x626f4291e1603dd5ull, \
    0x62b39508aa836d6full, 0x62f816eb585de1edull, 0x633cc85ad5122fbdull, 0x6381a978219b628full, \
    0x63c6ba6455dcd8aeull, 0x640bfb40a0b22959ull, 0x64516c2e47ff1623ull, 0x64970d4ea8bf8766ull, \
    0x64dcdec3371793d1ull, 0x6522e0ad7e639312ull, 0x6569132f21483ba7ull, 0x65af7669d9c2cbe4ull, \
    0x65f60a7f79393e2eull, 0x663ccf91e88a8873ull, 0x6683c5c3281ee6e9ull, 0x66caed354ff83222ull, \
    0x6712460a8fc24072ull, 0x6759d0652ee352afull, 0x67a18c678c8c8c61ull, 0x67e97a341fca775bull, \
    0x683199ed779592caull, 0x6879ebb63ae2edc6ull, 0x68c26fb128b4cd63ull, 0x690b2601182b5e56ull, \
    0x69540ec8f895722dull, 0x699d2a2bd181482aull, 0x69e6784cc2cd61bdull, 0x6a2ff94f04b962b0ull, \
    0x6a79ad55e7f6fd10ull, 0x6ac39484d5bae8c5ull, 0x6b0daeff4fcde703ull, 0x6b57fce8f09dd17full, \
    0x6ba27e656b4eb57aull, 0x6bed33988bcbfab5ull, 0x6c381ca636d99642ull, 0x6c8339b26a25494eull, \
    0x6cce8ae13c57ebdbull, 0x6d1a1056dd26c382ull, 0x6d65ca379564e639ull, 0x6db1b8a7c714a92bull, \
    0x6dfddbcbed791babull, 0x6e4a33c89d278e49ull, 0x6e96c0c284192610ull, 0x6ee382de69bc7bf8ull, \
    0x6f307a412f074892ull, 0x6f7da70fce881bf9ull, 0x6fcb096f5c782210ull, 0x7018a18506ccf314ull, \
    0x70666f76154a7089ull, 0x70b47367e994ae92ull, 0x7102ad7fff41e9b4ull, 0x71511de3ebec8913ull, \
    0x719fc4b95f452d29ull, 0x71eea2262324cb0cull, 0x723db6501b9ed447ull, 0x728d015d47136b40ull, \
    0x72dc8373be41a454ull, 0x732c3cb9b459d38bull, 0x737c2d55770fe711ull, 0x73cc556d6eadce5full, \
    0x741cb5281e25ee34ull, 0x746d4cac2325a155ull, 0x74be1c203627c62bull, 0x750f23ab2a87593eull, \
    0x75606373ee921c97ull, 0x75b1dba18b9b4c20ull, 0x76038c5b260e5eeeull, 0x765575c7fd81d5a0ull, \
    0x76a7980f6cca15c2ull, 0x76f9f358ea0c5249ull, 0x774c87cc06d1812eull, 0x779f559070195e36ull, \
    0x77f25ccdee6d7ae6ull, 0x78459dac65f45bb5ull, 0x78991853d684a285ull, 0x78ecccec5bb84661ull, \
    0x7940bb9e2cffd89dull, 0x7994e4919db5d74eull, 0x79e947ef1d320d2dull, 0x7a3de5df36dcfeefull, \
    0x7a92be8a92436616ull, 0x7ae7d219f329b948ull, 0x7b3d20b6399fc237ull, 0x7b92aa886214411cull, \
    0x7be86fb985689ddcull, 0x7c3e7072d904a6ceull, 0x7c94acddaeea5d3aull, 0x7ceb252375c9cf9bull, \
    0x7d41d96db915019dull, 0x7d98c9e62113e1faull, 0x7deff6b672f84e24ull, 0x7e47600890f223deull, \
    0x7e9f06067a4360baull, 0x7ef6e8da4b544f9aull, 0x7f4f08ae3dc7c426ull, 0x7fa765aca88f6453ull \

// reciprocals c_j times 2^16 and their logarithms -log2(c_j) times 2^60, j = 0 .. 127
#define CHEM_FX_RCP_VALUES \
    0x0ff01u, 0x0fd09u, 0x0fb19u, 0x0f930u, 0x0f74eu, 0x0f574u, 0x0f3a1u, 0x0f1d5u, \
    0x0f00fu, 0x0ee50u, 0x0ec98u, 0x0eae5u, 0x0e939u, 0x0e793u, 0x0e5f3u, 0x0e459u, \
    0x0e2c5u, 0x0e136u, 0x0dfacu, 0x0de28u, 0x0dca9u, 0x0db2fu, 0x0d9bau, 0x0d84au, \
    0x0d6dfu, 0x0d579u, 0x0d417u, 0x0d2bau, 0x0d161u, 0x0d00du, 0x0cebdu, 0x0cd71u, \
    0x0cc29u, 0x0cae6u, 0x0c9a6u, 0x0c86au, 0x0c733u, 0x0c5feu, 0x0c4ceu, 0x0c3a1u, \
    0x0c278u, 0x0c152u, 0x0c030u, 0x0bf11u, 0x0bdf6u, 0x0bcddu, 0x0bbc8u, 0x0bab6u, \
    0x0b9a8u, 0x0b89cu, 0x0b793u, 0x0b68du, 0x0b58au, 0x0b48au, 0x0b38du, 0x0b292u, \
    0x0b19bu, 0x0b0a6u, 0x0afb3u, 0x0aec3u, 0x0add6u, 0x0acebu, 0x0ac03u, 0x0ab1du, \
    0x0aa39u, 0x0a958u, 0x0a879u, 0x0a79cu, 0x0a6c2u, 0x0a5eau, 0x0a514u, 0x0a440u, \
    0x0a36eu, 0x0a29fu, 0x0a1d1u, 0x0a106u, 0x0a03cu, 0x09f74u, 0x09eafu, 0x09debu, \
    0x09d29u, 0x09c69u, 0x09babu, 0x09aeeu, 0x09a34u, 0x0997bu, 0x098c4u, 0x0980eu, \
    0x0975au, 0x096a8u, 0x095f8u, 0x09549u, 0x0949cu, 0x093f0u, 0x09346u, 0x0929du, \
    0x091f6u, 0x09150u, 0x090acu, 0x09009u, 0x08f68u, 0x08ec8u, 0x08e29u, 0x08d8cu, \
    0x08cf0u, 0x08c56u, 0x08bbcu, 0x08b24u, 0x08a8eu, 0x089f8u, 0x08964u, 0x088d2u, \
    0x08840u, 0x087afu, 0x08720u, 0x08692u, 0x08605u, 0x08579u, 0x084efu, 0x08465u, \
    0x083ddu, 0x08356u, 0x082cfu, 0x0824au, 0x081c6u, 0x08143u, 0x080c1u, 0x08040u \

#define CHEM_FX_LOG2_VALUES \
    0x001709ad583352d6ull, 0x0044d655203f1e64ull, 0x0072424988f847d7ull, 0x009f624dfe13bd58ull, \
    0x00cc33f197770506ull, 0x00f89ca86eb0ea55ull, 0x0124b1a9240426c1ull, 0x0150706c299032efull, \
    0x017bef0080d198caull, 0x01a7128f47ca269bull, 0x01d1d87c3ec9f6edull, 0x01fc7075022dc3afull, \
    0x0226a638cd411fcfull, 0x0250909cf237234cull, 0x027a2d76c4a432dbull, 0x02a37a95ccc39297ull, \
    0x02cc75c3f5c35fa1ull, 0x02f53702d667fdedull, 0x031dbc9c04ea1577ull, 0x0345ea3a657f8934ull, \
    0x036dd85a82420cccull, 0x03958536cd8a4278ull, 0x03bcef04f2fc2030ull, 0x03e413f5f59c5a72ull, \
    0x040af2365000681full, 0x043187ee16a3d5dcull, 0x0457ef1dc16d1d75ull, 0x047e0a648af1faa6ull, \
    0x04a3f416fe61a245ull, 0x04c98e6ff0117e1dull, 0x04eef41868f856fbull, 0x051423aaca6a8d90ull, \
    0x05391bbdcb5f7fdbull, 0x055dbdc4a55d2605ull, 0x05824260877ea3c9ull, 0x05a68b2bf4554399ull, \
    0x05ca790568938346ull, 0x05ee637190365f3cull, 0x0611eff3cae6d94dull, 0x063558eaaa2fab9bull, \
    0x06587ef9f40e32e8ull, 0x067b7f2c3853ed6bull, 0x069e39c312719a71ull, 0x06c0cc1fb5910e67ull, \
    0x06e31621ddec30c7ull, 0x070554cb6ff6107dull, 0x072748ad0479d612ull, 0x07490fd5d45902d3ull, \
    0x076a89628fb1fc85ull, 0x078bf3bc482d90b7ull, 0x07ad2e29099e644bull, 0x07ce3792ac463a74ull, \
    0x07ef0ee0bce160c0ull, 0x080fb2f88b3ffd9dull, 0x083022bd39a87175ull, 0x08507e274da9cb83ull, \
    0x08708214c3eaea1dull, 0x08906fbfb015533full, 0x08b0468d5e069fafull, 0x08cfe4110b685f32ull, \
    0x08ef4721a605e894ull, 0x090e90c0c4ecbd7full, 0x092d9df179ecea35ull, 0x094c900e03a86eb9ull, \
    0x096b66708fba146full, 0x0989fd8c6363326aull, 0x09a87741147dfbd5ull, 0x09c6d2e3be56487dull, \
    0x09e4ec581b8a9cdfull, 0x0a02e603729babbaull, 0x0a20bf360ef3d653ull, 0x0a3e773ebaa4b8acull, \
    0x0a5c0d6ac3849862ull, 0x0a795caf6f8b7ed9ull, 0x0a96acd60412d321ull, 0x0ab3b44c4e36210eull, \
    0x0ad0bb915e0b5617ull, 0x0aed9d66d58e0b7eull, 0x0b0a33d433e94cbdull, 0x0b26c869a2e4c532ull, \
    0x0b43355a4a96e141ull, 0x0b5f79e73bf62ebbull, 0x0b7b95505114b09full, 0x0b97acf85bbb7baaull, \
    0x0bb3740298efe19aull, 0x0bcf3621dfdfa53full, 0x0beacc6d2e4120eeull, 0x0c065cfb5b75fa94ull, \
    0x0c21c084e13b7867ull, 0x0c3cf6418ecd5957ull, 0x0c57fd683c3caf04ull, 0x0c72fcc42a333489ull, \
    0x0c8dcc50f556aa43ull, 0x0ca893341d425ddbull, 0x0cc3290afbea498dull, 0x0cddb555725b8bb3ull, \
    0x0cf80f5297ffc909ull, 0x0d125edcc87f98b2ull, 0x0d2c7ad4e55fedd9ull, 0x0d468b6fd45b1310ull, \
    0x0d6067305aa7abd9ull, 0x0d7a36a5ed76f799ull, 0x0d93f9868fc99fd4ull, 0x0dad85c7f5c48e6dull, \
    0x0dc7048198bb61ebull, 0x0de04b4b391265d0ull, 0x0df9ade0f3545859ull, 0x0e12d78f049181afull, \
    0x0e2bc77c0c3262c7ull, 0x0e44d277034f9b23ull, 0x0e5da2b4b7ac3beeull, 0x0e763759afc2ad01ull, \
    0x0e8ee647894157a0ull, 0x0ea784294492ae54ull, 0x0ebfe4f049faa5e2ull, 0x0ed833a7ceaa2ab7ull, \
    0x0ef06ffb4b030294ull, 0x0f08999594b7505full, 0x0f2083acc6458617ull, 0x0f3886a450bbc2feull, \
    0x0f50490ee2859847ull, 0x0f67f708d3673ae5ull, 0x0f7fbd666a03ba48ull, 0x0f9741a3907c3804ull, \
    0x0faeb0654925d4b7ull, 0x0fc609517967cbcfull, 0x0fdd4c0d751c4c37ull, 0x0ff4783e007ac54eull \

namespace chem {
namespace fx {
// 2^x = 1 + sum a_k x^k, a_k = ln(2)^k / k!, with x = u 2^-8, u in [0, 1):
// a_1, a_2 2^-8k scaled by 2^72 and 2^80, a_3 .. a_5 by 2^60
constexpr unsigned long long kE1 = 0xb17217f7d1cf79acull;
constexpr unsigned long long kE2 = 0x3d7f7bff058b1d51ull;
constexpr unsigned int kE3 = 0xe35846b8u;
constexpr unsigned int kE4 = 0x00276557u;
constexpr unsigned int kE5 = 0x00000576u;
// log2(1 + r) = sum b_k rho^k, r = rho 2^-8: b_k = (-1)^(k+1) 2^-8k / (k ln 2), times 2^70
constexpr long long kL1 = 6653256548922161246ll;
constexpr long long kL2 = -12994641697113596ll;
constexpr long long kL3 = 33840212752900ll;
constexpr long long kL4 = -99141248300ll;
constexpr long long kL5 = 309816401ll;
constexpr long long kL6 = -1008517ll;
constexpr long long kL7 = 3377ll;
// log2(e) times 2^63 and ln 2 as a double
constexpr unsigned long long kLog2e = 0xb8aa3b295c17f0bcull;
constexpr double kLn2 = 0x1.62e42fefa39efp-1;
}  // namespace fx
}  // namespace chem
