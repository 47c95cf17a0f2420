// Generated by gen_fixed_tables.py; do not edit.
#pragma once
// 2^(j / 256) times 2^63, j = 0 .. 255
#define CHEM_FX_EXP2_VALUES \
    0x8000000000000000ull, 0x8058d7d2d5e5f6b1ull, 0x80b1ed4fd999ab6cull, 0x810b40a1d81406d4ull, \
    0x8164d1f3bc030773ull, 0x81bea1708dde6056ull, 0x8218af4373fc25ecull, 0x8272fb97b2a5894cull, \
    0x82cd8698ac2ba1d7ull, 0x83285071e0fc4547ull, 0x8383594eefb6ee37ull, 0x83dea15b9541b132ull, \
    0x843a28c3acde4046ull, 0x8495efb3303efd30ull, 0x84f1f656379c1a29ull, 0x854e3cd8f9c8c95dull, \
    0x85aac367cc487b15ull, 0x86078a2f23642a9full, 0x8664915b923fba04ull, 0x86c1d919caef5c88ull, \
    0x871f61969e8d1010ull, 0x877d2afefd4e256cull, 0x87db357ff698d792ull, 0x88398146b919f1d4ull, \
    0x88980e8092da8527ull, 0x88f6dd5af155ac6bull, 0x8955ee03618e5fddull, 0x89b540a7902557a4ull, \
    0x8a14d575496efd9aull, 0x8a74ac9a79896e47ull, 0x8ad4c6452c728924ull, 0x8b3522a38e1e1032ull, \
    0x8b95c1e3ea8bd6e7ull, 0x8bf6a434adde0085ull, 0x8c57c9c4646f4ddeull, 0x8cb932c1bae97a95ull, \
    0x8d1adf5b7e5ba9e6ull, 0x8d7ccfc09c50e2f8ull, 0x8ddf042022e69cd6ull, 0x8e417ca940e35a01ull, \
    0x8ea4398b45cd53c0ull, 0x8f073af5a2013520ull, 0x8f6a8117e6c8e5c4ull, 0x8fce0c21c6726481ull, \
    0x9031dc431466b1dcull, 0x9095f1abc540ca6bull, 0x90fa4c8beee4b12bull, 0x915eed13c89689d3ull, \
    0x91c3d373ab11c336ull, 0x9228ffdc10a051adull, 0x928e727d9531f9acull, 0x92f42b88f673aa7cull, \
    0x935a2b2f13e6e92cull, 0x93c071a0eef94bc1ull, 0x9426ff0fab1c04b6ull, 0x948dd3ac8ddb7ed3ull, \
    0x94f4efa8fef70961ull, 0x955c5336887894d5ull, 0x95c3fe86d6cc7fefull, 0x962bf1cbb8d97560ull, \
    0x96942d3720185a00ull, 0x96fcb0fb20ac4ba3ull, 0x97657d49f17ab08eull, 0x97ce9255ec4357abull, \
    0x9837f0518db8a96full, 0x98a1976f7597e996ull, 0x990b87e266c189aaull, 0x9975c1dd47518c77ull, \
    0x99e0459320b7fa65ull, 0x9a4b13371fd166caull, 0x9ab62afc94ff864aull, 0x9b218d16f441d63dull, \
    0x9b8d39b9d54e5539ull, 0x9bf93118f3aa4cc1ull, 0x9c6573682ec32c2dull, 0x9cd200db8a0774cbull, \
    0x9d3ed9a72cffb751ull, 0x9dabfdff6367a2aaull, 0x9e196e189d472420ull, 0x9e872a276f0b98ffull, \
    0x9ef5326091a111aeull, 0x9f6386f8e28ba651ull, 0x9fd228256400dd06ull, 0xa041161b3d0121beull, \
    0xa0b0510fb9714fc2ull, 0xa11fd9384a344cf7ull, 0xa18faeca8544b6e4ull, 0xa1ffd1fc25cea188ull, \
    0xa27043030c496819ull, 0xa2e102153e918f9eull, 0xa3520f68e802bb93ull, 0xa3c36b345991b47cull, \
    0xa43515ae09e6809eull, 0xa4a70f0c95768ec5ull, 0xa5195786be9ef339ull, 0xa58bef536dbeb6eeull, \
    0xa5fed6a9b15138eaull, 0xa6720dc0be08a20cull, 0xa6e594cfeee86b1eull, 0xa7596c0ec55ff55bull, \
    0xa7cd93b4e965356aull, 0xa8420bfa298f70d1ull, 0xa8b6d5167b320e09ull, 0xa92bef41fa77771bull, \
    0xa9a15ab4ea7c0ef8ull, 0xaa1717a7b5693979ull, 0xaa8d2652ec907629ull, 0xab0386ef48868de1ull, \
    0xab7a39b5a93ed337ull, 0xabf13edf162675e9ull, 0xac6896a4be3fe929ull, 0xace0413ff83e5d04ull, \
    0xad583eea42a14ac6ull, 0xadd08fdd43d01491ull, 0xae493452ca35b80eull, 0xaec22c84cc5c9465ull, \
    0xaf3b78ad690a4375ull, 0xafb51906e75b8661ull, 0xb02f0dcbb6e04584ull, 0xb0a957366fb7a3c9ull, \
    0xb123f581d2ac2590ull, 0xb19ee8e8c94feb09ull, 0xb21a31a66618fe3bull, 0xb295cff5e47db4a4ull, \
    0xb311c412a9112489ull, 0xb38e0e38419fae18ull, 0xb40aaea2654b9841ull, 0xb487a58cf4a9c180ull, \
    0xb504f333f9de6484ull, 0xb58297d3a8b9f0d2ull, 0xb60093a85ed5f76cull, 0xb67ee6eea3b22b8full, \
    0xb6fd91e328d17791ull, 0xb77c94c2c9d725e9ull, 0xb7fbefca8ca41e7cull, 0xb87ba337a1743834ull, \
    0xb8fbaf4762fb9ee9ull, 0xb97c143756844dbfull, 0xb9fcd2452c0b9debull, 0xba7de9aebe5fea09ull, \
    0xbaff5ab2133e45fbull, 0xbb81258d5b704b6full, 0xbc034a7ef2e9fb0dull, 0xbc85c9c560e7b269ull, \
    0xbd08a39f580c36bfull, 0xbd8bd84bb67ed483ull, 0xbe0f6809860993e2ull, 0xbe935317fc378238ull, \
    0xbf1799b67a731083ull, 0xbf9c3c248e2486f8ull, 0xc0213aa1f0d08db0ull, 0xc0a6956e8836ca8dull, \
    0xc12c4cca66709456ull, 0xc1b260f5ca0fbb33ull, 0xc238d2311e3d6673ull, 0xc2bfa0bcfad907c9ull, \
    0xc346ccda24976407ull, 0xc3ce56c98d21b15dull, 0xc4563ecc5334cb33ull, 0xc4de8523c2c07baaull, \
    0xc5672a115506daddull, 0xc5f02dd6b0bbc3d9ull, 0xc67990b5aa245f79ull, 0xc70352f04336c51eull, \
    0xc78d74c8abb9b15dull, 0xc817f681416452b2ull, 0xc8a2d85c8ffe2c45ull, 0xc92e1a9d517f0eccull, \
    0xc9b9bd866e2f27a3ull, 0xca45c15afcc72624ull, 0xcad2265e4290774eull, 0xcb5eecd3b38597c9ull, \
    0xcbec14fef2727c5dull, 0xcc799f23d11510e5ull, 0xcd078b86503dcdd2ull, 0xcd95da6a9ff06445ull, \
    0xce248c151f8480e4ull, 0xceb3a0ca5dc6a55dull, 0xcf4318cf191918c1ull, 0xcfd2f4683f94eeb5ull, \
    0xd06333daef2b2595ull, 0xd0f3d76c75c5db8dull, 0xd184df6251699ac6ull, 0xd2164c023056bcabull, \
    0xd2a81d91f12ae45aull, 0xd33a5457a3029054ull, 0xd3ccf099859ac379ull, 0xd45ff29e0972c561ull, \
    0xd4f35aabcfedfa1full, 0xd5872909ab75d18aull, 0xd61b5dfe9f9bce07ull, 0xd6aff9d1e13ba2feull, \
    0xd744fccad69d6af4ull, 0xd7da67311797f56aull, 0xd870394c6db32c84ull, 0xd9067364d44a929cull, \
    0xd99d15c278afd7b6ull, 0xda3420adba4d8704ull, 0xdacb946f2ac9cc72ull, 0xdb63714f8e295255ull, \
    0xdbfbb797daf23755ull, 0xdc9467913a4f1c92ull, 0xdd2d818508324c20ull, 0xddc705bcd378f7f0ull, \
    0xde60f4825e0e9124ull, 0xdefb4e1f9d1037f2ull, 0xdf9612deb8f04420ull, 0xe031430a0d99e627ull, \
    0xe0ccdeec2a94e111ull, 0xe168e6cfd3295d23ull, 0xe2055afffe83d369ull, 0xe2a23bc7d7d91226ull, \
    0xe33f8972be8a5a51ull, 0xe3dd444c46499619ull, 0xe47b6ca0373da88dull, 0xe51a02ba8e26d681ull, \
    0xe5b906e77c8348a8ull, 0xe658797368b3a717ull, 0xe6f85aaaee1fce22ull, 0xe798aadadd5b9cbfull, \
    0xe8396a503c4bdc68ull, 0xe8da9958464b42abull, 0xe97c38406c4f8c57ull, 0xea1e4756550eb27bull, \
    0xeac0c6e7dd24392full, 0xeb63b74317369840ull, 0xec0718b64c1cbddcull, 0xecaaeb8ffb03ab41ull, \
    0xed4f301ed9942b84ull, 0xedf3e6b1d418a491ull, 0xee990f980da3025bull, 0xef3eab20e032bc6bull, \
    0xefe4b99bdcdaf5cbull, 0xf08b3b58cbe8b76aull, 0xf13230a7ad094509ull, 0xf1d999d8b7708cc1ull, \
    0xf281773c59ffb13aull, 0xf329c9233b6bae9cull, 0xf3d28fde3a641a5bull, 0xf47bcbbe6db9fddfull, \
    0xf5257d152486cc2cull, 0xf5cfa433e6537290ull, 0xf67a416c733f846eull, 0xf7255510c4288239ull, \
    0xf7d0df730ad13bb9ull, 0xf87ce0e5b2094d9cull, 0xf92959bb5dd4ba74ull, 0xf9d64a46eb939f35ull, \
    0xfa83b2db722a033aull, 0xfb3193cc4227c3f4ull, 0xfbdfed6ce5f09c49ull, 0xfc8ec01121e447bbull, \
    0xfd3e0c0cf486c175ull, 0xfdedd1b496a89f35ull, 0xfe9e115c7b8f884cull, 0xff4ecb59511ec8a5ull \

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
