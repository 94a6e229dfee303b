// flb_normal64.cuh -- standard normals of the FP64 paths (Box-Muller) in 64-bit
// integer arithmetic.
//
// The FP64 pipe of the part issues one warp instruction of an SM in 16 cycles;
// log, sqrt and sincospi cost a pair of normals about 75 of them, two thirds of
// an FP64 step.  Integer multiplies run beside it at 32 times the rate, and 64
// fixed-point bits leave room below the 53 of the result: the largest error
// over both normals is 1.1e-16 of their radius (root mean square 3.4e-17;
// correctly rounded logarithm, root, cosine and product: 5.7e-17).  Measured
// per step: D2Q9 32 x 32 27.4 -> 15.1 us, D3Q19 64^3 force model 840 -> 450 us.
//
// Table-driven reduction and short series (P.T.P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic",
// ACM TOMS 16, 1990, and its sine counterpart):
//   u0 = (2a + 1) 2^-33 = m 2^-k, m in [1, 2); c_j <= 1 / (upper end of the
//   interval j = the leading 8 fraction bits of m) with 16 bits, so that
//   x = 1 - m c_j in (0, 2^-7.9) is exact, and
//   -ln u0 = k ln 2 + ln c_j - ln(1 - x), the series x + x^2/2 + .. + x^8/8;
//   the last interval has c_j = 1/2, where the first two terms cancel for u0
//   near 1 and x carries the whole precision.
//   r = sqrt(-2 ln u0): a single-precision estimate y of 1 / sqrt(M) and
//   sqrt(M) = M y (1 + e/2 + 3 e^2/8), e = 1 - M y^2 below 2^-20.
//   2 pi u1, u1 = (2b + 1) 2^-33: quadrant, table angle j pi / 512 and a rest
//   below 2^-7.3 by the Taylor series, joined by the addition theorems.
#pragma once

#include <cstdint>

namespace flb {

// ln(1 / c_j) 2^96 (t: the upper 64 bits of the fraction, lo: the rest) and c_j 2^16
struct LogEntry {
    unsigned long long t;
    uint32_t lo, c;
};
__device__ const LogEntry kLogTable[256] = {
    {0x010080559588b357ull, 0xe598e33eu, 65280u}, {0x01fefca72b18c809ull, 0x0b013c4cu, 65027u}, {0x02fc70ec59418e5full, 0x252316adu, 64776u}, {0x03f8d9166a88a2c6ull, 0x1f2e61a8u, 64527u},
    {0x04f43110f5c96a07ull, 0x2797b775u, 64280u}, {0x05ee74c1f98e4729ull, 0x0763bcf8u, 64035u}, {0x06e8a70a2d4d052aull, 0xd2cfb30du, 63791u}, {0x07e0b6c39e8cc018ull, 0x93949a47u, 63550u},
    {0x08d8aec49a6ec157ull, 0xbd5fd858u, 63310u}, {0x09cf83dd075eb129ull, 0xd642e577u, 63072u}, {0x0ac531d7e47a6a46ull, 0x4a9cfef9u, 62836u}, {0x0bbac07b44368ea0ull, 0x36f4e5dbu, 62601u},
    {0x0caf2187c6722ee9ull, 0x844bc592u, 62368u}, {0x0da250b8f07b1a17ull, 0x9abf73bbu, 62137u}, {0x0e9449c5984db986ull, 0x0e5e2e10u, 61908u}, {0x0f86186088b1a886ull, 0x53ba4140u, 61680u},
    {0x1075993598e4f130ull, 0x1b9fbbceu, 61455u}, {0x1165faeeee830734ull, 0x8daf2a4bu, 61230u}, {0x1254062f0a9416feull, 0x50bf3c56u, 61008u}, {0x1341db961bd9d092ull, 0xaed8cba6u, 60787u},
    {0x142f79bed66b83eaull, 0xb00235aeu, 60567u}, {0x151bc93f4f9a648cull, 0x3f5485e5u, 60349u}, {0x1606c5a94e854a48ull, 0x1d5994c9u, 60133u}, {0x16f1828b21eb6756ull, 0x9d90ac75u, 59918u},
    {0x17dae56d93235379ull, 0x0bc3e274u, 59705u}, {0x18c403d6781d43d8ull, 0xbd74e547u, 59493u}, {0x19abc1463fb43747ull, 0x1af97e2fu, 59283u}, {0x1a93353a98f58c15ull, 0xce54682eu, 59074u},
    {0x1b79412bcd862a0aull, 0xff4d857cu, 58867u}, {0x1c5efe8f94395c13ull, 0x0534b38du, 58661u}, {0x1d434cd6730bde4full, 0x669e9916u, 58457u}, {0x1e27476e32f2e73full, 0x401d5544u, 58254u},
    {0x1f0aecc0566ac82dull, 0x7a117749u, 58052u}, {0x1fed1932000ac775ull, 0x88bff579u, 57852u}, {0x20ceeb25dd7380e5ull, 0x0694356fu, 57653u}, {0x21af3cf9a91cb422ull, 0x847849e4u, 57456u},
    {0x228f2f08d10d590eull, 0x04105a15u, 57260u}, {0x236ebfaa74c14660ull, 0xdb3fc084u, 57065u}, {0x244ded32a4267c35ull, 0xae9405dbu, 56871u}, {0x252b8df0a90a861bull, 0x8c399aa6u, 56679u},
    {0x2608c632622015a4ull, 0xd9b3ee4eu, 56488u}, {0x26e46a405680f000ull, 0xb5b1d526u, 56299u}, {0x27bfa061daf8d3aeull, 0xd25e679cu, 56111u}, {0x289a66d9977a3cd4ull, 0xfd083746u, 55924u},
    {0x2974bbe7408dcd1eull, 0x349b19c2u, 55738u}, {0x2a4e9dc7998a9e60ull, 0x7cfe9d50u, 55553u}, {0x2b26dbb3463311b5ull, 0x5aac448du, 55370u}, {0x2bfea0e15727a8e6ull, 0x3d596970u, 55188u},
    {0x2cd5eb84f22b2471ull, 0xbb6afd7fu, 55007u}, {0x2dacb9ce61f64baeull, 0x3ea3a43bu, 54827u}, {0x2e8309eb198fb93bull, 0x17eb5ed9u, 54648u}, {0x2f57a6044c7a22b4ull, 0xe351efb8u, 54471u},
    {0x302bbe428df456d4ull, 0x936a09ccu, 54295u}, {0x30ff50ca42122125ull, 0x95679851u, 54120u}, {0x31d25bbd110c8155ull, 0xfe92d1eeu, 53946u}, {0x32a4dd39ebcd693full, 0xd7c003c8u, 53773u},
    {0x3376d35d10af8c3aull, 0x831ba6dau, 53601u}, {0x34483c401072ec7eull, 0x99767403u, 53430u}, {0x3517daf9105eb185ull, 0xcf770f25u, 53261u}, {0x35e8229d29fff4e1ull, 0xa3287552u, 53092u},
    {0x36b7d73dd8b3dd7aull, 0x04c330ccu, 52924u}, {0x3785b8e894e1c635ull, 0x95fd1ab4u, 52758u}, {0x385301ab1ce201dfull, 0x40f98de9u, 52593u}, {0x3920ef8fb53498adull, 0xe105c66fu, 52428u},
    {0x39ed019c40144a14ull, 0xd7187873u, 52265u}, {0x3ab874d6a4592359ull, 0xe4dd4e25u, 52103u}, {0x3b848a41e969e23eull, 0xb3ee15f3u, 51941u}, {0x3c4ebadc8fade5b5ull, 0x7770085cu, 51781u},
    {0x3d1846a55d36c148ull, 0x97d3ee93u, 51622u}, {0x3de271984fa4d9ebull, 0xbd681d2fu, 51463u}, {0x3eaaaeacc54880a1ull, 0xc56dea23u, 51306u}, {0x3f7240dabcfc551full, 0xffe26dc5u, 51150u},
    {0x403a6f16fbc295fdull, 0x460c3b29u, 50994u}, {0x4100a652d3c10370ull, 0xdf44d82du, 50840u}, {0x41c7777f6156459eull, 0xebab1a3du, 50686u}, {0x428d978a524be6e3ull, 0x7ea1a2a0u, 50533u},
    {0x4351b75e6b0f2c83ull, 0x439640ffu, 50382u}, {0x44166de6c0ad5598ull, 0xd165b5ecu, 50231u}, {0x44da6d0a5b73442full, 0x61cdc4d7u, 50081u}, {0x459db2aeb6983963ull, 0xc8b4ab26u, 49932u},
    {0x46603cb750adbd9dull, 0xe7c5bcf8u, 49784u}, {0x47235b061e883983ull, 0xfd42af5bu, 49636u}, {0x47e46879387dd044ull, 0xd13d4df4u, 49490u}, {0x48a607efbde5ebdeull, 0x9f6a7f26u, 49344u},
    {0x496590437e58e7c1ull, 0x77a43938u, 49200u}, {0x4a25a84f821a8ed0ull, 0x27e16952u, 49056u}, {0x4ae4f9eae8cd1367ull, 0xb7c86c4du, 48913u}, {0x4ba4daec60f58361ull, 0x71117180u, 48770u},
    {0x4c629a25a7fac3b2ull, 0xb1124c4au, 48629u}, {0x4d1f8c6a62e75366ull, 0xf2f379d1u, 48489u}, {0x4ddd0a8b1851f320ull, 0x1bc4f554u, 48349u}, {0x4e99b955c937b3e8ull, 0x17459150u, 48210u},
    {0x4f55969716fc4194ull, 0x2fddaf78u, 48072u}, {0x5011fe1adda82f73ull, 0x5a351023u, 47934u}, {0x50cc32a82ed25731ull, 0xcd21d67du, 47798u}, {0x5186ef08b97b2df4ull, 0x422ceaf3u, 47662u},
    {0x5240d30142ffe364ull, 0x6104fe4eu, 47527u}, {0x52f9dc55ef2487a6ull, 0xb0e4528du, 47393u}, {0x53b36bca0f7a8bf8ull, 0x6236e258u, 47259u}, {0x546aba1cb7e8b427ull, 0x3a4ad8d4u, 47127u},
    {0x55228c0eb74a0b3full, 0x31d963d1u, 46995u}, {0x55dae25d9b7c0cccull, 0x4e67904du, 46863u}, {0x5690efc3dc8c081dull, 0x029e9905u, 46733u}, {0x57477efd8447360dull, 0x90a69948u, 46603u},
    {0x57fd27c2b2a15487ull, 0x992512e4u, 46474u}, {0x58b351cbb6b104f6ull, 0x58754ffdu, 46345u}, {0x596727cc1ca9ccd5ull, 0x5a2db1c4u, 46218u}, {0x5a1b7c7a7cdabf06ull, 0xf6b4338du, 46091u},
    {0x5ad05089cdd9dba1ull, 0xd4969f98u, 45964u}, {0x5b82c8a8d5e99cc0ull, 0x91b0bce6u, 45839u}, {0x5c35bd8a202af406ull, 0x160a4a6fu, 45714u}, {0x5ce7bfdb01401ef3ull, 0x8a75504du, 45590u},
    {0x5d9a3e496d81967eull, 0x78a14068u, 45466u}, {0x5e4bc7802c011bacull, 0xf20fbc5du, 45343u}, {0x5efc5929419fb868ull, 0x2d6529b9u, 45221u}, {0x5fabf0ee0b3f0d98ull, 0x23ed3428u, 45100u},
    {0x605c01768802d770ull, 0x0ca14e52u, 44979u}, {0x610c8b6947350a24ull, 0x50880e08u, 44858u}, {0x61baa168dc5b03fdull, 0x2abdcd33u, 44739u}, {0x62692e1b17096f56ull, 0x9da604a2u, 44620u},
    {0x6318322243477046ull, 0xf27d05e0u, 44501u}, {0x63c4ba1ce18b1f4dull, 0xb33cab08u, 44384u}, {0x6471b6ad17a9762eull, 0xf6fd98a8u, 44267u}, {0x651f2870df7c1e2bull, 0x53e42bd9u, 44150u},
    {0x65cb9304d357bd1full, 0xa4298ccdu, 44034u}, {0x6676f40490443f3eull, 0x80afb363u, 43919u}, {0x6722c80c0da9fef0ull, 0xccafaf16u, 43804u}, {0x67cd8fb37e618520ull, 0x6f8b6246u, 43690u},
    {0x6877489360bed762ull, 0x1a923392u, 43577u}, {0x69217243af6c2fd5ull, 0x4a487262u, 43464u}, {0x69cc0d5ac7f53d41ull, 0x2776d08du, 43351u}, {0x6a74126a7a212ab5ull, 0x2283d51eu, 43240u},
    {0x6b1c860965281068ull, 0x002b42adu, 43129u}, {0x6bc568c968e9d290ull, 0xf9643b65u, 43018u}, {0x6c6d343b3cf98f70ull, 0x44de0e7du, 42908u}, {0x6d13e5ef325d8a33ull, 0xa6615a51u, 42799u},
    {0x6dbb0474f7ef76f3ull, 0xe19996b5u, 42690u}, {0x6e62905afe66797eull, 0xcd63aa4du, 42581u}, {0x6f08ff2d5239c258ull, 0x99701dc5u, 42473u}, {0x6fae4e77358e5f85ull, 0xc961c829u, 42366u},
    {0x705408c5856a4f6full, 0x19be5471u, 42259u}, {0x70f8a0a00137df9full, 0x1c8c8e76u, 42153u}, {0x719c139005bfe0f4ull, 0xb078bf34u, 42048u}, {0x723fef1e6ae886b5ull, 0xecb61121u, 41943u},
    {0x72e433d173cd44a5ull, 0x380e0821u, 41838u}, {0x7387502e4297be6bull, 0x112abf98u, 41734u}, {0x742ad4ba980c40ceull, 0x01694ec7u, 41630u}, {0x74cd2df8bcf7ea24ull, 0x6be77fadu, 41527u},
    {0x756e596b9b469301ull, 0x581b2b06u, 41425u}, {0x760fea96349efbabull, 0x2dfbbf59u, 41323u}, {0x76b1e1f93eba338dull, 0xb956ddf7u, 41221u}, {0x7752a8138712d851ull, 0x2df01afdu, 41120u},
    {0x77f23a641dded53eull, 0xa14007d7u, 41020u}, {0x78923069f2309878ull, 0x4b92ababu, 40920u}, {0x79328aa1ece436ffull, 0x67e50408u, 40820u}, {0x79d1ad878ea635fdull, 0x6bfff564u, 40721u},
    {0x7a713397363a8c5bull, 0x63b47fc0u, 40622u}, {0x7b0f7f49b3537005ull, 0x24a63947u, 40524u}, {0x7bac8e1903b450d7ull, 0xd739773fu, 40427u}, {0x7c4b9d7fae1c90a3ull, 0xac291547u, 40329u},
    {0x7ce7cdf20a61f00cull, 0xa43c7fabu, 40233u}, {0x7d85ffeac923af00ull, 0xd1a517ceu, 40136u}, {0x7e214ddbfd2788f3ull, 0x7f416b9bu, 40041u}, {0x7ebe9e3ea6d51be5ull, 0xe8baabfau, 39945u},
    {0x7f5aaa84ddf8c088ull, 0x9b0ed5e4u, 39850u}, {0x7ff57021a1f28105ull, 0xc5aabc5au, 39756u}, {0x80909389767e73a3ull, 0x97aabf04u, 39662u}, {0x812c152e4e891636ull, 0x274c70c6u, 39568u},
    {0x81c64c7f56372390ull, 0x18ec4410u, 39475u}, {0x825f36ed4fc8942dull, 0xf38884fau, 39383u}, {0x82fa27ea553004dcull, 0x245d7ef7u, 39290u}, {0x83921ee0eac202e1ull, 0xa76abb75u, 39199u},
    {0x842c1d4319818ed8ull, 0xb7a8d811u, 39107u}, {0x84c4ca7b9629c6b9ull, 0xbcc1af66u, 39016u}, {0x855c23f6884894c7ull, 0xa845d99bu, 38926u}, {0x85f3d7213154170aull, 0x1a532f01u, 38836u},
    {0x868be4661b47e67full, 0x82123d12u, 38746u}, {0x87229a2e9a466221ull, 0x3fbc285bu, 38657u}, {0x87b9a8e4fe6bf740ull, 0x62f5cf36u, 38568u}, {0x885110f278adbdc5ull, 0xfcc21858u, 38479u},
    {0x88e71dbd2c4d1a3aull, 0xfa5c8b5eu, 38391u}, {0x897bccaca77de3edull, 0x5eae23a1u, 38304u}, {0x8a12892a4e0b59f6ull, 0xc6fe3246u, 38216u}, {0x8aa62e97a72f4d51ull, 0xcef2b208u, 38130u},
    {0x8b3be25dda35427bull, 0x6fa19637u, 38043u}, {0x8bd033df250f3da4ull, 0x7ca52724u, 37957u}, {0x8c64db80afd5a3a8ull, 0x080cb09eu, 37871u}, {0x8cf81da3a76bb5e6ull, 0x666f7463u, 37786u},
    {0x8d8bb4ac7c85dcbaull, 0x7b5a3afbu, 37701u}, {0x8e1de2fb8c232617ull, 0xd521d558u, 37617u}, {0x8eb223f487097bf8ull, 0xb813dadbu, 37532u}, {0x8f433af38a068344ull, 0xb8628501u, 37449u},
    {0x8fd6655d0e4798d4ull, 0xb81812edu, 37365u}, {0x9068228d58640d19ull, 0xabd393feu, 37282u}, {0x90f86fe32e775f14ull, 0x2dcf4c91u, 37200u}, {0x918ad2becd42ce38ull, 0x9169a3d6u, 37117u},
    {0x921bc47b40530e5bull, 0x47a32123u, 37035u}, {0x92ab4274db465ef6ull, 0x38a9a495u, 36954u}, {0x933b1109a1877e69ull, 0x56fdd38fu, 36873u}, {0x93cb30945588d8b1ull, 0x178f432du, 36792u},
    {0x945ba170535d103dull, 0x9c3c0f01u, 36711u}, {0x94ea99f672568af4ull, 0xeb08bb0bu, 36631u}, {0x9579e281ea1a7c11ull, 0x15d5e04du, 36551u}, {0x9607af6a3674624bull, 0xd6258e33u, 36472u},
    {0x9695cb097a816dc5ull, 0x5a092ca0u, 36393u}, {0x972435b74adb527full, 0xbd87c975u, 36314u}, {0x97b2efcbce98128dull, 0x329b179bu, 36235u}, {0x9840299b8106ee79ull, 0x6879349eu, 36157u},
    {0x98cbe07d407350f0ull, 0x6f9d720eu, 36080u}, {0x9959b5c92e73fe12ull, 0x7650ccccu, 36002u}, {0x99e606d205bd6d72ull, 0xf9e6dd42u, 35925u}, {0x9a72a4edd90f768dull, 0x96b11529u, 35848u},
    {0x9afdbb6ec63d108full, 0x99c2157au, 35772u}, {0x9b891daa4c3db2aeull, 0xe9564288u, 35696u}, {0x9c14cbf30ed41c49ull, 0x73ac4dc0u, 35620u}, {0x9ca0c69c395296a5ull, 0xcfab9f6bu, 35544u},
    {0x9d2b34f50e7d614bull, 0x6adbaf78u, 35469u}, {0x9db5ee519d2b0492ull, 0xa78084dfu, 35394u}, {0x9e3f180014b06183ull, 0x9f9469bfu, 35320u}, {0x9ec88b53a6d7ddeaull, 0x2448ed7fu, 35246u},
    {0x9f52489b9342f600ull, 0x7032f471u, 35172u}, {0x9fdc502799c318b1ull, 0x5247c2e2u, 35098u}, {0xa064c34478581047ull, 0x14c7e59eu, 35025u}, {0xa0ed7f42b395c878ull, 0xbb3ba02cu, 34952u},
    {0xa17684704fa7ea37ull, 0x8b5c691bu, 34879u}, {0xa1fdf11840d583e9ull, 0x89a319ddu, 34807u}, {0xa285a589f4cd0249ull, 0xc82f3e03u, 34735u}, {0xa30da211affec0e7ull, 0xc010341eu, 34663u},
    {0xa39401f9af556e0dull, 0x6e341304u, 34592u}, {0xa41aa88f5478fb9full, 0xfc9b389au, 34521u}, {0xa4a1961d20623d50ull, 0x70f0eeb8u, 34450u}, {0xa528caee0a1635a7ull, 0x865c7cefu, 34379u},
    {0xa5ae5e4ad0e8242bull, 0x5ce309d4u, 34309u}, {0xa634377e7d63d39aull, 0x169dd845u, 34239u}, {0xa6ba56d23d9cc5efull, 0x3fab80d6u, 34169u}, {0xa73ed08dbb5d84eaull, 0xda184782u, 34100u},
    {0xa7c57bfbe3aacd66ull, 0xcdabd079u, 34030u}, {0xa84a8061d10793f1ull, 0x00ca6584u, 33961u}, {0xa8cddb06119ed15full, 0x7878bb02u, 33893u}, {0xa9517932dead5779ull, 0x139b0e03u, 33825u},
    {0xa9d74c2f96662605ull, 0xb5b05ca3u, 33756u}, {0xaa59813cdde6c182ull, 0x289384d0u, 33689u}, {0xaaddeba67e2fac8full, 0x2a01fc0bu, 33621u}, {0xab60a6adfabcfd4bull, 0x03809397u, 33554u},
    {0xabe3a49a1df94142ull, 0x36089d95u, 33487u}, {0xac66e5af7fed57e5ull, 0x16bea3e3u, 33420u}, {0xace873300596024dull, 0xcb75d63bu, 33354u}, {0xad6a4261b4f9692eull, 0xa2ea84e3u, 33288u},
    {0xadec53874ed59eeeull, 0x960a5c4eu, 33222u}, {0xae6ea6e3f9db940full, 0x680b1832u, 33156u}, {0xaeef41b8b0f99e3bull, 0xef599968u, 33091u}, {0xaf701d4920d3ab87ull, 0x5af5ad3du, 33026u},
    {0xaff139d6950d45f2ull, 0x87e01808u, 32961u}, {0xb07297a2bc471ba9ull, 0x79a058e3u, 32896u}, {0xb0f237ed2b233611ull, 0xe7457983u, 32832u}, {0xb17217f7d1cf79abull, 0xc9e3b398u, 32768u},
};
// sin and cos of j pi / 512, times 2^63
__device__ const ulonglong2 kSinCosTable[256] = {
    {0x0000000000000000ull, 0x8000000000000000ull}, {0x00c90f87f3380389ull, 0x7fff62163a2a4936ull},
    {0x01921d1fcdec7846ull, 0x7ffd885a6e4b6d5eull}, {0x025b26d77c61dfa7ull, 0x7ffa72d12d4684aeull},
    {0x03242abef46ccfbfull, 0x7ff62182133432edull}, {0x03ed26e63a39e020ull, 0x7ff09477c74fe0bdull},
    {0x04b6195d65157346ull, 0x7fe9cbbffbdd7275ull}, {0x057f0034a43350daull, 0x7fe1c76b6e077cc6ull},
    {0x0647d97c437604faull, 0x7fd8878de5b5f78full}, {0x0710a344b035f8b4ull, 0x7fce0c3e355d6f35ull},
    {0x07d95b9e7e0837fbull, 0x7fc2559639c6b502ull}, {0x08a2009a6b84d940ull, 0x7fb563b2d9cf0f0dull},
    {0x096a9049670cfae6ull, 0x7fa736b40620e855ull}, {0x0a3308bc93904ad7ull, 0x7f97cebcb8e501b2ull},
    {0x0afb68054d520c61ull, 0x7f872bf2f56c2469ull}, {0x0bc3ac352ead90acull, 0x7f754e7fc7d1572aull},
    {0x0c8bd35e14da15f1ull, 0x7f62368f44949678ull}, {0x0d53db9224ae01bdull, 0x7f4de450882e1153ull},
    {0x0e1bc2e3cf616a7bull, 0x7f3857f5b699eb51ull}, {0x0ee38765d74fe489ull, 0x7f2191b3fadc8531ull},
    {0x0fab272b54b9871aull, 0x7f0991c3867f4d1full}, {0x1072a047ba831d23ull, 0x7ef0585f910617eaull},
    {0x1139f0cedaf576abull, 0x7ed5e5c6575d048eull}, {0x120116d4ec7bceb7ull, 0x7eba3a391b3eeb63ull},
    {0x12c8106e8e613a22ull, 0x7e9d55fc22945a86ull}, {0x138edbb0cd8d13baull, 0x7e7f3956b6cb20f9ull},
    {0x145576b1293e59dbull, 0x7e5fe49324266a1dull}, {0x151bdf8597c5f1faull, 0x7e3f57feb9076b3aull},
    {0x15e214448b3fc655ull, 0x7e1d93e9c52ea4d6ull}, {0x16a81304f64ab23eull, 0x7dfa98a798f5b9bbull},
    {0x176dd9de50bf3147ull, 0x7dd6668e8481dd85ull}, {0x183366e89c64c5baull, 0x7db0fdf7d6eedcc3ull},
    {0x18f8b83c69a60ab6ull, 0x7d8a5f3fdd72c0abull}, {0x19bdcbf2dc436666ull, 0x7d628ac5e27a1090ull},
    {0x1a82a025b004509eull, 0x7d3980ec2cbcb339ull}, {0x1b4732ef3d67226full, 0x7d0f4217fe4b7270ull},
    {0x1c0b826a7e4f62fdull, 0x7ce3ceb193962314ull}, {0x1ccf8cb312b28624ull, 0x7cb72724226a7415ull},
    {0x1d934fe54543115dull, 0x7c894bddd8eb66dfull}, {0x1e56ca1e101a1b52ull, 0x7c5a3d4fdc8173b6ull},
    {0x1f19f97b215f1aafull, 0x7c29fbee48c35ca9ull}, {0x1fdcdc1adfedf8b5ull, 0x7bf888302e57b1c8ull},
    {0x209f701c6ffb5bffull, 0x7bc5e28f91cf0963ull}, {0x2161b39fb7b72027ull, 0x7b920b896a76ef25ull},
    {0x2223a4c563eceec1ull, 0x7b5d039da1258cf4ull}, {0x22e541aeeca2ee49ull, 0x7b26cb4f0efe108dull},
    {0x23a6887e99b67ba3ull, 0x7aef63237c2dd0e3ull}, {0x246777578776e2cdull, 0x7ab6cba39ea2366dull},
    {0x25280c5dab3e0b51ull, 0x7a7d055b18b76976ull}, {0x25e845b5d8070d45ull, 0x7a4210d877dfc9ceull},
    {0x26a82185c302a362ull, 0x7a05eead33443318ull}, {0x27679df408296efaull, 0x79c89f6daa5d1121ull},
    {0x2826b9282ecc0286ull, 0x798a23b1238447baull}, {0x28e5714aae20a77full, 0x794a7c11ca7ff190ull},
    {0x29a3c484f1ced449ull, 0x7909a92caf05f9a8ull}, {0x2a61b1015e784703ull, 0x78c7aba1c3389322ull},
    {0x2b1f34eb563fb9fcull, 0x78848413da1b92ffull}, {0x2bdc4e6f3d4d26b2ull, 0x78403328a602afbfull},
    {0x2c98fbba7e4f8c22ull, 0x77fab988b6f8aaafull}, {0x2d553afb8efc2d64ull, 0x77b417df791f66d3ull},
    {0x2e110a61f48b3d5eull, 0x776c4edb3308f184ull}, {0x2ecc681e4831ec96ull, 0x77235f2d040980b6ull},
    {0x2f8752623b99ce03ull, 0x76d94988e2826b29ull}, {0x3041c7609d5587e7ull, 0x768e0ea59a261ea8ull},
    {0x30fbc54d5d52c5a3ull, 0x7641af3cca3518a3ull}, {0x31b54a5d91495fa3ull, 0x75f42c0ae3b3e580ull},
    {0x326e54c77927ae5aull, 0x75a585cf279a2b0cull}, {0x3326e2c2837bfd75ull, 0x7555bd4ba4fac27full},
    {0x33def28751db145bull, 0x7504d3453724e6b1ull}, {0x3496824fbd43c921ull, 0x74b2c88383be7b08ull},
    {0x354d9056da7f9315ull, 0x745f9dd0f8d76fdeull}, {0x36041ad8fe801228ull, 0x740b53facaf64919ull},
    {0x36ba2013c2b98057ull, 0x73b5ebd0f31dcbc3ull}, {0x376f9e46097a0268ull, 0x735f66262ccbd783ull},
    {0x382493b0023dcd3full, 0x7307c3cff3f170f3ull}, {0x38d8fe932e001521ull, 0x72af05a682e401c4ull},
    {0x398cdd326388bc2dull, 0x72552c84d047d3daull}, {0x3a402dd1d3b6b58eull, 0x71fa39488cf3cc6dull},
    {0x3af2eeb70dc712abull, 0x719e2cd221ce6c76ull}, {0x3ba51e290398afe2ull, 0x71410804ada41ba9ull},
    {0x3c56ba700dec763cull, 0x70e2cbc602f6c349ull}, {0x3d07c1d5f0a227a1ull, 0x708378fea5c6be4bull},
    {0x3db832a5def1ab11ull, 0x70231099c9552436ull}, {0x3e680b2c7fa0ce83ull, 0x6fc193854ddf7448ull},
    {0x3f1749b7f13573f7ull, 0x6f5f02b1be54a67eull}, {0x3fc5ec97ce241f6bull, 0x6efb5f124e03a81cull},
    {0x4073f21d30fadb66ull, 0x6e96a99cd643497full}, {0x4121589ab88869b9ull, 0x6e30e349d413a2ebull},
    {0x41ce1e648bffb65aull, 0x6dca0d1465b8f644ull}, {0x427a41d05f178202ull, 0x6d6227fa48501388ull},
    {0x4325c13576263a73ull, 0x6cf934fbd55c4615ull}, {0x43d09aecaa39f645ull, 0x6c8f351c004ed0adull},
    {0x447acd506d2c8a11ull, 0x6c2429605407fe6eull}, {0x452456bccdb3acfaull, 0x6bb812d0f051cec6ull},
    {0x45cd358f7b6d2281ull, 0x6b4af278875442b8ull}, {0x46756827cae6dfb3ull, 0x6adcc9645b0351a9ull},
    {0x471cece6b9a321b2ull, 0x6a6d98a43a868c0dull}, {0x47c3c22ef2186bbcull, 0x69fd614a7f9a7268ull},
    {0x4869e664cfad62c6ull, 0x698c246c0beb870bull}, {0x490f57ee62b07ce3ull, 0x6919e320466b211bull},
    {0x49b41533744b7aa2ull, 0x68a69e81189e0777ull}, {0x4a581c9d8a72a0abull, 0x683257aaebe4da1full},
    {0x4afb6c97ebcfa7ddull, 0x67bd0fbca6be50d9ull}, {0x4b9e038fa3a85a4eull, 0x6746c7d7aa0355c6ull},
    {0x4c3fdff385c0d384ull, 0x66cf811fce1d02cfull}, {0x4ce1003432395a54ull, 0x66573cbb603488bcull},
    {0x4d8162c41967cae0ull, 0x65ddfbd31f5d06ebull}, {0x4e2106177fac8730ull, 0x6563bf9239b75aaaull},
    {0x4ebfe8a48142e4f2ull, 0x64e88926498fed3dull}, {0x4f5e08e3160d0efeull, 0x646c59bf527687b1ull},
    {0x4ffb654d155b5137ull, 0x63ef328fbe5033a5ull}, {0x5097fc5e39aec57bull, 0x637114cc5a633047ull},
    {0x5133cc9424775860ull, 0x62f201ac545d02d4ull}, {0x51ced46e61cd1c73ull, 0x6271fa693752a9dbull},
    {0x5269126e6c24e2d8ull, 0x61f1003ee8bafad2ull}, {0x53028517b0001025ull, 0x616f146ba5633146ull},
    {0x539b2aef8f97a44full, 0x60ec382ffe5db748ull}, {0x5433027d66826cb5ull, 0x60686cced5eb2ea2ull},
    {0x54ca0a4a8d56572full, 0x5fe3b38d5c5dc263ull}, {0x556040e25d44dd45ull, 0x5f5e0db30cf6c88bull},
    {0x55f5a4d233b27e8bull, 0x5ed77c89aabebb78ull}, {0x568a34a975c94158ull, 0x5e50015d3d5792f5ull},
    {0x571deef994063107ull, 0x5dc79d7c0dc984aeull}, {0x57b0d2560dc1d0efull, 0x5d3e5236a34a3401ull},
    {0x5842dd5474b37b6dull, 0x5cb420dfbffe590dull}, {0x58d40e8c706fa445ull, 0x5c290acc5db5e713ull},
    {0x59646497c1e0f5c4ull, 0x5b9d1153aaa2ba24ull}, {0x59f3de1246bc4017ull, 0x5b1035cf0609d449ull},
    {0x5a827999fcef3242ull, 0x5a827999fcef3242ull}, {0x5b1035cf0609d449ull, 0x59f3de1246bc4017ull},
    {0x5b9d1153aaa2ba24ull, 0x59646497c1e0f5c4ull}, {0x5c290acc5db5e713ull, 0x58d40e8c706fa445ull},
    {0x5cb420dfbffe590dull, 0x5842dd5474b37b6dull}, {0x5d3e5236a34a3401ull, 0x57b0d2560dc1d0efull},
    {0x5dc79d7c0dc984aeull, 0x571deef994063107ull}, {0x5e50015d3d5792f5ull, 0x568a34a975c94158ull},
    {0x5ed77c89aabebb78ull, 0x55f5a4d233b27e8bull}, {0x5f5e0db30cf6c88bull, 0x556040e25d44dd45ull},
    {0x5fe3b38d5c5dc263ull, 0x54ca0a4a8d56572full}, {0x60686cced5eb2ea2ull, 0x5433027d66826cb5ull},
    {0x60ec382ffe5db748ull, 0x539b2aef8f97a44full}, {0x616f146ba5633146ull, 0x53028517b0001025ull},
    {0x61f1003ee8bafad2ull, 0x5269126e6c24e2d8ull}, {0x6271fa693752a9dbull, 0x51ced46e61cd1c73ull},
    {0x62f201ac545d02d4ull, 0x5133cc9424775860ull}, {0x637114cc5a633047ull, 0x5097fc5e39aec57bull},
    {0x63ef328fbe5033a5ull, 0x4ffb654d155b5137ull}, {0x646c59bf527687b1ull, 0x4f5e08e3160d0efeull},
    {0x64e88926498fed3dull, 0x4ebfe8a48142e4f2ull}, {0x6563bf9239b75aaaull, 0x4e2106177fac8730ull},
    {0x65ddfbd31f5d06ebull, 0x4d8162c41967cae0ull}, {0x66573cbb603488bcull, 0x4ce1003432395a54ull},
    {0x66cf811fce1d02cfull, 0x4c3fdff385c0d384ull}, {0x6746c7d7aa0355c6ull, 0x4b9e038fa3a85a4eull},
    {0x67bd0fbca6be50d9ull, 0x4afb6c97ebcfa7ddull}, {0x683257aaebe4da1full, 0x4a581c9d8a72a0abull},
    {0x68a69e81189e0777ull, 0x49b41533744b7aa2ull}, {0x6919e320466b211bull, 0x490f57ee62b07ce3ull},
    {0x698c246c0beb870bull, 0x4869e664cfad62c6ull}, {0x69fd614a7f9a7268ull, 0x47c3c22ef2186bbcull},
    {0x6a6d98a43a868c0dull, 0x471cece6b9a321b2ull}, {0x6adcc9645b0351a9ull, 0x46756827cae6dfb3ull},
    {0x6b4af278875442b8ull, 0x45cd358f7b6d2281ull}, {0x6bb812d0f051cec6ull, 0x452456bccdb3acfaull},
    {0x6c2429605407fe6eull, 0x447acd506d2c8a11ull}, {0x6c8f351c004ed0adull, 0x43d09aecaa39f645ull},
    {0x6cf934fbd55c4615ull, 0x4325c13576263a73ull}, {0x6d6227fa48501388ull, 0x427a41d05f178202ull},
    {0x6dca0d1465b8f644ull, 0x41ce1e648bffb65aull}, {0x6e30e349d413a2ebull, 0x4121589ab88869b9ull},
    {0x6e96a99cd643497full, 0x4073f21d30fadb66ull}, {0x6efb5f124e03a81cull, 0x3fc5ec97ce241f6bull},
    {0x6f5f02b1be54a67eull, 0x3f1749b7f13573f7ull}, {0x6fc193854ddf7448ull, 0x3e680b2c7fa0ce83ull},
    {0x70231099c9552436ull, 0x3db832a5def1ab11ull}, {0x708378fea5c6be4bull, 0x3d07c1d5f0a227a1ull},
    {0x70e2cbc602f6c349ull, 0x3c56ba700dec763cull}, {0x71410804ada41ba9ull, 0x3ba51e290398afe2ull},
    {0x719e2cd221ce6c76ull, 0x3af2eeb70dc712abull}, {0x71fa39488cf3cc6dull, 0x3a402dd1d3b6b58eull},
    {0x72552c84d047d3daull, 0x398cdd326388bc2dull}, {0x72af05a682e401c4ull, 0x38d8fe932e001521ull},
    {0x7307c3cff3f170f3ull, 0x382493b0023dcd3full}, {0x735f66262ccbd783ull, 0x376f9e46097a0268ull},
    {0x73b5ebd0f31dcbc3ull, 0x36ba2013c2b98057ull}, {0x740b53facaf64919ull, 0x36041ad8fe801228ull},
    {0x745f9dd0f8d76fdeull, 0x354d9056da7f9315ull}, {0x74b2c88383be7b08ull, 0x3496824fbd43c921ull},
    {0x7504d3453724e6b1ull, 0x33def28751db145bull}, {0x7555bd4ba4fac27full, 0x3326e2c2837bfd75ull},
    {0x75a585cf279a2b0cull, 0x326e54c77927ae5aull}, {0x75f42c0ae3b3e580ull, 0x31b54a5d91495fa3ull},
    {0x7641af3cca3518a3ull, 0x30fbc54d5d52c5a3ull}, {0x768e0ea59a261ea8ull, 0x3041c7609d5587e7ull},
    {0x76d94988e2826b29ull, 0x2f8752623b99ce03ull}, {0x77235f2d040980b6ull, 0x2ecc681e4831ec96ull},
    {0x776c4edb3308f184ull, 0x2e110a61f48b3d5eull}, {0x77b417df791f66d3ull, 0x2d553afb8efc2d64ull},
    {0x77fab988b6f8aaafull, 0x2c98fbba7e4f8c22ull}, {0x78403328a602afbfull, 0x2bdc4e6f3d4d26b2ull},
    {0x78848413da1b92ffull, 0x2b1f34eb563fb9fcull}, {0x78c7aba1c3389322ull, 0x2a61b1015e784703ull},
    {0x7909a92caf05f9a8ull, 0x29a3c484f1ced449ull}, {0x794a7c11ca7ff190ull, 0x28e5714aae20a77full},
    {0x798a23b1238447baull, 0x2826b9282ecc0286ull}, {0x79c89f6daa5d1121ull, 0x27679df408296efaull},
    {0x7a05eead33443318ull, 0x26a82185c302a362ull}, {0x7a4210d877dfc9ceull, 0x25e845b5d8070d45ull},
    {0x7a7d055b18b76976ull, 0x25280c5dab3e0b51ull}, {0x7ab6cba39ea2366dull, 0x246777578776e2cdull},
    {0x7aef63237c2dd0e3ull, 0x23a6887e99b67ba3ull}, {0x7b26cb4f0efe108dull, 0x22e541aeeca2ee49ull},
    {0x7b5d039da1258cf4ull, 0x2223a4c563eceec1ull}, {0x7b920b896a76ef25ull, 0x2161b39fb7b72027ull},
    {0x7bc5e28f91cf0963ull, 0x209f701c6ffb5bffull}, {0x7bf888302e57b1c8ull, 0x1fdcdc1adfedf8b5ull},
    {0x7c29fbee48c35ca9ull, 0x1f19f97b215f1aafull}, {0x7c5a3d4fdc8173b6ull, 0x1e56ca1e101a1b52ull},
    {0x7c894bddd8eb66dfull, 0x1d934fe54543115dull}, {0x7cb72724226a7415ull, 0x1ccf8cb312b28624ull},
    {0x7ce3ceb193962314ull, 0x1c0b826a7e4f62fdull}, {0x7d0f4217fe4b7270ull, 0x1b4732ef3d67226full},
    {0x7d3980ec2cbcb339ull, 0x1a82a025b004509eull}, {0x7d628ac5e27a1090ull, 0x19bdcbf2dc436666ull},
    {0x7d8a5f3fdd72c0abull, 0x18f8b83c69a60ab6ull}, {0x7db0fdf7d6eedcc3ull, 0x183366e89c64c5baull},
    {0x7dd6668e8481dd85ull, 0x176dd9de50bf3147ull}, {0x7dfa98a798f5b9bbull, 0x16a81304f64ab23eull},
    {0x7e1d93e9c52ea4d6ull, 0x15e214448b3fc655ull}, {0x7e3f57feb9076b3aull, 0x151bdf8597c5f1faull},
    {0x7e5fe49324266a1dull, 0x145576b1293e59dbull}, {0x7e7f3956b6cb20f9ull, 0x138edbb0cd8d13baull},
    {0x7e9d55fc22945a86ull, 0x12c8106e8e613a22ull}, {0x7eba3a391b3eeb63ull, 0x120116d4ec7bceb7ull},
    {0x7ed5e5c6575d048eull, 0x1139f0cedaf576abull}, {0x7ef0585f910617eaull, 0x1072a047ba831d23ull},
    {0x7f0991c3867f4d1full, 0x0fab272b54b9871aull}, {0x7f2191b3fadc8531ull, 0x0ee38765d74fe489ull},
    {0x7f3857f5b699eb51ull, 0x0e1bc2e3cf616a7bull}, {0x7f4de450882e1153ull, 0x0d53db9224ae01bdull},
    {0x7f62368f44949678ull, 0x0c8bd35e14da15f1ull}, {0x7f754e7fc7d1572aull, 0x0bc3ac352ead90acull},
    {0x7f872bf2f56c2469ull, 0x0afb68054d520c61ull}, {0x7f97cebcb8e501b2ull, 0x0a3308bc93904ad7ull},
    {0x7fa736b40620e855ull, 0x096a9049670cfae6ull}, {0x7fb563b2d9cf0f0dull, 0x08a2009a6b84d940ull},
    {0x7fc2559639c6b502ull, 0x07d95b9e7e0837fbull}, {0x7fce0c3e355d6f35ull, 0x0710a344b035f8b4ull},
    {0x7fd8878de5b5f78full, 0x0647d97c437604faull}, {0x7fe1c76b6e077cc6ull, 0x057f0034a43350daull},
    {0x7fe9cbbffbdd7275ull, 0x04b6195d65157346ull}, {0x7ff09477c74fe0bdull, 0x03ed26e63a39e020ull},
    {0x7ff62182133432edull, 0x03242abef46ccfbfull}, {0x7ffa72d12d4684aeull, 0x025b26d77c61dfa7ull},
    {0x7ffd885a6e4b6d5eull, 0x01921d1fcdec7846ull}, {0x7fff62163a2a4936ull, 0x00c90f87f3380389ull},
};

// (x y) >> 32 of a 64-bit and a 32-bit factor
__device__ __forceinline__ uint64_t mul_64x32(uint64_t x, uint32_t y)
{
    return (uint64_t)(uint32_t)(x >> 32) * y + __umulhi((uint32_t)x, y);
}

// sign * m * 2^q as a double, m rounded to 53 bits (m > 0, result normal)
__device__ __forceinline__ double assemble_double(bool neg, uint64_t m, int q)
{
    const int lz = __clzll((long long)m);
    const uint64_t r = ((m << lz) + 0x400ull) >> 11;  // 2^52 .. 2^53
    const uint64_t bits = ((uint64_t)(q - lz + 11 + 52 + 1023 - 1) << 52) + r;
    return __longlong_as_double((long long)(bits | ((uint64_t)neg << 63)));
}

// Box-Muller on a pair of 32-bit words: r cos(2 pi u1), r sin(2 pi u1) with
// r = sqrt(-2 ln u0), u = (word + 1/2) 2^-32.
__device__ __forceinline__ void box_muller(uint32_t a, uint32_t b, double& z0, double& z1)
{
    // -ln u0 / 2 = H 2^(-64 - s)
    const uint64_t n = 2ull * a + 1ull;
    const int lz = __clzll((long long)n), k = lz - 30;
    const uint64_t N = n << lz;
    const LogEntry T = kLogTable[(N >> 55) & 255];
    const uint64_t x = 0ull - (((N >> 31) * T.c) << 16);
    const uint32_t xh = (uint32_t)(x >> 32);
    uint32_t q = 0x24924924u + __umulhi(0x20000000u, xh);  // 1/7 + x/8
    q = 0x2aaaaaaau + __umulhi(q, xh);
    q = 0x33333333u + __umulhi(q, xh);
    uint64_t p = 0x4000000000000000ull + mul_64x32(x, q);
    p = 0x5555555555555555ull + __umul64hi(x, p);
    p = 0x8000000000000000ull + __umul64hi(x, p);
    p = 0x8000000000000000ull + (__umul64hi(x, p) >> 1);  // -ln(1 - x) / (2 x) 2^64
    // k ln 2 - ln(1 / c_j) with 96 fraction bits (ah, al, el), shifted left with x
    // where it is small: the sum keeps 64 significant bits
    constexpr uint64_t kLn2 = 0xb17217f7d1cf79abull;
    constexpr uint32_t kLn2Lo = 0xc9e3b398u;
    const uint64_t kl = kLn2 * (uint64_t)k, ke = (uint64_t)kLn2Lo * (uint32_t)k;
    const uint64_t km = kl + (ke >> 32), tm = km - T.t;
    const uint32_t el = (uint32_t)ke - T.lo, br = (uint32_t)ke < T.lo ? 1u : 0u;
    const uint64_t al = tm - br;
    const uint32_t ah = (uint32_t)(mul_64x32(kLn2, (uint32_t)k) >> 32) + (km < kl ? 1u : 0u) - (km < T.t ? 1u : 0u) -
                        (tm < br ? 1u : 0u);
    const int s = ah ? 0 : __clzll((long long)(al | x));
    const uint64_t X = __umul64hi(x << s, p), as = (al << s) | (((uint64_t)el << s) >> 32);
    const uint64_t lo = (((uint64_t)ah << 63) | (as >> 1)) + X;
    const uint32_t hi = (ah >> 1) + (lo < X ? 1u : 0u);
    // normalise: r^2 = M 2^E, E even
    const int w = 32 - __clz((int)hi);  // bits of hi
    const int sh = hi ? -w : __clzll((long long)lo);
    uint64_t M = hi ? ((uint64_t)hi << (64 - w)) | (lo >> w) : lo << sh;
    int E = -62 - s - sh;
    if (E & 1) {
        M >>= 1;
        E += 1;
    }
    // r = R 2^(E/2 - 31)
    const float y = rsqrt_approx((float)(uint32_t)(M >> 40) * 5.9604644775390625e-8f);
    const uint32_t Y = __float2uint_rz(y * 2147483648.0f);
    const long long e = (long long)(0x4000000000000000ull - __umul64hi(M, (uint64_t)Y * Y));
    const uint64_t G = mul_64x32(M, Y);
    const long long eh = e >> 16;
    const long long c = (e >> 1) + ((((eh * eh) >> 30) * 3) >> 3);
    const uint64_t R = G + (uint64_t)__mul64hi((long long)(G >> 1), c << 3);
    // quadrant, table angle and rest d 2^-64
    const uint32_t quad = b >> 30, fr = 2u * (b & 0x3fffffffu) + 1u;
    const ulonglong2 t = kSinCosTable[fr >> 23];
    const uint64_t d = mul_64x32(0x6487ed5110b4611aull, (fr & 0x7fffffu) << 3);
    const uint64_t d2 = __umul64hi(d, d);
    const uint64_t sd = d - __umul64hi(d, __umul64hi(d2, 0x2aaaaaaaaaaaaaaaull - (mul_64x32(d2, 2290649224u) >> 6)));
    const uint64_t cd =
        __umul64hi(d2, 0x8000000000000000ull - __umul64hi(d2, 0x0aaaaaaaaaaaaaaaull - (mul_64x32(d2, 1527099483u) >> 8)));
    const uint64_t cs = t.y - __umul64hi(t.y, cd) - __umul64hi(t.x, sd);
    const uint64_t sn = t.x - __umul64hi(t.x, cd) + __umul64hi(t.y, sd);
    const bool odd = quad & 1;
    const int qx = (E >> 1) - 30;
    z0 = assemble_double(quad == 1 || quad == 2, __umul64hi(R, odd ? sn : cs), qx);
    z1 = assemble_double(quad >= 2, __umul64hi(R, odd ? cs : sn), qx);
}

}  // namespace flb
