// tanh of an FP64 number to 0.52 units in the last place (CUDA's tanh: up to
// 1), in 64-bit integer arithmetic.  The FP64 pipe retires 2 lanes a clock and SM; CUDA's
// tanh() takes 1370 clocks a warp and scheduler there (10.3 ms for 302 M
// values), this about a tenth, on the integer pipe.
//
// With x = |theta| and k = round(16 x), b = x - k / 16 (|b| <= 1/32):
//   tanh b = b (1 - c), c = z/3 - 2 z^2/15 + 17 z^3/315 - 62 z^4/2835 + 1382
//     z^5/155925, z = b^2 (the Maclaurin series; the next term is below 2^-68);
//   tanh x = ta + tb (1 - ta^2) / (1 + ta tb), ta = tanh(k / 16) and 1 - ta^2
//     from a table of 307 pairs (rounded from 60 digits), tb = tanh b, the
//     division by a reciprocal of 24 bits, r, improved to r (1 + e + e^2) with
//     e = 1 - r (1 + ta tb).
// Fixed point throughout, each step within a few units of 2^-63; x below 1/32
// multiplies its own mantissa by 1 - c, so small results keep their relative
// accuracy; x below 2^-28 is its own tanh, x from 19.0625 on gives 1.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace nk {
namespace {

#define NK_TANH_TABLE_ROWS 307
#define NK_TANH_TABLE \
    {0x0000000000000000ULL, 0xffffffffffffffffULL}, {0x0ffaaccbf0186b83ULL, 0xff00aa4a26e9869dULL}, \
    {0x1fd5992bc4b834fcULL, 0xfc0a92af27e0b003ULL}, {0x2f71ff2077eeec65ULL, 0xf734f18edb0ab13aULL}, \
    {0x3eb2fd4d34390be2ULL, 0xf0a4d02960b60e69ULL}, {0x4d7e6283a99437c7ULL, 0xe88aba57ac78d6ffULL}, \
    {0x5bbd4f7a323ebfc5ULL, 0xdf1fdd80ad2c8dacULL}, {0x695ca7b92200dce2ULL, 0xd4a2dce12727c9f0ULL}, \
    {0x764d4f5d5a2bcd94ULL, 0xc954a37d1a1ca070ULL}, {0x82843797b6a5b4ecULL, 0xbd75734089f8cefaULL}, \
    {0x8dfa3f55dc7caa44ULL, 0xb142619ba7c0a9a3ULL}, {0x98abeff4fb8ad9ffULL, 0xa4f35f92a317b984ULL}, \
    {0xa2991f2a9791413aULL, 0x98b9d8f7d377a608ULL}, {0xabc47f88694cc375ULL, 0x8cbfe6cc3ae9942dULL}, \
    {0xb433285c6100a8d0ULL, 0x81280504fc6b6cb2ULL}, {0xbbec1c71a02be187ULL, 0x760d34ad8b578624ULL}, \
    {0xc2f7d5a8a79ca2acULL, 0x6b83703e6431132aULL}, {0xc95fd9b86cdb8cc7ULL, 0x6198583915044495ULL}, \
    {0xcf2e5add226b4970ULL, 0x585400a99a9de576ULL}, {0xd46de5e18c4bd30aULL, 0x4fb9cc14df23a62fULL}, \
    {0xd9291ddb596f713bULL, 0x47c944c78ea2fe22ULL}, {0xdd6a8525345e0c37ULL, 0x407ee9cb3b869335ULL}, \
    {0xe13c52952723bd98ULL, 0x39d4e89f00a4f000ULL}, {0xe4a8519a0645fbf7ULL, 0x33c3bffa70a846b2ULL}, \
    {0xe7b7cbc36fabbb07ULL, 0x2e42ca5058dee4a7ULL}, {0xea737a321435854eULL, 0x2948b0856fbc3b28ULL}, \
    {0xece37d7f30e3c28fULL, 0x24cbc675b0c5e86dULL}, {0xef0f5ac9ba8c7951ULL, 0x20c2538f91d762e3ULL}, \
    {0xf0fdfcbf19a93607ULL, 0x1d22ca1c24a13911ULL}, {0xf2b5b79f7d5fe7caULL, 0x19e3efd94bb9fb8bULL}, \
    {0xf43c4f67606ed2fcULL, 0x16fcfa6d9f169299ULL}, {0xf596ff6eaf6498d8ULL, 0x1465a205cfb6384aULL}, \
    {0xf6ca82f0de1e9e9aULL, 0x12162c262e051aa6ULL}, {0xf7db1e0f99ccc3d2ULL, 0x1007707172fe10cbULL}, \
    {0xf8cca6fb927e41a8ULL, 0x0e32d8de064eae5dULL}, {0xf9a28f044cf1078dULL, 0x0c925e9050fbf03aULL}, \
    {0xfa5feb616fe8f131ULL, 0x0b20845526aff17dULL}, {0xfb077d9609424553ULL, 0x09d84f83ae07ad75ULL}, \
    {0xfb9bbb595516dadfULL, 0x08b53fe26bdc83a7ULL}, {0xfc1ed5f91f0bb6b4ULL, 0x07b34706b1a52978ULL}, \
    {0xfc92c130538e0e3cULL, 0x06cebf87ee971ed7ULL}, {0xfcf9397127f3631aULL, 0x060464486e5587a0ULL}, \
    {0xfd53c9a5baf5e807ULL, 0x055148020c290d0eULL}, {0xfda3d06c7b691d1eULL, 0x04b2cd36803c9e15ULL}, \
    {0xfdea84d73d71f32dULL, 0x04269e977221c4b2ULL}, {0xfe28fab4e03eda95ULL, 0x03aaa7f1c4f76cd6ULL}, \
    {0xfe60266de6e25de7ULL, 0x033d0fa111a4d429ULL}, {0xfe90e07c8e32c05cULL, 0x02dc308b84d91bbeULL}, \
    {0xfebbe888d057ff10ULL, 0x028694a2f778be8fULL}, {0xfee1e8308068ffafULL, 0x023aefe5c955fa22ULL}, \
    {0xff03758344109209ULL, 0x01f81bd887622528ULL}, {0xff211539ba03ec60ULL, 0x01bd137084c7b48cULL}, \
    {0xff3b3cae9a9d02b6ULL, 0x0188ef67211da0abULL}, {0xff5253a01a6ba824ULL, 0x015ae2ed5d7b64cfULL}, \
    {0xff66b5bf5189406eULL, 0x013238b786137ffeULL}, {0xff78b412e912d77fULL, 0x010e505903475be0ULL}, \
    {0xff889631d483b9ddULL, 0x00ee9be8cd915906ULL}, {0xff969b5a6816ca30ULL, 0x00d29de7786a0486ULL}, \
    {0xffa2fb69b099d70aULL, 0x00b9e760498196f5ULL}, {0xffade7b68c922010ULL, 0x00a4163f557ff2c5ULL}, \
    {0xffb78bd3aa3b9035ULL, 0x0090d3d71de06bafULL}, {0xffc00e3b399d77d5ULL, 0x007fd390a9975712ULL}, \
    {0xffc790e6d553178dULL, 0x0070d1c18a204fc6ULL}, {0xffce31d5df4f9e38ULL, 0x006392a3af386c80ULL}, \
    {0xffd40b84505a10b4ULL, 0x0057e16b5442da43ULL}, {0xffd93553c0bd1b7cULL, 0x004d8f77b2eeb971ULL}, \
    {0xffddc3e83e2ef796ULL, 0x0044739b7f37703fULL}, {0xffe1c97a55c6a9a5ULL, 0x003c697a81821dabULL}, \
    {0xffe5561f90732ee8ULL, 0x003550f9ecc8e18aULL}, {0xffe8780a7c6268b1ULL, 0x002f0dc150e8ac08ULL}, \
    {0xffeb3bc33dabfbf7ULL, 0x002986ca44bc92f4ULL}, {0xffedac598403109fULL, 0x0024a5fd193b0e86ULL}, \
    {0xffefd390a9cc1bbaULL, 0x002057d916c68c02ULL}, {0xfff1ba06aa64d38dULL, 0x001c8b26f0d0a0efULL}, \
    {0xfff367568966e544ULL, 0x001930b442456a1aULL}, {0xfff4e236b2ec18e6ULL, 0x00163b170763f4bdULL}, \
    {0xfff63093cd1d23f7ULL, 0x00139e782819fc19ULL}, {0xfff757a86562b2beULL, 0x00115064410dd7c7ULL}, \
    {0xfff85c11d7373153ULL, 0x000f47a1f1923cdfULL}, {0xfff941e2bfa9ef2dULL, 0x000d7c0d0a1daec6ULL}, \
    {0xfffa0cb346f889a8ULL, 0x000be67609d4f423ULL}, {0xfffabfaf8115ae98ULL, 0x000a80856a8754e5ULL}, \
    {0xfffb5da41e63c866ULL, 0x000944a24960f7ceULL}, {0xfffbe9099f3a1c53ULL, 0x00082ddc07c97b6aULL}, \
    {0xfffc640e36e19f21ULL, 0x000737d68b935d20ULL}, {0xfffcd09e857d71afULL, 0x00065eb8cff74d78ULL}, \
    {0xfffd306d4bb552f5ULL, 0x00059f1d81fbf548ULL}, {0xfffd84fa36e466e0ULL, 0x0004f6056b017e70ULL}, \
    {0xfffdcf97e0f48b8eULL, 0x000460cb734f36b9ULL}, {0xfffe11711bdffb03ULL, 0x0003dd1a0cd441ccULL}, \
    {0xfffe4b8d9e03a6fdULL, 0x000368e1dbe2e127ULL}, {0xfffe7ed621f186adULL, 0x00030251789dfde6ULL}, \
    {0xfffeac180a4128a2ULL, 0x0002a7ce282d87b8ULL}, {0xfffed40897ed9cd6ULL, 0x000257ed70a8ea20ULL}, \
    {0xfffef747c01a8b7cULL, 0x0002116f6e0e60a3ULL}, {0xffff1662ac984702ULL, 0x0001d339d19faf7bULL}, \
    {0xffff31d5f129deeeULL, 0x00019c5377a48b5bULL}, {0xffff4a0f7e6363a5ULL, 0x00016be081eb3f7bULL}, \
    {0xffff5f7059ecfc2bULL, 0x0001411ee7722777ULL}, {0xffff724e230d05d2ULL, 0x00011b636b788b65ULL}, \
    {0xffff82f4698c8c95ULL, 0x0000fa16efd29564ULL}, {0xffff91a5dc52c8ddULL, 0x0000dcb417c8d7dfULL}, \
    {0xffff9e9d54731c7eULL, 0x0000c2c5320ddafbULL}, {0xffffaa0ec0dac12cULL, 0x0000abe261706662ULL}, \
    {0xffffb427f64dc733ULL, 0x000097affcec259bULL}, {0xffffbd1166f42da1ULL, 0x000085dd2097bf73ULL}, \
    {0xffffc4eec4560b17ULL, 0x0000762269b2f728ULL}, {0xffffcbdf8e4f691fULL, 0x00006840d8c3fb76ULL}, \
    {0xffffd1ff913841bbULL, 0x00005c00d54b54b9ULL}, {0xffffd7675539cfecULL, 0x000051314f1c4fbfULL}, \
    {0xffffdc2c808f0a75ULL, 0x000047a6f9de6782ULL}, {0xffffe0622e39bf9dULL, 0x00003f3b9fa4e6acULL}, \
    {0xffffe4193a878ed7ULL, 0x000037cd87e664a4ULL}, {0xffffe76086993192ULL, 0x0000313ef06f52c0ULL}, \
    {0xffffea4533fa83c0ULL, 0x00002b759632cab9ULL}, {0xffffecd2d939f64dULL, 0x0000265a4c1c57afULL}, \
    {0xffffef13b0520b7aULL, 0x000021d89e3d84f3ULL}, {0xfffff110bf9ebdc0ULL, 0x00001dde7fe379ddULL}, \
    {0xfffff2d1fe02daeaULL, 0x00001a5c034c95b4ULL}, {0xfffff45e72ce1738ULL, 0x0000174319dc897aULL}, \
    {0xfffff5bc51e399caULL, 0x000014875bcf70ecULL}, {0xfffff6f11491c0f2ULL, 0x0000121dd68a70b0ULL}, \
    {0xfffff8018f7e9db3ULL, 0x00000ffce0c2dd90ULL}, {0xfffff8f20600f4eaULL, 0x00000e1bf3cc51bdULL}, \
    {0xfffff9c63b33435cULL, 0x00000c738972b705ULL}, {0xfffffa818105271dULL, 0x00000afcfdd7824fULL}, \
    {0xfffffb26c58787afULL, 0x000009b274d96e79ULL}, {0xfffffbb89ea8beffULL, 0x0000088ec29c3310ULL}, \
    {0xfffffc39548fc348ULL, 0x0000078d56d2373dULL}, {0xfffffcaaeabfcc3fULL, 0x000006aa2a754cbcULL}, \
    {0xfffffd0f28290e18ULL, 0x000005e1afa53ddcULL}, {0xfffffd679e46d80fULL, 0x00000530c36b93a7ULL}, \
    {0xfffffdb5af67984dULL, 0x00000494a12b9092ULL}, {0xfffffdfa9437ed8bULL, 0x0000040ad78c0f1eULL}, \
    {0xfffffe3760a6fa1dULL, 0x000003913eaedd4fULL}, {0xfffffe6d08379024ULL, 0x00000325ef8e6569ULL}, \
    {0xfffffe9c61cf815aULL, 0x000002c73c5f0f4dULL}, {0xfffffec62b1454beULL, 0x00000273a9d5d5caULL}, \
    {0xfffffeeb0b62d980ULL, 0x00000229e9392160ULL}, {0xffffff0b966d7952ULL, 0x000001e8d3242403ULL}, \
    {0xffffff284e8bc6fcULL, 0x000001af62e7bc4dULL}, {0xffffff41a6c48a6aULL, 0x0000017cb2765da4ULL}, \
    {0xffffff58049a7530ULL, 0x0000014ff6caa767ULL}, {0xffffff6bc1a2b4a8ULL, 0x000001287cba40d8ULL}, \
    {0xffffff7d2cebbe21ULL, 0x00000105a62840e4ULL}, {0xffffff8c8c39f21cULL, 0x000000e6e78be7b7ULL}, \
    {0xffffff9a1d1f0ae0ULL, 0x000000cbc5c1c1b4ULL}, {0xffffffa615f0b57aULL, 0x000000b3d41e7578ULL}, \
    {0xffffffb0a6a230ecULL, 0x0000009eb2bb8590ULL}, {0xffffffb9f9845b1dULL, 0x0000008c0cf7369fULL}, \
    {0xffffffc233ef2cc0ULL, 0x0000007b98219795ULL}, {0xffffffc976d74b07ULL, 0x0000006d12515e53ULL}, \
    {0xffffffcfdf52062dULL, 0x00000060415bea99ULL}, {0xffffffd58709d581ULL, 0x00000054f1ec4df2ULL}, \
    {0xffffffda84a52380ULL, 0x0000004af6b5b384ULL}, {0xffffffdeec2105b5ULL, 0x0000004227bdf051ULL}, \
    {0xffffffe2cf214bbaULL, 0x0000003a61bd6538ULL}, {0xffffffe63d3725fdULL, 0x000000338591b16eULL}, \
    {0xffffffe9441f7f48ULL, 0x0000002d77c0ff6bULL}, {0xffffffebeffa02bbULL, 0x00000028200bf8f7ULL}, \
    {0xffffffee4b79aaa9ULL, 0x00000023690ca974ULL}, {0xfffffff0600f9ac6ULL, 0x0000001f3fe0c980ULL}, \
    {0xfffffff23610f14bULL, 0x0000001b93de1cacULL}, {0xfffffff3d4d82692ULL, 0x00000018564fb247ULL}, \
    {0xfffffff542e280c3ULL, 0x000000157a3afe06ULL}, {0xfffffff685ea1194ULL, 0x00000012f42bdc7eULL}, \
    {0xfffffff7a2fca636ULL, 0x00000010ba06b34eULL}, {0xfffffff89e900547ULL, 0x0000000ec2dff53cULL}, \
    {0xfffffff97c93cbdeULL, 0x0000000d06d8681aULL}, {0xfffffffa40813142ULL, 0x0000000b7efd9d5bULL}, \
    {0xfffffffaed68f068ULL, 0x0000000a252e1f17ULL}, {0xfffffffb85ff8ef5ULL, 0x00000008f400e203ULL}, \
    {0xfffffffc0ca832f2ULL, 0x00000007e6af9a0dULL}, {0xfffffffc837e3292ULL, 0x00000006f9039ad0ULL}, \
    {0xfffffffcec5d845bULL, 0x000000062744f740ULL}, {0xfffffffd48ea317dULL, 0x000000056e2b9cffULL}, \
    {0xfffffffd9a96e821ULL, 0x00000004cad22fb9ULL}, {0xfffffffde2aac817ULL, 0x000000043aaa6fceULL}, \
    {0xfffffffe22468106ULL, 0x00000003bb72fdf0ULL}, {0xfffffffe5a68d6adULL, 0x000000034b2e52a2ULL}, \
    {0xfffffffe8bf29d46ULL, 0x00000002e81ac573ULL}, {0xfffffffeb7aa3dffULL, 0x0000000290ab8401ULL}, \
    {0xfffffffede3ed1aeULL, 0x0000000243825ca2ULL}, {0xffffffff004ade1aULL, 0x00000001ff6a43ccULL}, \
    {0xffffffff1e56c0dfULL, 0x00000001c3527e42ULL}, {0xffffffff38dad19dULL, 0x000000018e4a5cc4ULL}, \
    {0xffffffff504143f8ULL, 0x000000015f7d780fULL}, {0xffffffff64e7d0f0ULL, 0x0000000136305e1fULL}, \
    {0xffffffff77212e45ULL, 0x0000000111bda375ULL}, {0xffffffff873659bdULL, 0x00000000f1934c86ULL}, \
    {0xffffffff9567bd79ULL, 0x00000000d530850eULL}, {0xffffffffa1ee31f8ULL, 0x00000000bc239c11ULL}, \
    {0xffffffffacfbe1c0ULL, 0x00000000a6083c7fULL}, {0xffffffffb6bd1251ULL, 0x000000009285db5dULL}, \
    {0xffffffffbf58d570ULL, 0x00000000814e5520ULL}, {0xffffffffc6f1a5a4ULL, 0x00000000721cb4b7ULL}, \
    {0xffffffffcda5f052ULL, 0x0000000064b41f5cULL}, {0xffffffffd3908f96ULL, 0x0000000058dee0d5ULL}, \
    {0xffffffffd8c935d0ULL, 0x000000004e6d9460ULL}, {0xffffffffdd64cc92ULL, 0x00000000453666dcULL}, \
    {0xffffffffe175c85cULL, 0x000000003d146f49ULL}, {0xffffffffe50c7289ULL, 0x0000000035e71aeeULL}, \
    {0xffffffffe8372a8cULL, 0x000000002f91aae7ULL}, {0xffffffffeb029f7fULL, 0x0000000029fac102ULL}, \
    {0xffffffffed7a02f0ULL, 0x00000000250bfa20ULL}, {0xffffffffefa735b6ULL, 0x0000000020b19494ULL}, \
    {0xfffffffff192ef85ULL, 0x000000001cda20f6ULL}, {0xfffffffff344e1d3ULL, 0x0000000019763c5aULL}, \
    {0xfffffffff4c3d6acULL, 0x00000000167852a7ULL}, {0xfffffffff615cbe4ULL, 0x0000000013d46838ULL}, \
    {0xfffffffff7400b11ULL, 0x00000000117fe9deULL}, {0xfffffffff8473ebeULL, 0x000000000f718284ULL}, \
    {0xfffffffff92f8519ULL, 0x000000000da0f5ceULL}, {0xfffffffff9fc8071ULL, 0x000000000c06ff1eULL}, \
    {0xfffffffffab165c5ULL, 0x000000000a9d3476ULL}, {0xfffffffffb51099cULL, 0x00000000095decc8ULL}, \
    {0xfffffffffbddeb5aULL, 0x000000000844294cULL}, {0xfffffffffc5a3f42ULL, 0x00000000074b817dULL}, \
    {0xfffffffffcc7f749ULL, 0x000000000670116fULL}, {0xfffffffffd28cae2ULL, 0x0000000005ae6a3dULL}, \
    {0xfffffffffd7e3ddcULL, 0x0000000005038448ULL}, {0xfffffffffdc9a676ULL, 0x00000000046cb314ULL}, \
    {0xfffffffffe0c32b6ULL, 0x0000000003e79a94ULL}, {0xfffffffffe46ed26ULL, 0x00000000037225b4ULL}, \
    {0xfffffffffe7ac0feULL, 0x00000000030a7e04ULL}, {0xfffffffffea87dd3ULL, 0x0000000002af045aULL}, \
    {0xfffffffffed0dad5ULL, 0x00000000025e4a56ULL}, {0xfffffffffef479aeULL, 0x0000000002170ca4ULL}, \
    {0xffffffffff13e909ULL, 0x0000000001d82deeULL}, {0xffffffffff2fa6cdULL, 0x0000000001a0b266ULL}, \
    {0xffffffffff482216ULL, 0x00000000016fbbd4ULL}, {0xffffffffff5dbcf3ULL, 0x000000000144861bULL}, \
    {0xffffffffff70cdeaULL, 0x00000000011e642cULL}, {0xffffffffff81a15aULL, 0x0000000000fcbd4bULL}, \
    {0xffffffffff907aa8ULL, 0x0000000000df0ab1ULL}, {0xffffffffff9d954aULL, 0x0000000000c4d56bULL}, \
    {0xffffffffffa925bfULL, 0x0000000000adb481ULL}, {0xffffffffffb35a57ULL, 0x0000000000994b51ULL}, \
    {0xffffffffffbc5bf2ULL, 0x000000000087481bULL}, {0xffffffffffc44ea3ULL, 0x00000000007762baULL}, \
    {0xffffffffffcb523eULL, 0x0000000000695b83ULL}, {0xffffffffffd182ddULL, 0x00000000005cfa47ULL}, \
    {0xffffffffffd6f948ULL, 0x0000000000520d6fULL}, {0xffffffffffdbcb62ULL, 0x000000000048693bULL}, \
    {0xffffffffffe00c7aULL, 0x00000000003fe70dULL}, {0xffffffffffe3cd98ULL, 0x00000000003864cfULL}, \
    {0xffffffffffe71dc8ULL, 0x000000000031c471ULL}, {0xffffffffffea0a4dULL, 0x00000000002beb66ULL}, \
    {0xffffffffffec9edeULL, 0x000000000026c244ULL}, {0xffffffffffeee5d1ULL, 0x000000000022345eULL}, \
    {0xfffffffffff0e844ULL, 0x00000000001e2f78ULL}, {0xfffffffffff2ae44ULL, 0x00000000001aa377ULL}, \
    {0xfffffffffff43eecULL, 0x0000000000178228ULL}, {0xfffffffffff5a07fULL, 0x000000000014bf01ULL}, \
    {0xfffffffffff6d887ULL, 0x0000000000124ef2ULL}, {0xfffffffffff7ebe4ULL, 0x0000000000102837ULL}, \
    {0xfffffffffff8dee7ULL, 0x00000000000e4232ULL}, {0xfffffffffff9b55bULL, 0x00000000000c954aULL}, \
    {0xfffffffffffa729dULL, 0x00000000000b1ac7ULL}, {0xfffffffffffb19a1ULL, 0x000000000009ccbeULL}, \
    {0xfffffffffffbad06ULL, 0x000000000008a5f5ULL}, {0xfffffffffffc2f18ULL, 0x000000000007a1cfULL}, \
    {0xfffffffffffca1e2ULL, 0x000000000006bc3bULL}, {0xfffffffffffd0730ULL, 0x000000000005f1a1ULL}, \
    {0xfffffffffffd6095ULL, 0x0000000000053ed5ULL}, {0xfffffffffffdaf7aULL, 0x000000000004a10cULL}, \
    {0xfffffffffffdf51aULL, 0x00000000000415cdULL}, {0xfffffffffffe328bULL, 0x0000000000039aeaULL}, \
    {0xfffffffffffe68c4ULL, 0x0000000000032e78ULL}, {0xfffffffffffe989eULL, 0x000000000002cec4ULL}, \
    {0xfffffffffffec2d8ULL, 0x0000000000027a4fULL}, {0xfffffffffffee81dULL, 0x0000000000022fc7ULL}, \
    {0xffffffffffff0900ULL, 0x000000000001ee00ULL}, {0xffffffffffff2606ULL, 0x000000000001b3f4ULL}, \
    {0xffffffffffff3fa3ULL, 0x00000000000180baULL}, {0xffffffffffff563dULL, 0x0000000000015385ULL}, \
    {0xffffffffffff6a30ULL, 0x0000000000012ba0ULL}, {0xffffffffffff7bcaULL, 0x000000000001086bULL}, \
    {0xffffffffffff8b53ULL, 0x000000000000e959ULL}, {0xffffffffffff9909ULL, 0x000000000000cdeeULL}, \
    {0xffffffffffffa522ULL, 0x000000000000b5bcULL}, {0xffffffffffffafd0ULL, 0x000000000000a061ULL}, \
    {0xffffffffffffb93cULL, 0x0000000000008d89ULL}, {0xffffffffffffc18cULL, 0x0000000000007ce7ULL}, \
    {0xffffffffffffc8e3ULL, 0x0000000000006e3aULL}, {0xffffffffffffcf5dULL, 0x0000000000006146ULL}, \
    {0xffffffffffffd514ULL, 0x00000000000055d8ULL}, {0xffffffffffffda1fULL, 0x0000000000004bc2ULL}, \
    {0xffffffffffffde92ULL, 0x00000000000042dbULL}, {0xffffffffffffe280ULL, 0x0000000000003b00ULL}, \
    {0xffffffffffffe5f7ULL, 0x0000000000003411ULL}, {0xffffffffffffe907ULL, 0x0000000000002df3ULL}, \
    {0xffffffffffffebbaULL, 0x000000000000288dULL}, {0xffffffffffffee1bULL, 0x00000000000023c9ULL}, \
    {0xfffffffffffff036ULL, 0x0000000000001f95ULL}, {0xfffffffffffff211ULL, 0x0000000000001bdfULL}, \
    {0xfffffffffffff3b4ULL, 0x0000000000001898ULL}, {0xfffffffffffff526ULL, 0x00000000000015b4ULL}, \
    {0xfffffffffffff66cULL, 0x0000000000001328ULL}, {0xfffffffffffff78cULL, 0x00000000000010e7ULL}, \
    {0xfffffffffffff88bULL, 0x0000000000000eebULL}, {0xfffffffffffff96bULL, 0x0000000000000d2aULL}, \
    {0xfffffffffffffa31ULL, 0x0000000000000b9eULL}, {0xfffffffffffffae0ULL, 0x0000000000000a41ULL}, \
    {0xfffffffffffffb7aULL, 0x000000000000090cULL}, {0xfffffffffffffc02ULL, 0x00000000000007fcULL}, \
    {0xfffffffffffffc7aULL, 0x000000000000070cULL}

__device__ const ulonglong2 g_tanh_table[NK_TANH_TABLE_ROWS] = {NK_TANH_TABLE};

__host__ __device__ __forceinline__ unsigned long long mulhi64(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}

// table: the rows of NK_TANH_TABLE (tanh(k / 16) and 1 - tanh^2, times 2^64).
__host__ __device__ __forceinline__ double tanh64_with(double theta, const ulonglong2 *table) {
    typedef unsigned long long u64;
    u64 bits;
#ifdef __CUDA_ARCH__
    bits = (u64)__double_as_longlong(theta);
#else
    memcpy(&bits, &theta, 8);
#endif
    const u64 sign = bits & 0x8000000000000000ULL;
    const int be = (int)((bits >> 52) & 0x7FF);
    const u64 m = (bits & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
    u64 out;
    const u64 mag = bits ^ sign;
    if (mag < (u64)(1023 - 28) << 52) {
        out = mag;  // x < 2^-28 (zeros and subnormals too)
    } else if (mag >= 0x4033100000000000ULL) {
        out = mag > 0x7FF0000000000000ULL ? mag : 0x3FF0000000000000ULL;  // NaN, or 1 from 19.0625 on
    } else {
        // x 2^58 (x < 2^5: below 2^63); be - 1075 + 58 is between -50 and 10
        const int sh = be - 1017;
        const u64 X = sh >= 0 ? m << sh : m >> (-sh);
        const u64 k = (X + (1ULL << 53)) >> 54;  // round(16 x)
        const long long bs = (long long)(X - (k << 54));
        const u64 b = (bs < 0 ? (u64)-bs : (u64)bs) << 10;  // |b| 2^68 <= 2^63
        u64 w = mulhi64(b, b);                              // b^2 2^72 <= 2^62
        w = (w - (w >> 62)) << 2;                           // (b^2 2^10) 2^64
        const uint32_t w32 = (uint32_t)(w >> 32);
        // c 2^10 = w (1/3 - 2^-10 w (2/15 - 2^-10 w (17/315 - ...))), the inner
        // terms in 32 bits
#ifdef __CUDA_ARCH__
        const uint32_t q4 = 93928738U - (__umulhi(w32, 38067306U) >> 10);
        const uint32_t q3 = 231791885U - (__umulhi(w32, q4) >> 10);
#else
        const uint32_t q4 = 93928738U - ((uint32_t)(((u64)w32 * 38067306U) >> 32) >> 10);
        const uint32_t q3 = 231791885U - ((uint32_t)(((u64)w32 * q4) >> 32) >> 10);
#endif
        const u64 q2 = 0x2222222222222222ULL - (((u64)w32 * q3) >> 10);
        const u64 q1 = 0x5555555555555555ULL - (mulhi64(w, q2) >> 10);
        const u64 c = mulhi64(w, q1);
        const u64 a = k == 0 ? m << 11 : b;  // x's mantissa, or |b| 2^68
        const u64 tb = a - (mulhi64(a, c) >> 10);
        u64 n;   // leading one at bit 63
        int e;   // its exponent
        if (k == 0) {
            const int z = (int)(1 - (tb >> 63));  // 1 - c > 1/2
            n = tb << z;
            e = be - z;
        } else {
            const ulonglong2 row = table[k];
            const u64 eps = mulhi64(row.x, tb);                             // ta |tb| 2^68
            const u64 num = mulhi64(row.y, tb);                             // |tb| (1 - ta^2) 2^68
            const u64 den = bs < 0 ? (1ULL << 63) - (eps >> 5) : (1ULL << 63) + (eps >> 5);  // (1 + ta tb) 2^63
            const float df = (float)(uint32_t)(den >> 32) * 4.656612873077393e-10f;          // 2^-31
#ifdef __CUDA_ARCH__
            const uint32_t r = __float2uint_rn(__frcp_rn(df) * 2147483648.0f);
#else
            const uint32_t r = (uint32_t)(1.0f / df * 2147483648.0f + 0.5f);
#endif
            const u64 rq = (u64)r << 32;                                    // 2^63 / (1 + ta tb)
            const long long er = (long long)((1ULL << 62) - mulhi64(rq, den));  // e 2^62, |e| < 2^-20
            const long long eh = er >> 16;
            const long long g = er + ((eh * eh) >> 30);                     // (e + e^2) 2^62
            const u64 n1 = mulhi64(num, rq);                                // 2^67
            const u64 ga = g < 0 ? (u64)-g : (u64)g;
            const u64 cg = mulhi64(n1, ga << 20) >> 18;                     // n1 |g|, 2^67
            const u64 d = (g < 0 ? n1 - cg : n1 + cg) >> 3;
            const u64 t = bs < 0 ? row.x - d : row.x + d;                   // 2^64
#ifdef __CUDA_ARCH__
            const int z = __clzll((long long)t);
#else
            const int z = __builtin_clzll(t);
#endif
            n = t << z;
            e = 1022 - z;
        }
        // round to 53 bits (a carry lifts the exponent)
        out = ((u64)(e - 1) << 52) + (((n >> 10) + 1ULL) >> 1);
    }
    out |= sign;
    double v;
#ifdef __CUDA_ARCH__
    v = __longlong_as_double((long long)out);
#else
    memcpy(&v, &out, 8);
#endif
    return v;
}

__device__ __forceinline__ double tanh64(double theta) { return tanh64_with(theta, g_tanh_table); }

// t as an FP32 pair, h = fl32(t) and l = fl32(t - h) (t - h is exact in FP64),
// with integer operations only for |t| in [2^-64, 1]: the top 24 bits of the
// mantissa rounded to nearest even, and the signed rest.
__device__ __forceinline__ float2 fp32_pair(double t) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(t);
    const int be = (int)((bits >> 52) & 0x7FF);
    if (be < 1023 - 64 || be > 1023) {
        const float h = __double2float_rn(t);
        return make_float2(h, __double2float_rn(t - (double)h));
    }
    const uint32_t sign = (uint32_t)(bits >> 63) << 31;
    const uint32_t top = (uint32_t)(bits >> 29) & 0x7FFFFFU, rest = (uint32_t)bits & 0x1FFFFFFFU;
    const uint32_t up = rest > 0x10000000U || (rest == 0x10000000U && (top & 1U)) ? 1U : 0U;
    const uint32_t h = ((uint32_t)(be - 896) << 23) + top + up;  // a carry lifts the exponent
    const int low = (int)rest - (int)(up << 29);                 // t - h in units of 2^(be - 1075)
    const float l = __fmul_rn(__int2float_rn(low), __uint_as_float((uint32_t)(be - 948) << 23));
    return make_float2(__uint_as_float(sign | h), __uint_as_float(__float_as_uint(l) ^ sign));
}

}  // namespace
}  // namespace nk
