// Constants of mlkd_fixed.h, written by gen_fixed.py beside this file.
// MLKD_CONSTANT is defined there: constant memory on the device.
#pragma once
#include <cstdint>
namespace mlkd {
namespace fx {
// 2 h(s)/s^2, h(s) = exp(-s) + s - 1, and f(s)/s^3, f(s) = 2(exp(-s) - 1) + s(exp(-s) + 1), 0 <= s <= 1
struct PolyHF {
    static constexpr int kLead = 11, kTail = 2;
    static constexpr int kShift0 = 31;
    static constexpr uint32_t tail0[kTail] = {0xa4dbf70au, 0x08364b2au};
    static constexpr int kShift1 = 32;
    static constexpr uint32_t tail1[kTail] = {0x8d1fb798u, 0x07165888u};
};
MLKD_CONSTANT uint64_t kPolyHF[11][2] = {
    {0xffffffffffffffffull, 0x2aaaaaaaaaaaaaaaull},
    {0x5555555555555497ull, 0x1555555555555502ull},
    {0x1555555555552bb4ull, 0x0666666666665440ull},
    {0x044444444440aecbull, 0x016c16c16c153164ull},
    {0x00b60b60b5e24f07ull, 0x0041041040f2280aull},
    {0x001a01a018e9499dull, 0x0009c09c09465f15ull},
    {0x00034033fe7271faull, 0x000143a270f27f92ull},
    {0x00005c77807075d9ull, 0x000024fc9943e9eaull},
    {0x0000093f0b47c9ddull, 0x000003c8554bee00ull},
    {0x000000d70a5c1a4eull, 0x0000005998df72b8ull},
    {0x00000011c91f3c8bull, 0x0000000785d2a9f9ull}};
// sqrt(2 (exp(-h) + h - 1))/h, 0 <= h <= exp(-1)
struct PolyW {
    static constexpr int kLead = 7, kTail = 3;
    static constexpr int kShift0 = 22;
    static constexpr uint32_t tail0[kTail] = {0x837f243au, 0x098fe4d6u, 0x00a41374u};
};
MLKD_CONSTANT uint64_t kPolyW[7][1] = {
    {0xffffffffffffffffull},
    {0x2aaaaaaaaaaaaa9bull},
    {0x071c71c71c71c174ull},
    {0x00f2b9d6480e6752ull},
    {0x001948b0fcc96afaull},
    {0x00020bfad21b8142ull},
    {0x000021e78ee38e7bull}};
// (1 - 2^-f)/f, 0 <= f <= 1
struct PolyE {
    static constexpr int kLead = 10, kTail = 2;
    static constexpr int kShift0 = 31;
    static constexpr uint32_t tail0[kTail] = {0xeadd7cbeu, 0x0a46767du};
};
MLKD_CONSTANT uint64_t kPolyE[10][1] = {
    {0xb17217f7d1cf79aaull},
    {0x3d7f7bff058b1acbull},
    {0x0e35846b824fe76cull},
    {0x0276556df74104a4ull},
    {0x005761ff9dd4a2dfull},
    {0x000a184895de347aull},
    {0x0000ffe5f74da630ull},
    {0x0000162bf1b6bc61ull},
    {0x000001b50af3e60dull},
    {0x0000001e31028c6aull}};
// (1 - sin(z)/z)/z^2 and (1 - cos(z))/z^2 in z^2, |z| <= pi/4
struct PolySC {
    static constexpr int kLead = 5, kTail = 4;
    static constexpr int kShift0 = 32;
    static constexpr uint32_t tail0[kTail] = {0xb092309du, 0x00d73f9fu, 0x0000ca96u, 0x00000098u};
    static constexpr int kShift1 = 28;
    static constexpr uint32_t tail1[kTail] = {0x8f76c780u, 0x00c9cba5u, 0x0000d740u, 0x000000b4u};
};
MLKD_CONSTANT uint64_t kPolySC[5][2] = {
    {0x2aaaaaaaaaaaaaabull, 0x8000000000000000ull},
    {0x0222222222222222ull, 0x0aaaaaaaaaaaaaabull},
    {0x000d00d00d00d00dull, 0x005b05b05b05b05bull},
    {0x00002e3bc74aad8eull, 0x0001a01a01a01a02ull},
    {0x0000006b99159fd5ull, 0x0000049f93edde28ull}};
constexpr uint64_t kLn2_64 = 0xb17217f7d1cf79acull;   // ln 2 in 2^-64
constexpr uint64_t kLn2_58 = 0x02c5c85fdf473de7ull;   // ln 2 in 2^-58
constexpr uint64_t kLog2e_63 = 0xb8aa3b295c17f0bcull; // log2 e in 2^-63
constexpr uint64_t kTwoPi_61 = 0xc90fdaa22168c235ull; // 2 pi in 2^-61
constexpr uint64_t kInvTwoPi_64 = 0x28be60db9391054aull; // 1/(2 pi) in 2^-64
// floor(2^15 256/(129 + j)) and ln of that fraction, in 2^-64
#define MLKD_LOG_RECIPROCALS \
    65027u, 64527u, 64035u, 63550u, 63072u, 62601u, 62137u, 61680u, 61230u, 60787u, 60349u, 59918u, \
    59493u, 59074u, 58661u, 58254u, 57852u, 57456u, 57065u, 56679u, 56299u, 55924u, 55553u, 55188u, \
    54827u, 54471u, 54120u, 53773u, 53430u, 53092u, 52758u, 52428u, 52103u, 51781u, 51463u, 51150u, \
    50840u, 50533u, 50231u, 49932u, 49636u, 49344u, 49056u, 48770u, 48489u, 48210u, 47934u, 47662u, \
    47393u, 47127u, 46863u, 46603u, 46345u, 46091u, 45839u, 45590u, 45343u, 45100u, 44858u, 44620u, \
    44384u, 44150u, 43919u, 43690u, 43464u, 43240u, 43018u, 42799u, 42581u, 42366u, 42153u, 41943u, \
    41734u, 41527u, 41323u, 41120u, 40920u, 40721u, 40524u, 40329u, 40136u, 39945u, 39756u, 39568u, \
    39383u, 39199u, 39016u, 38836u, 38657u, 38479u, 38304u, 38130u, 37957u, 37786u, 37617u, 37449u, \
    37282u, 37117u, 36954u, 36792u, 36631u, 36472u, 36314u, 36157u, 36002u, 35848u, 35696u, 35544u, \
    35394u, 35246u, 35098u, 34952u, 34807u, 34663u, 34521u, 34379u, 34239u, 34100u, 33961u, 33825u, \
    33689u, 33554u, 33420u, 33288u, 33156u, 33026u, 32896u, 32768u
#define MLKD_LOG_TABLE \
    0xaf731b50a6b6b1a3ull, 0xad793ee16746d6e6ull, 0xab83a335d8413283ull, 0xa99161343342b993ull, \
    0xa7a2941aca70c882ull, 0xa5b7577c8d98eb0cull, 0xa3cfc73ee1545f94ull, 0xa1ebff97491dd125ull, \
    0xa00c1d08e34c7277ull, 0x9e303c61b5f5a919ull, 0x9c564eb882351520ull, 0x9a80956cafe41255ull, \
    0x98ae142159b235d3ull, 0x96dee2bd38d9ed96ull, 0x951319683d961d99ull, 0x934ad0899edc926dull, \
    0x9184fec5d1c4b236ull, 0x8fc2dafe28b2c589ull, 0x8e03584d5d0e334bull, 0x8c468a0728c4f390ull, \
    0x8a8dadb77b4e89abull, 0x88d7b11e3a553cd7ull, 0x87237a303844db4bull, 0x857377167aa7d0c6ull, \
    0x83c55e296fd92dfeull, 0x821a71f3855556f7ull, 0x8072c72d8fbd5886ull, 0x7ecd3abde602106cull, \
    0x7d29dbb7c15c8d2dull, 0x7b89f55aa7cf84caull, 0x79ec5f0f3cedb376ull, 0x785128681c9ae0feull, \
    0x76b9a3212d765652ull, 0x75235d1b422193f6ull, 0x738fa65f822a9fc0ull, 0x71ffd71d14d3248cull, \
    0x707171a4fe0e763bull, 0x6ee4806d7f8392c8ull, 0x6d5baa1111222413ull, 0x6bd465491b374048ull, \
    0x6a4ebcf1b3474028ull, 0x68cc100813e98dcdull, 0x674c6fa84fb4eadcull, 0x65cd3d0b70d9f64aull, \
    0x64528b8d6ee82645ull, 0x62d85ea20897c5c4ull, 0x616019dcf4274a38ull, 0x5feb28ef18544bb8ull, \
    0x5e783ba1e2aaf205ull, 0x5d075ddb19e6c585ull, 0x5b97359a36536cdfull, 0x5a2a98fa4d88439eull, \
    0x58bec62c1b1e74b5ull, 0x57569b7d54f4baa5ull, 0x55ef4f4efbe5dcebull, 0x548a581cd08f5ab8ull, \
    0x53265077a5ce5dffull, 0x51c62709c6906c14ull, 0x50658c8e8a9a6f87ull, 0x4f08e9dcbac60a55ull, \
    0x4dad5ddaf0445a5eull, 0x4c52ef86f2535b80ull, 0x4afb23f3418b3a6dull, 0x49a48844536df48bull, \
    0x4850a5b4226349d6ull, 0x46fe058d57ae4ef7ull, 0x45acaf2e68e5a71bull, 0x445e32089f71ef78ull, \
    0x430f879cd369002dull, 0x41c3c9809c411a26ull, 0x40797757d0979a0dull, 0x3f3228d966e6f2f6ull, \
    0x3deac7c98f37bb41ull, 0x3ca4e9ff14d78f87ull, 0x3b622d619d307e01ull, 0x3a1f6fe44abca15bull, \
    0x38dfe78ddf9ee133ull, 0x37a06a70432943aeull, 0x366298ae1e7c09a7ull, 0x35267a7823b2e908ull, \
    0x33ec180d08abcaabull, 0x32b379b92afa5dc6ull, 0x317ca7d62fdcf8a6ull, 0x304602c983466376ull, \
    0x2f12e10a8206e57eull, 0x2ddff916e70d76caull, 0x2cad4d7c3ba5b2f2ull, 0x2b7e40d6a07b62a2ull, \
    0x2a4f7dc93789178bull, 0x292107055921bbe6ull, 0x27f64b4b2a5195beull, 0x26cbe9602aa02c5aull, \
    0x25a1e418acc03c07ull, 0x2479fa542a63c3c5ull, 0x235434fc45ac5394ull, 0x222edd0447c8f667ull, \
    0x2109f56a796b6c92ull, 0x1fe74539048cab73ull, 0x1ec6d582f6891ab6ull, 0x1da6e7637c46a0fbull, \
    0x1c877e015f78eeb7ull, 0x1b6a688d9b5b1760ull, 0x1a4de24086f4272cull, 0x1931ee5c50c88b32ull, \
    0x1818622ea35b7b99ull, 0x16ff7309f8c0031eull, 0x15e8fa4d8591c6fdull, 0x14d1515b987ce306ull, \
    0x13bc29a634a47519ull, 0x12a98ca42af79bc2ull, 0x1195c7d0380c60faull, 0x108498b51e39b133ull, \
    0x0f7426df90f9f5c2ull, 0x0e6475e621d0b8c4ull, 0x0d576f687d567e0cull, 0x0c494d09c7b94404ull, \
    0x0b3de079546ba612ull, 0x0a33476a1671f4c1ull, 0x0927979600c7e5bbull, 0x08209ec4f3222233ull, \
    0x071896baf3e8b82aull, 0x06117149d7127c61ull, 0x050b324851e221c7ull, 0x0407d5961cd6107dull, \
    0x03037113d7f3e59cull, 0x0201faaeb0fbce24ull, 0x00ff805515885e02ull, 0x0000000000000000ull
}  // namespace fx
}  // namespace mlkd
