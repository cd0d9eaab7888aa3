// fx64_tables.h -- fixed-point constants of fx64.cuh: values of ln, sin, cos
// and powers of two at the cell points of its tables and Taylor coefficients
// of its polynomials, each rounded to nearest at the stated scale.
#pragma once
#include <stdint.h>

// ln 2 at 2^64
constexpr uint64_t FX_LN2_64 = 0xb17217f7d1cf79acull;
// 1 / (2 64^0) at 2^64
constexpr uint64_t FX_LOG_C0 = 0x8000000000000000ull;
// 1 / (3 64^1) at 2^64
constexpr uint64_t FX_LOG_C1 = 0x155555555555555ull;
// 1 / (4 64^2) at 2^64
constexpr uint64_t FX_LOG_C2 = 0x4000000000000ull;
// 1 / (5 64^3) at 2^64
constexpr uint64_t FX_LOG_C3 = 0xccccccccccdull;
// 1 / (6 64^4) at 2^64
constexpr uint64_t FX_LOG_C4 = 0x2aaaaaaaabull;
// 1 / (7 64^5) at 2^64
constexpr uint64_t FX_LOG_C5 = 0x92492492ull;
// 1 / (8 64^6) at 2^64
constexpr uint64_t FX_LOG_C6 = 0x2000000ull;
// (pi/128)^1 / 1! at 2^64
constexpr uint64_t FX_TRIG_K1 = 0x6487ed5110b4612ull;
// (pi/128)^2 / 2! at 2^64
constexpr uint64_t FX_TRIG_K2 = 0x13bd3cc9be45deull;
// (pi/128)^3 / 3! at 2^64
constexpr uint64_t FX_TRIG_K3 = 0x295779cc4b7dull;
// (pi/128)^4 / 4! at 2^64
constexpr uint64_t FX_TRIG_K4 = 0x40f07c206dull;
// (pi/128)^5 / 5! at 2^64
constexpr uint64_t FX_TRIG_K5 = 0x519af19eull;
// (pi/128)^6 / 6! at 2^64
constexpr uint64_t FX_TRIG_K6 = 0x5574f2ull;
// (pi/128)^7 / 7! at 2^64
constexpr uint64_t FX_TRIG_K7 = 0x4cb5ull;
// 2 log2(e) at 2^62
constexpr uint64_t FX_2LOG2E_62 = 0xb8aa3b295c17f0bcull;
// log2(e) at 2^63
constexpr uint64_t FX_LOG2E_63 = 0xb8aa3b295c17f0bcull;
// (ln 2 / 128)^1 / 1! at 2^64
constexpr uint64_t FX_EXP_L1 = 0x162e42fefa39ef3ull;
// (ln 2 / 128)^2 / 2! at 2^64
constexpr uint64_t FX_EXP_L2 = 0xf5fdeffc162cull;
// (ln 2 / 128)^3 / 3! at 2^64
constexpr uint64_t FX_EXP_L3 = 0x71ac235c13ull;
// (ln 2 / 128)^4 / 4! at 2^64
constexpr uint64_t FX_EXP_L4 = 0x276556dfull;
// (ln 2 / 128)^5 / 5! at 2^64
constexpr uint64_t FX_EXP_L5 = 0xaec40ull;
// (ln 2 / 128)^6 / 6! at 2^64
constexpr uint64_t FX_EXP_L6 = 0x286ull;

// cell j of y in [1/2, 1), y in [(128 + j)/256, (129 + j)/256): c = floor(2^23 / (129 + j)) (at
// 2^15, so that y c < 1), ln c at 2^59
FX_TABLE uint64_t FX_LOG_TAB[256] = {
    0xfe03ull, 0x57b98da8535b58dull, 0xfc0full, 0x56bc9f70b3a36b7ull,
    0xfa23ull, 0x55c1d19aec20994ull, 0xf83eull, 0x54c8b09a19a15cdull,
    0xf660ull, 0x53d14a0d6538644ull, 0xf489ull, 0x52dbabbe46cc758ull,
    0xf2b9ull, 0x51e7e39f70aa2fdull, 0xf0f0ull, 0x50f5ffcba48ee89ull,
    0xef2eull, 0x50060e8471a6394ull, 0xed73ull, 0x4f181e30dafad49ull,
    0xebbdull, 0x4e2b275c411a8a9ull, 0xea0eull, 0x4d404ab657f2093ull,
    0xe865ull, 0x4c570a10acd91afull, 0xe6c2ull, 0x4b6f715e9c6cf6dull,
    0xe525ull, 0x4a898cb41ecb0edull, 0xe38eull, 0x49a56844cf6e493ull,
    0xe1fcull, 0x48c27f62e8e2592ull, 0xe070ull, 0x47e16d7f145962cull,
    0xdee9ull, 0x4701ac26ae8719aull, 0xdd67ull, 0x46234503946279dull,
    0xdbebull, 0x4546d6dbbda744dull, 0xda74ull, 0x446bd88f1d2a9e7ull,
    0xd901ull, 0x4391bd181c226daull, 0xd794ull, 0x42b9bb8b3d53e86ull,
    0xd62bull, 0x41e2af14b7ec970ull, 0xd4c7ull, 0x410d38f9c2aaab8ull,
    0xd368ull, 0x40396396c7deac4ull, 0xd20dull, 0x3f669d5ef301083ull,
    0xd0b6ull, 0x3e94eddbe0ae469ull, 0xcf64ull, 0x3dc4faad53e7c26ull,
    0xce16ull, 0x3cf62f879e76d9cull, 0xccccull, 0x3c2894340e4d708ull,
    0xcb87ull, 0x3b5cd19096bb2b3ull, 0xca45ull, 0x3a91ae8da110ca0ull,
    0xc907ull, 0x39c7d32fc1154feull, 0xc7ceull, 0x38ffeb8e8a69924ull,
    0xc698ull, 0x3838b8d27f073b2ull, 0xc565ull, 0x37724036bfc1c96ull,
    0xc437ull, 0x36add5088891121ull, 0xc30cull, 0x35ea32a48d9ba02ull,
    0xc1e4ull, 0x35275e78d9a3a01ull, 0xc0c0ull, 0x3466080409f4c6eull,
    0xbfa0ull, 0x33a637d427da757ull, 0xbe82ull, 0x32e69e85b86cfb2ull,
    0xbd69ull, 0x322945c6b774132ull, 0xbc52ull, 0x316c2f51044be2eull,
    0xbb3eull, 0x30b00cee7a13a52ull, 0xba2eull, 0x2ff594778c2a25eull,
    0xb921ull, 0x2f3c1dd0f155790ull, 0xb817ull, 0x2e83aeed8cf362cull,
    0xb70full, 0x2dcb9acd1b29b67ull, 0xb60bull, 0x2d154c7d26c421dull,
    0xb509ull, 0x2c5f63160d8f3a6ull, 0xb40bull, 0x2bab4dbeaa7a5d5ull,
    0xb30full, 0x2af7a7a77df2ee7ull, 0xb216ull, 0x2a452c0e6847ad6ull,
    0xb11full, 0x2993283bd2e72f0ull, 0xb02cull, 0x28e31384e348361ull,
    0xaf3aull, 0x2832c647454d37cull, 0xae4cull, 0x278474ee5d63053ull,
    0xad60ull, 0x26d6aeed78222d3ull, 0xac76ull, 0x262977c37929adcull,
    0xab8full, 0x257d91f9a0c59d3ull, 0xaaaaull, 0x24d2442229b6fa4ull,
    0xa9c8ull, 0x242852da1131a4full, 0xa8e8ull, 0x237f02c6abd7278ull,
    0xa80aull, 0x22d657973472d39ull, 0xa72full, 0x222f19044fb8f7cull,
    0xa655ull, 0x2187c3ce69b4801ull, 0xa57eull, 0x20e1e4c04e208d1ull,
    0xa4a9ull, 0x203cbbabe84bcd0ull, 0xa3d7ull, 0x1f99146cb373798ull,
    0xa306ull, 0x1ef563e4c79bddaull, 0xa237ull, 0x1e5274ff8a6bc7cull,
    0xa16bull, 0x1db116b0ce983f0ull, 0xa0a0ull, 0x1d0fb7f2255e50bull,
    0x9fd8ull, 0x1c6ff3c6efcf70aull, 0x9f11ull, 0x1bd035382194a1dull,
    0x9e4cull, 0x1b314c570f3e04dull, 0x9d89ull, 0x1a933d3c11d9748ull,
    0x9cc8ull, 0x19f60c068455e55ull, 0x9c09ull, 0x1959bcdc957d2eeull,
    0x9b4cull, 0x18be53eb17ee7c5ull, 0x9a90ull, 0x18230164c1a331cull,
    0x99d7ull, 0x17897085410372cull, 0x991full, 0x16effc8b7386bb6ull,
    0x9868ull, 0x1656a6be1dd2d98ull, 0x97b4ull, 0x15bf206b503db15ull,
    0x9701ull, 0x1527bee49bc48bcull, 0x964full, 0x14908382ac90ddfull,
    0x95a0ull, 0x13fb25a59528caeull, 0x94f2ull, 0x1365f4b01550163ull,
    0x9445ull, 0x12d0f20c56601e0ull, 0x939aull, 0x123cfd2a1531e1eull,
    0x92f1ull, 0x11aa1a7e22d629dull, 0x9249ull, 0x11176e8223e47b3ull,
    0x91a2ull, 0x1084fab53cb5b65ull, 0x90fdull, 0xff3a29c824655cull,
    0x905aull, 0xf636ac17b448d6ull, 0x8fb8ull, 0xed373b1be23508ull,
    0x8f17ull, 0xe43bf00afbc776ull, 0x8e78ull, 0xdb53446cdad8bbull,
    0x8ddaull, 0xd26f120437a139ull, 0x8d3dull, 0xc98f72e286445aull,
    0x8ca2ull, 0xc0c311751adbddull, 0x8c08ull, 0xb7fb984fc60019ull,
    0x8b70ull, 0xaf47d26c2c8e38ull, 0x8ad8ull, 0xa68a8adcc3e718ull,
    0x8a42ull, 0x9de14d31a523a9ull, 0x89aeull, 0x954c652157bcdeull,
    0x891aull, 0x8cae3e81c06308ull, 0x8888ull, 0x8424c5a8f1cd8aull,
    0x87f7ull, 0x7ba136fc87cfaeull, 0x8767ull, 0x7323af310e85c6ull,
    0x86d9ull, 0x6abb7b43eab3f0ull, 0x864bull, 0x624a684e3dca20ull,
    0x85bfull, 0x59ef03caa35d31ull, 0x8534ull, 0x519a3b50b38fa6ull,
    0x84a9ull, 0x493cbcb0063f2eull, 0x8421ull, 0x4104f627991112ull,
    0x8399ull, 0x38c4b5d79f45c1ull, 0x8312ull, 0x308b8a4eb893e3ull,
    0x828cull, 0x285992428f110eull, 0x8208ull, 0x203eacb0e6b084ull,
    0x8184ull, 0x181b889ebf9f2dull, 0x8102ull, 0x100fd57587de71ull,
    0x8080ull, 0x7fc02a8ac42f0ull, 0x8000ull, 0x0ull,
};
// sin and cos of (j + 1/2) pi/128 at 2^63
FX_TABLE uint64_t FX_TRIG_TAB[128] = {
    0x1921d1fcdec7846ull, 0x7ffd885a6e4b6d5eull, 0x4b6195d65157346ull, 0x7fe9cbbffbdd7275ull,
    0x7d95b9e7e0837fbull, 0x7fc2559639c6b502ull, 0xafb68054d520c61ull, 0x7f872bf2f56c2469ull,
    0xe1bc2e3cf616a7bull, 0x7f3857f5b699eb51ull, 0x1139f0cedaf576abull, 0x7ed5e5c6575d048eull,
    0x145576b1293e59dbull, 0x7e5fe49324266a1dull, 0x176dd9de50bf3147ull, 0x7dd6668e8481dd85ull,
    0x1a82a025b004509eull, 0x7d3980ec2cbcb339ull, 0x1d934fe54543115dull, 0x7c894bddd8eb66dfull,
    0x209f701c6ffb5bffull, 0x7bc5e28f91cf0963ull, 0x23a6887e99b67ba3ull, 0x7aef63237c2dd0e3ull,
    0x26a82185c302a362ull, 0x7a05eead33443318ull, 0x29a3c484f1ced449ull, 0x7909a92caf05f9a8ull,
    0x2c98fbba7e4f8c22ull, 0x77fab988b6f8aaafull, 0x2f8752623b99ce03ull, 0x76d94988e2826b29ull,
    0x326e54c77927ae5aull, 0x75a585cf279a2b0cull, 0x354d9056da7f9315ull, 0x745f9dd0f8d76fdeull,
    0x382493b0023dcd3full, 0x7307c3cff3f170f3ull, 0x3af2eeb70dc712abull, 0x719e2cd221ce6c76ull,
    0x3db832a5def1ab11ull, 0x70231099c9552436ull, 0x4073f21d30fadb66ull, 0x6e96a99cd643497full,
    0x4325c13576263a73ull, 0x6cf934fbd55c4615ull, 0x45cd358f7b6d2281ull, 0x6b4af278875442b8ull,
    0x4869e664cfad62c6ull, 0x698c246c0beb870bull, 0x4afb6c97ebcfa7ddull, 0x67bd0fbca6be50d9ull,
    0x4d8162c41967cae0ull, 0x65ddfbd31f5d06ebull, 0x4ffb654d155b5137ull, 0x63ef328fbe5033a5ull,
    0x5269126e6c24e2d8ull, 0x61f1003ee8bafad2ull, 0x54ca0a4a8d56572full, 0x5fe3b38d5c5dc263ull,
    0x571deef994063107ull, 0x5dc79d7c0dc984aeull, 0x59646497c1e0f5c4ull, 0x5b9d1153aaa2ba24ull,
    0x5b9d1153aaa2ba24ull, 0x59646497c1e0f5c4ull, 0x5dc79d7c0dc984aeull, 0x571deef994063107ull,
    0x5fe3b38d5c5dc263ull, 0x54ca0a4a8d56572full, 0x61f1003ee8bafad2ull, 0x5269126e6c24e2d8ull,
    0x63ef328fbe5033a5ull, 0x4ffb654d155b5137ull, 0x65ddfbd31f5d06ebull, 0x4d8162c41967cae0ull,
    0x67bd0fbca6be50d9ull, 0x4afb6c97ebcfa7ddull, 0x698c246c0beb870bull, 0x4869e664cfad62c6ull,
    0x6b4af278875442b8ull, 0x45cd358f7b6d2281ull, 0x6cf934fbd55c4615ull, 0x4325c13576263a73ull,
    0x6e96a99cd643497full, 0x4073f21d30fadb66ull, 0x70231099c9552436ull, 0x3db832a5def1ab11ull,
    0x719e2cd221ce6c76ull, 0x3af2eeb70dc712abull, 0x7307c3cff3f170f3ull, 0x382493b0023dcd3full,
    0x745f9dd0f8d76fdeull, 0x354d9056da7f9315ull, 0x75a585cf279a2b0cull, 0x326e54c77927ae5aull,
    0x76d94988e2826b29ull, 0x2f8752623b99ce03ull, 0x77fab988b6f8aaafull, 0x2c98fbba7e4f8c22ull,
    0x7909a92caf05f9a8ull, 0x29a3c484f1ced449ull, 0x7a05eead33443318ull, 0x26a82185c302a362ull,
    0x7aef63237c2dd0e3ull, 0x23a6887e99b67ba3ull, 0x7bc5e28f91cf0963ull, 0x209f701c6ffb5bffull,
    0x7c894bddd8eb66dfull, 0x1d934fe54543115dull, 0x7d3980ec2cbcb339ull, 0x1a82a025b004509eull,
    0x7dd6668e8481dd85ull, 0x176dd9de50bf3147ull, 0x7e5fe49324266a1dull, 0x145576b1293e59dbull,
    0x7ed5e5c6575d048eull, 0x1139f0cedaf576abull, 0x7f3857f5b699eb51ull, 0xe1bc2e3cf616a7bull,
    0x7f872bf2f56c2469ull, 0xafb68054d520c61ull, 0x7fc2559639c6b502ull, 0x7d95b9e7e0837fbull,
    0x7fe9cbbffbdd7275ull, 0x4b6195d65157346ull, 0x7ffd885a6e4b6d5eull, 0x1921d1fcdec7846ull,
};
// 2^(-j/128) at 2^63
FX_TABLE uint64_t FX_EXP_TAB[128] = {
    0x8000000000000000ull, 0x7f4f08ae3dc7c426ull, 0x7e9f06067a4360baull, 0x7deff6b672f84e24ull,
    0x7d41d96db915019dull, 0x7c94acddaeea5d3aull, 0x7be86fb985689ddcull, 0x7b3d20b6399fc237ull,
    0x7a92be8a92436616ull, 0x79e947ef1d320d2dull, 0x7940bb9e2cffd89dull, 0x78991853d684a285ull,
    0x77f25ccdee6d7ae6ull, 0x774c87cc06d1812eull, 0x76a7980f6cca15c2ull, 0x76038c5b260e5eeeull,
    0x75606373ee921c97ull, 0x74be1c203627c62bull, 0x741cb5281e25ee34ull, 0x737c2d55770fe711ull,
    0x72dc8373be41a454ull, 0x723db6501b9ed447ull, 0x719fc4b95f452d29ull, 0x7102ad7fff41e9b4ull,
    0x70666f76154a7089ull, 0x6fcb096f5c782210ull, 0x6f307a412f074892ull, 0x6e96c0c284192610ull,
    0x6dfddbcbed791babull, 0x6d65ca379564e639ull, 0x6cce8ae13c57ebdbull, 0x6c381ca636d99642ull,
    0x6ba27e656b4eb57aull, 0x6b0daeff4fcde703ull, 0x6a79ad55e7f6fd10ull, 0x69e6784cc2cd61bdull,
    0x69540ec8f895722dull, 0x68c26fb128b4cd63ull, 0x683199ed779592caull, 0x67a18c678c8c8c61ull,
    0x6712460a8fc24072ull, 0x6683c5c3281ee6e9ull, 0x65f60a7f79393e2eull, 0x6569132f21483ba7ull,
    0x64dcdec3371793d1ull, 0x64516c2e47ff1623ull, 0x63c6ba6455dcd8aeull, 0x633cc85ad5122fbdull,
    0x62b39508aa836d6full, 0x622b1f66299a6599ull, 0x61a3666d124bb204ull, 0x611c69188f1eb339ull,
    0x6096266533384a2bull, 0x60109d50f86846d8ull, 0x5f8bccdb3d398841ull, 0x5f07b404c304c9f1ull,
    0x5e8451cfac061b5full, 0x5e01a53f7974fd86ull, 0x5d7fad59099f22feull, 0x5cfe69229605cef5ull,
    0x5c7dd7a3b17dcf75ull, 0x5bfdf7e546520f3eull, 0x5b7ec8f19468bbc9ull, 0x5b0049d42f6afbb6ull,
    0x5a827999fcef3242ull, 0x5a05575132a5cc20ull, 0x5988e20954889245ull, 0x590d18d3330c7f1eull,
    0x5891fac0e95612c8ull, 0x581786e5db7022c2ull, 0x579dbc56b48521baull, 0x57249a29651adc07ull,
    0x56ac1f752150a563ull, 0x56344b525f1ff495ull, 0x55bd1cdad49f699cull, 0x5546932976483b15ull,
    0x54d0ad5a753e077cull, 0x545b6a8b3d990704ull, 0x53e6c9da74b29ab5ull, 0x5372ca67f774358full,
    0x52ff6b54d8a89c75ull, 0x528cabc35f4f799dull, 0x521a8ad704f3404full, 0x51a907b474015dc9ull,
    0x513821818624b40cull, 0x50c7d76542a25b72ull, 0x50582887dcb8a7e1ull, 0x4fe91412b2006e83ull,
    0x4f7a993048d088d7ull, 0x4f0cb70c4ea39210ull, 0x4e9f6cd3967fdba8ull, 0x4e32b9b417619617ull,
    0x4dc69cdceaa72a9cull, 0x4d5b157e4a7fc325ull, 0x4cf022c9905bfd32ull, 0x4c85c3f13360c4d5ull,
    0x4c1bf828c6dc54b8ull, 0x4bb2bea4f8bd5847ull, 0x4b4a169b900c2d00ull, 0x4ae1ff436b663ff7ull,
    0x4a7a77d47f7b84b1ull, 0x4a137f87d58e025bull, 0x49ad159789f37496ull, 0x4947393eca98fcd6ull,
    0x48e1e9b9d588e19bull, 0x487d2645f7725895ull, 0x4818ee218a3358eeull, 0x47b5408bf36472e2ull,
    0x47521cc5a2e6a9e0ull, 0x46ef821011734e6bull, 0x468d6fadbf2dd4f3ull, 0x462be4e23237a6efull,
    0x45cae0f1f545eb73ull, 0x456a632296394492ull, 0x450a6abaa4b77ecdull, 0x44aaf701b0c72feeull,
    0x444c0740496d4294ull, 0x43ed9abffb4c6bc9ull, 0x438fb0cb4f468808ull, 0x433248adc91fdd02ull,
    0x42d561b3e6243d8aull, 0x4278fb2b1bce0d15ull, 0x421d1461d66f2023ull, 0x41c1aca777db771bull,
    0x4166c34c5615d0ecull, 0x410c57a1b9fe12f6ull, 0x40b268f9de0183baull, 0x4058f6a7ecccd5b6ull,
};
