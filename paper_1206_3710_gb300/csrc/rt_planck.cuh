// rt_planck.cuh -- the Planck term of the dust emission in 64-bit integer
// arithmetic.
//
// A cell's emission in a bin is mass * C_b / (e^x - 1), x = h nu / (k T),
// C_b = 4 pi kappa dnu 2 h nu^3 / c^2.  Evaluated with expm1 and divisions it
// takes about 58 FP64 operations, and GB300 has two FP64 lanes per SM and
// clock against 128 for 32-bit integers: the emission of 2.8e8 (cell, bin)
// pairs took 26.6 ms, all of it on the FP64 pipe.  Here every step works on
// 64-bit fixed-point numbers (products by 32 x 32 -> 64 multiply-adds):
//   z = x log2 e, 2^-z = 2^-k 2^-f, 2^-f = T_j e^-r with j the leading 9 bits
//   of f (the table-driven exponential of Tang, ACM TOMS 15, 1989, and, for
//   1 - 2^-f at small z, TOMS 18, 1992), e^-r by its Taylor series,
//   1 / (e^x - 1) = 2^-z / (1 - 2^-z), the reciprocal by Newton's iteration.
// Fixed point keeps about 2^-62 (the reciprocal 2^-57 for arguments within
// 2^-57 of a power of two, 2^-59 otherwise), so the error of a term (against 64
// bits and more) is that of its rounded inputs h nu and k T, as before.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define RT_HD __host__ __device__ __forceinline__
#else
#define RT_HD inline
#endif

namespace rtk {

RT_HD uint64_t mul_hi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
// rounded
RT_HD uint32_t mul_hi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b + 0x80000000ull) >> 32); }
RT_HD int clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}
RT_HD uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  return u;
#endif
}
RT_HD double of_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double v;
  __builtin_memcpy(&v, &u, 8);
  return v;
#endif
}

// value = m 2^(e - 63), m in [2^63, 2^64); m = 0: not a positive normal number
struct Norm64 {
  uint64_t m;
  int e;
};
RT_HD Norm64 norm64(double v) {
  const uint64_t b = bits_of(v);
  const uint32_t ex = (uint32_t)(b >> 52);  // sign bit set: above 2046
  Norm64 r;
  r.m = ex - 1u < 2046u ? (0x8000000000000000ull | (b << 11)) : 0ull;
  r.e = (int)ex - 1023;
  return r;
}

// about 2^127 / d for d in [2^63, 2^64): relative error below 2^-59 (2e8 random
// arguments and the neighbours of powers of two: 2^-59.5), for d below 2^63 + 64,
// where the quotient is held at 2^64 - 1, below 2^-57
RT_HD uint64_t recip64(uint64_t d) {
  const uint32_t dh = (uint32_t)(d >> 32), dl = (uint32_t)d;
  // seed to about 2^-21, held below 2^32
#ifdef __CUDA_ARCH__
  const uint32_t y0 = (uint32_t)(__fdividef(1.0f, (float)dh) * 9.223366e18f);
#else
  const uint32_t y0 = (uint32_t)((1.0f / (float)dh) * 9.223366e18f);
#endif
  // 1 - d y0 / 2^95 = e 2^-63, |e| < 2^43; 1 / (1 - e) = 1 + e + e^2
  const uint64_t t = (uint64_t)dh * y0 + (((uint64_t)dl * y0) >> 32);
  const int64_t e = (int64_t)(0x8000000000000000ull - t);
  const int32_t eh = (int32_t)(e >> 21);
  const int64_t es = e + (((int64_t)eh * eh) >> 21);
  const int64_t c = (((es >> 16) * (int64_t)y0) >> 15) + (int64_t)(((es & 0xFFFF) * (uint64_t)y0) >> 31);
  // at d = 2^63 the quotient is 2^64, and the iteration may reach that a
  // little above: held below it
  return d < 0x8000000000000040ull ? ~0ull : ((uint64_t)y0 << 32) + (uint64_t)c;
}

// round((1 - 2^(-j / 512)) 2^64)
#define RT_EXP2_BITS 9
#define RT_EXP2_TABLE (1 << RT_EXP2_BITS)
#ifdef __CUDACC__
static __device__ const uint64_t
#else
static const uint64_t
#endif
    exp2_table[RT_EXP2_TABLE] = {
    0x0000000000000000ull, 0x0058A9ADE372512Eull, 0x00B134A6AEE1375Bull, 0x0109A0F504E75C36ull, 0x0161EEA3847077B4ull,
    0x01BA1DBCC8BA96A3ull, 0x02122E4B695760CBull, 0x026A2059FA2D5EA2ull, 0x02C1F3F30B793E8Bull, 0x0319A92129CF19ACull,
    0x03713FEEDE1BB845ull, 0x03C8B866ADA5D5A9ull, 0x042012931A0F63B7ull, 0x04774E7EA156CDEFull, 0x04CE6C33BDD83C0Cull,
    0x05256BBCE64ED436ull, 0x057C4D248DD5FCC6ull, 0x05D3107523EA9D90ull, 0x0629B5B9146C60CBull, 0x06803CFAC79EF37Full,
    0x06D6A644A22B458Cull, 0x072CF1A10520C93Aull, 0x07831F1A4DF6B264ull, 0x07D92EBAD68D352Dull, 0x082F208CF52EC447ull,
    0x0884F49AFC914ED2ull, 0x08DAAAEF3BD77DC7ull, 0x09304393FE91F0F5ull, 0x0985BE938CC07B92ull, 0x09DB1BF82AD36064ull,
    0x0A305BCC19AC8D70ull, 0x0A857E1996A0D743ull, 0x0ADA82EADB7933D4ull, 0x0B2F6A4A1E73F4E9ull, 0x0B84344192460221ull,
    0x0BD8E0DB661C1282ull, 0x0C2D7021C59BE5A5ull, 0x0C81E21ED8E57C70ull, 0x0CD636DCC4945164ull, 0x0D2A6E65A9C09083ull,
    0x0D7E88C3A6004EC6ull, 0x0DD28600D368C126ull, 0x0E266627488F733Full, 0x0E7A2941188B7D80ull, 0x0ECDCF5852F6BAF7ull,
    0x0F21587703EEFEACull, 0x0F74C4A734174896ull, 0x0FC813F2E898FA1Bull, 0x101B466423250A35ull, 0x106E5C04E1F5391Dull,
    0x10C154DF1FCD4395ull, 0x111430FCD3FC15C3ull, 0x1166F067F25CFDA5ull, 0x11B9932A6B58DD16ull, 0x120C194E2BE75B6Full,
    0x125E82DD1D9016BAull, 0x12B0CFE1266BD47Cull, 0x130300642925B216ull, 0x1355147004FC54BFull, 0x13A70C0E95C3190Full,
    0x13F8E749B3E34224ull, 0x144AA62B345D2861ull, 0x149C48BCE8C967C0ull, 0x14EDCF089F5A0DBCull, 0x153F391822DBC6D1ull,
    0x159086F53AB70B9Cull, 0x15E1B8A9AAF14D85ull, 0x1632CE3F342E230Bull, 0x1683C7BF93B073A9ull, 0x16D4A534835BA348ull,
    0x172566A7B9B4BD55ull, 0x17760C22E9E39F6Cull, 0x17C695AFC3B42398ull, 0x18170357F3974A2Dull, 0x1867552522A46341ull,
    0x18B78B20F69A37B5ull, 0x1907A55511E031DEull, 0x1957A3CB138785BFull, 0x19A7868C974C58E9ull, 0x19F74DA33596E9EAull,
    0x1A46F918837CB758ull, 0x1A9688F612C1A678ull, 0x1AE5FD4571D9297Full, 0x1B3556102BE7656Aull, 0x1B84935FC8C25773ull,
    0x1BD3B53DCCF2FA1Eull, 0x1C22BBB3B9B669E7ull, 0x1C71A6CB0CFF097Full, 0x1CC0768D4175A5AFull, 0x1D0F2B03CE7A98CEull,
    0x1D5DC4382826EDDAull, 0x1DAC4233BF4D8323ull, 0x1DFAA500017C2C97ull, 0x1E48ECA658FCD5ACull, 0x1E9719302CD6A2DDull,
    0x1EE52AA6E0CF12C9ull, 0x1F332113D56B1EEFull, 0x1F80FC8067F05C02ull, 0x1FCEBCF5F26619D9ull, 0x201C627DCB968300ull,
    0x2069ED21470FBBE0ull, 0x20B75CE9B5250188ull, 0x2104B1E062EFC80Eull, 0x2151EC0E9A50D893ull, 0x219F0B7DA1F16EDCull,
    0x21EC1036BD445691ull, 0x2238FA432C870810ull, 0x2285C9AC2CC2C4E6ull, 0x22D27E7AF7CDB3E0ull, 0x231F18B8C44BFCBAull,
    0x236B986EC5B0E36Eull, 0x23B7FDA62C3FE322ull, 0x24044868250DC8ABull, 0x245078BDDA01CCBDull, 0x249C8EB071D6ADABull,
    0x24E88A49101BC8D0ull, 0x25346B90D536338Eull, 0x25803290DE61D3F4ull, 0x25CBDF5245B278FCull, 0x261771DE2214F269ull,
    0x2662EA3D8750284Aull, 0x26AE487986063215ull, 0x26F98C9B2BB56D64ull, 0x2744B6AB82B99454ull, 0x278FC6B3924CD37Cull,
    0x27DABCBC5E88DF90ull, 0x282598CEE8680A96ull, 0x28705AF42DC658C9ull, 0x28BB03352962950Cull, 0x2905919AD2DF650Eull,
    0x2950062E1EC45D02ull, 0x299A60F7FE7F12FFull, 0x29E4A201606431F9ull, 0x2A2EC9532FB08C66ull, 0x2A78D6F6548A2E76ull,
    0x2AC2CAF3B4016FFAull, 0x2B0CA554301205E1ull, 0x2B566620A7A4135Bull, 0x2BA00D61F68D3A9Full, 0x2BE99B20F591AD51ull,
    0x2C330F667A653C87ull, 0x2C7C6A3B57AC6872ull, 0x2CC5ABA85CFD6FACull, 0x2D0ED3B656E15E22ull, 0x2D57E26E0ED51BA6ull,
    0x2DA0D7D84B4A7A1Dull, 0x2DE9B3FDCFA94355ull, 0x2E3276E75C50467Dull, 0x2E7B209DAE96653Aull, 0x2EC3B12980CBA068ull,
    0x2F0C28938A3A2473ull, 0x2F5486E47F275560ull, 0x2F9CCC2510D4DA6Bull, 0x2FE4F85DED81A955ull, 0x302D0B97C06B114Bull,
    0x307505DB31CDC57Aull, 0x30BCE730E6E6E73Full, 0x3104AFA181F50FFFull, 0x314C5F35A2395AA3ull, 0x3193F5F5E3F86CB3ull,
    0x31DB73EAE07B7F1Cull, 0x3222D91D2E116699ull, 0x326A2595600F9BBBull, 0x32B1595C06D3429Bull, 0x32F87479AFC2322Eull,
    0x333F76F6E54BFB43ull, 0x338660DC2EEAEF1Bull, 0x33CD3232112525B1ull, 0x3413EB010D8D83A3ull, 0x345A8B51A2C4BFBFull,
    0x34A1132C4C7A6837ull, 0x34E78299836DE77Aull, 0x352DD9A1BD6F88B2ull, 0x3574184D6D617BECull, 0x35BA3EA50338D9DCull,
    0x36004CB0EBFEA756ull, 0x3646427991D0D85Dull, 0x368C20075BE352E6ull, 0x36D1E562AE80F134ull, 0x37179293EB0C83ECull,
    0x375D27A37001D3BBull, 0x37A2A49998F6A2B4ull, 0x37E8097EBE9BAD4Eull, 0x382D565B36BDAB03ull, 0x38728B3754464EA3ull,
    0x38B7A81B673D4646ull, 0x38FCAD0FBCC93AE2ull, 0x39419A1C9F30CF95ull, 0x39866F4A55DBA087ull, 0x39CB2CA125534181ull,
    0x3A0FD2294F443C27ull, 0x3A545FEB127F0DD2ull, 0x3A98D5EEAAF92523ull, 0x3ADD343C51CDDF2Dull, 0x3B217ADC3D3F8456ull,
    0x3B65A9D6A0B844D0ull, 0x3BA9C133ACCB34CDull, 0x3BEDC0FB8F35484Full, 0x3C31A93672DE4EA3ull, 0x3C7579EC7FD9ED87ull,
    0x3CB93325DB689BF9ull, 0x3CFCD4EAA7F89CAFull, 0x3D405F430526F837ull, 0x3D83D2370FC076C0ull, 0x3DC72DCEE1C2998Dull,
    0x3E0A7212925C9417ull, 0x3E4D9F0A35F044CDull, 0x3E90B4BDDE132D88ull, 0x3ED3B335998F6BAAull, 0x3F169A797464AFD8ull,
    0x3F596A9177C93573ull, 0x3F9C2385AA2AB9AEull, 0x3FDEC55E0F2F7250ull, 0x40215022A7B70421ull, 0x4063C3DB71DB7908ull,
    0x40A6209068F235CBull, 0x40E86649858CEF7Dull, 0x412A950EBD7AA09Aull, 0x416CACE803C87DC8ull, 0x41AEADDD48C2EA4Cull,
    0x41F097F679F66C1Eull, 0x42326B3B82309FB7ull, 0x427427B449812B7Dull, 0x42B5CD68B53AB2E8ull, 0x42F75C60A7F3C941ull,
    0x4338D4A40187E424ull, 0x437A363A9F184D97ull, 0x43BB812C5B0D15DEull, 0x43FCB5810D1604F3ull, 0x443DD3408A2B8BADull,
    0x447EDA72A48FB491ull, 0x44BFCB1F2BCF1454ull, 0x4500A54DECC1BA05ull, 0x45416906B18C1EE7ull, 0x4582165141A015F7ull,
    0x45C2AD3561BDBB1Full, 0x46032DBAD3F46215ull, 0x464397E957A384E9ull, 0x4683EBC8A97BB241ull, 0x46C42960837F7B3Full,
    0x470450B89D046117ull, 0x474461D8AAB3C255ull, 0x47845CC85E8BC7CCull, 0x47C4418F67E05137ull, 0x48041035735BE184ull,
    0x4843C8C22B008AD1ull, 0x48836B3D3628DA17ull, 0x48C2F7AE3988C280ull, 0x49026E1CD72E886Full, 0x4941CE90AE83AC34ull,
    0x498119115C4DD471ull, 0x49C04DA67AAFB82Dull, 0x49FF6C57A12A0894ull, 0x4A3E752C649C5A6Cull, 0x4A7D682C57460F2Eull,
    0x4ABC455F08C73DDCull, 0x4AFB0CCC06219B7Cull, 0x4B39BE7AD9B96345ull, 0x4B785A730B563E80ull, 0x4BB6E0BC20242C13ull,
    0x4BF5515D9AB467BFull, 0x4C33AC5EFAFE510Dull, 0x4C71F1C7BE6051E8ull, 0x4CB0219F5FA0C4F2ull, 0x4CEE3BED56EEDB77ull,
    0x4D2C40B919E38323ull, 0x4D6A300A1B824B5Cull, 0x4DA809E7CC3A4A54ull, 0x4DE5CE5999E701C5ull, 0x4E237D66EFD14361ull,
    0x4E61171736B014F7ull, 0x4E9E9B71D4A99443ull, 0x4EDC0A7E2D53DA70ull, 0x4F196443A1B5DF4Eull, 0x4F56A8C990485C37ull,
    0x4F93D81754F6AEA4ull, 0x4FD0F234491FBA7Cull, 0x500DF727C396CC07ull, 0x504AE6F918A4799Full, 0x5087C1AF9A078509ull,
    0x50C4875296F5BC8Bull, 0x510137E95C1CDBA9ull, 0x513DD37B33A36B9Bull, 0x517A5A0F6529A372ull, 0x51B6CBAD35CA47F2ull,
    0x51F3285BE81B8B1Dull, 0x522F7022BC2FEB6Full, 0x526BA308EF9712D1ull, 0x52A7C115BD5EB53Aull, 0x52E3CA505E136F05ull,
    0x531FBEC007C1A2FCull, 0x535B9E6BEDF65813ull, 0x5397695B41C016D7ull, 0x53D31F9531AFC68Full, 0x540EC120E9D98A17ull,
    0x544A4E0593D59C65ull, 0x5485C64A56C12CC9ull, 0x54C129F6573F3ADAull, 0x54FC7910B779721Full, 0x5537B3A097210568ull,
    0x5572D9AD136F89D7ull, 0x55ADEB3D4727D1A1ull, 0x55E8E8584A96C687ull, 0x5623D105339443FDull, 0x565EA54B1583F108ull,
    0x56996531015619CFull, 0x56D410BE058888E5ull, 0x570EA7F92E276042ull, 0x57492AE984CDF1F7ull, 0x5783999610A79890ull,
    0x57BDF405D6708F2Full, 0x57F83A3FD876C95Full, 0x58326C4B169ACA96ull, 0x586C8A2E8E507D72ull, 0x58A693F13AA00AA5ull,
    0x58E0899A1426AF9Eull, 0x591A6B30111794E2ull, 0x595438BA253CA421ull, 0x598DF23F41F75DF4ull, 0x59C797C65641AF64ull,
    0x5A0129564EAEC716ull, 0x5A3AA6F6156BEA35ull, 0x5A7410AC92414912ull, 0x5AAD6680AA92D37Cull, 0x5AE6A87941610CC7ull,
    0x5B1FD69D3749DF90ull, 0x5B58F0F36A89713Bull, 0x5B91F782B6FAF51Cull, 0x5BCAEA51F6197F62ull, 0x5C03C967FF00D7B4ull,
    0x5C3C94CBA66E4B84ull, 0x5C754C83BEC18020ull, 0x5CADF09717FD446Dull, 0x5CE6810C7FC8626Cull, 0x5D1EFDEAC16E7062ull,
    0x5D576738A5E0A1C7ull, 0x5D8FBCFCF3B697E7ull, 0x5DC7FF3E6F2F323Bull, 0x5E002E03DA315E78ull, 0x5E384953F44CE858ull,
    0x5E7051357ABB491Cull, 0x5EA845AF286076C7ull, 0x5EE026C7B5CBB309ull, 0x5F17F485D93859EEull, 0x5F4FAEF0468EB03Eull,
    0x5F87560DAF64B197ull, 0x5FBEE9E4C2FEDE42ull, 0x5FF66A7C2E5108BBull, 0x602DD7DA9BFF22FAull, 0x60653206B45E0B6Dull,
    0x609C79071D7459AFull, 0x60D3ACE27AFB2AFCull, 0x610ACD9F6E5EEE52ull, 0x6141DB4496C0305Bull, 0x6178D5D890F46701ull,
    0x61AFBD61F786BCC9ull, 0x61E691E762B8DBE0ull, 0x621D536F6883B8E0ull, 0x625402009C985D56ull, 0x628A9DA19060B1FDull,
    0x62C12658D30048AFull, 0x62F79C2CF155261Eull, 0x632DFF2475F88B35ull, 0x63644F45E93FBE42ull, 0x639A8C97D13CD3D3ull,
    0x63D0B720B1BF774Cull, 0x6406CEE70C55B33Full, 0x643CD3F1604CB978ull, 0x6472C6462AB1AAC7ull, 0x64A8A5EBE6525E82ull,
    0x64DE72E90BBE29C3ull, 0x65142D441146A665ull, 0x6549D5036B0079B6ull, 0x657F6A2D8AC41AE6ull, 0x65B4ECC8E02E9936ull,
    0x65EA5CDBD8A261D9ull, 0x661FBA6CDF48059Bull, 0x665505825D0EFE3Cull, 0x668A3E22B8AE7389ull, 0x66BF645456A60031ull,
    0x66F4781D993E7656ull, 0x67297984E08AA3DBull, 0x675E68908A68166Aull, 0x67934546F27FDF3Aull, 0x67C80FAE72475691ull,
    0x67FCC7CD6100DEFDull, 0x68316DAA13BCA855ull, 0x6866014ADD597267ull, 0x689A82B60E854F72ull, 0x68CEF1F1F5BE664Dull,
    0x69034F04DF53B45Dull, 0x693799F51565CF35ull, 0x696BD2C8DFE7A600ull, 0x699FF986849F42A4ull, 0x69D40E3447268AA0ull,
    0x6A0810D868EBFFACull, 0x6A3C017929338011ull, 0x6A6FE01CC51706C0ull, 0x6AA3ACC977876B2Bull, 0x6AD76785794D20D4ull,
    0x6B0B10570108F69Full, 0x6B3EA7444334D5E1ull, 0x6B722C537224812Dull, 0x6BA59F8ABE0652D8ull, 0x6BD900F054E3FB4Aull,
    0x6C0C508A62A33EFBull, 0x6C3F8E5F1106B43Full, 0x6C72BA7487AE80C4ull, 0x6CA5D4D0EC1916D4ull, 0x6CD8DD7A61A3F254ull,
    0x6D0BD477098C5584ull, 0x6D3EB9CD02F00577ull, 0x6D718D826ACE0654ull, 0x6DA44F9D5C07574Cull, 0x6DD70023EF5FAE53ull,
    0x6E099F1C3B7E339Cull, 0x6E3C2C8C54EE3CCAull, 0x6E6EA87A4E2007EBull, 0x6EA112EC3769762Dull, 0x6ED36BE81F06C64Dull,
    0x6F05B374111B4ED5ull, 0x6F37E99617B23807ull, 0x6F6A0E543ABF3595ull, 0x6F9C21B4801F4011ull, 0x6FCE23BCEB994E24ull,
    0x700014737EDF0D7Bull, 0x7031F3DE398D9B7Full, 0x7063C203192E3DC3ull, 0x70957EE819371A3Cull, 0x70C72A93330BEF2Dull,
    0x70F8C50A5DFECAE0ull, 0x712A4E538F50C317ull, 0x715BC674BA32AC40ull, 0x718D2D73CFC5D06Bull, 0x71BE8356BF1CA5FFull,
    0x71EFC823753B862Dull, 0x7220FBDFDD19632Aull, 0x72521E91DFA07E28ull, 0x7283303F63AF1D08ull, 0x72B430EE4E183FDCull,
    0x72E520A481A4561Aull, 0x7315FF67DF11F3A0ull, 0x7346CD3E4516856Bull, 0x73778A2D905F0617ull, 0x73A8363B9B90B222ull,
    0x73D8D16E3F49BBECull, 0x74095BCB5221FF7Bull, 0x7439D558A8ABB5FFull, 0x746A3E1C15742919ull, 0x749A961B690465E8ull,
    0x74CADD5C71E1EFCEull, 0x74FB13E4FC8F7302ull, 0x752B39BAD38D76DCull, 0x755B4EE3BF5B0FE8ull, 0x758B5365867691B9ull,
    0x75BB4745ED5E4081ull, 0x75EB2A8AB6910266ull, 0x761AFD39A28F10A2ull, 0x764ABF586FDAA85Cull, 0x767A70ECDAF8BB4Eull,
    0x76AA11FC9E71A023ull, 0x76D9A28D72D1C2A2ull, 0x770922A50EAA5395ull, 0x773892492691F874ull, 0x7767F17F6D257AD9ull,
    0x7797404D930877AFull, 0x77C67EB946E60E2Cull, 0x77F5ACC835718E84ull, 0x7824CA800967286Eull, 0x7853D7E66B8C9960ull,
    0x7882D50102B1DA94ull, 0x78B1C1D573B1CECFull, 0x78E09E696172EFF0ull, 0x790F6AC26CE7FC3Dull, 0x793E26E63510A378ull,
    0x796CD2DA56FA33B6ull, 0x799B6EA46DC045FCull, 0x79C9FA4A128D6A9Dull, 0x79F875D0DC9BD561ull, 0x7A26E13E6136096Cull,
    0x7A553C9833B784EBull, 0x7A8387E3E58D6C8Aull, 0x7AB1C327063736A3ull, 0x7ADFEE6723475640ull, 0x7B0E09A9C863E5D7ull,
    0x7B3C14F47F4751D0ull, 0x7B6A104CCFC102D0ull, 0x7B97FBB83FB607C4ull, 0x7BC5D73C5321BFBAull, 0x7BF3A2DE8C168375ull,
    0x7C215EA46ABE4ECEull, 0x7C4F0A936D5B69D8ull, 0x7C7CA6B1104911C9ull, 0x7CAA3302CDFC21A6ull, 0x7CD7AF8E1F03BAB9ull,
    0x7D051C587A09ECCDull, 0x7D32796753D45E29ull, 0x7D5FC6C01F44F358ull, 0x7D8D04684D5A76B4ull, 0x7DBA32654D313FB8ull,
    0x7DE750BC8C03DA14ull, 0x7E145F73752BAC90ull, 0x7E415E8F72219FAAull, 0x7E6E4E15EA7EC403ull, 0x7E9B2E0C43FCF88Dull,
    0x7EC7FE77E2779084ull, 0x7EF4BF5E27EBF92Cull, 0x7F2170C4747A5F51ull, 0x7F4E12B026665494ull, 0x7F7AA5269A17747Cull,
    0x7FA7282D2A1A094Full, 0x7FD39BC92F1FB0AFull,
};

// one wavelength bin of the emission
struct PlanckBin {
  Norm64 z;    // h nu / k log2 e
  Norm64 c;    // 4 pi kappa dnu 2 h nu^3 / c^2
};

// log2 e 2^63 and ln 2 2^64
#define RT_LOG2E_64 0xB8AA3B295C17F0BCull
#define RT_LN2_64 0xB17217F7D1CF79ACull

// hnu: h nu (erg); coef: 4 pi kappa dnu 2 h nu^3 / c^2, >= 0
RT_HD PlanckBin planck_bin(double hnu, double coef) {
  PlanckBin B;
  const Norm64 a = norm64(hnu);
  const uint64_t p = mul_hi64(a.m, RT_LOG2E_64);  // in [2^62, 2^64): log2 e = 1.44
  const int s = p >> 63 ? 0 : 1;
  B.z.m = a.m ? p << s : 0ull;
  B.z.e = a.e + 1 - s;
  B.c = norm64(coef);
  return B;
}

// The inverse of k T (erg) for planck_term; m = 0: T outside what it takes.
RT_HD Norm64 planck_inverse(double kT) {
  const Norm64 a = norm64(kT);
  Norm64 r;
  r.m = 0ull;
  r.e = 0;
  if (!a.m) return r;
  const uint64_t y = recip64(a.m);  // 2^127 / m in (2^63, 2^64]
  const bool one = a.m == 0x8000000000000000ull;
  r.m = one ? 0x8000000000000000ull : y;
  r.e = -a.e - (one ? 0 : 1);
  return r;
}

// mass C_b / (e^x - 1).  ok = false where the arguments lie outside the
// fixed-point range (x below 1/370, results near the subnormal range, zero
// or non-finite inputs): the caller then evaluates the term in FP64.
// x >= 709.78 (e^x beyond the double range) gives 0.
RT_HD double planck_term(const PlanckBin& B, Norm64 inv, Norm64 mass, const uint64_t* table, bool& ok) {
  // z = zh 2^(e - 126 + 64), as k + f 2^-64
  const uint64_t zh = mul_hi64(B.z.m, inv.m);
  const int e = B.z.e + inv.e + 2;  // zh 2^(e - 64) = z
  ok = e > -8 && e <= 12 && zh != 0ull && mass.m != 0ull && B.c.m != 0ull;
  if (e > 12 && zh != 0ull && mass.m != 0ull && B.c.m != 0ull) {
    ok = true;  // z >= 2^10
    return 0.0;
  }
  if (!ok) return 0.0;
  const uint32_t k = e > 0 ? (uint32_t)(zh >> (64 - e)) : 0u;
  const uint64_t f = e > 0 ? zh << e : zh >> -e;
  if (k >= 1020u) {  // towards the end of the double range: exactly 0 beyond it
    ok = k >= 1024u;
    return 0.0;
  }
  // 1 - 2^-f = D + T (1 - e^-r), T = 1 - D
  const uint64_t D = table[f >> (64 - RT_EXP2_BITS)];
  const uint64_t R = mul_hi64(f << RT_EXP2_BITS, RT_LN2_64);  // r 2^73, r < ln 2 / 512
  const uint64_t R2 = mul_hi64(R, R);                         // r^2 2^82
  // 1 - e^-r = r - r^2 / 2 (1 - r/3 (1 - r/4 (1 - r/5 (1 - r/6)))): the
  // inner factors at 2^41
  const uint32_t r = (uint32_t)(R >> 32);
  uint32_t w = mul_hi32(r, 715827883u);                                  // r/6
  w = mul_hi32(r - (uint32_t)(((uint64_t)r * w) >> 41), 858993459u);     // r/5 (1 - w)
  w = mul_hi32(r - (uint32_t)(((uint64_t)r * w) >> 41), 1073741824u);    // r/4 (1 - w)
  w = mul_hi32(r - (uint32_t)(((uint64_t)r * w) >> 41), 1431655765u);    // r/3 (1 - w)
  const uint64_t S = R2 - (((R2 >> 32) * (uint64_t)w) >> 9);             // r^2 (1 - w) 2^82
  const uint64_t E = R - (S >> 10);                                      // (1 - e^-r) 2^73
  uint64_t v = D + (mul_hi64(~D, E) >> 9);                               // (1 - 2^-f) 2^64
  v = v ? v : 1ull;
  const uint64_t mu = 0ull - v;                                          // 2^-f 2^64
  uint64_t u = k < 64u ? mu >> k : 0ull;
  u = u ? u : 1ull;
  const uint64_t d = 0ull - u;                                           // (1 - 2^-z) 2^64
  const int lz = clz64(d);
  const uint64_t q = mul_hi64(mu, recip64(d << lz));                     // mu / (d 2^lz) 2^63
  // mass C_b q 2^(lz - 63 - k)
  const uint64_t mc = mul_hi64(mass.m, B.c.m);                           // 2^126 -> 2^62 units
  const uint64_t p = mul_hi64(mc, q);
  const int lp = clz64(p);
  // value = p 2^x: mass.m 2^(em-63) c.m 2^(ec-63) q 2^(lz-63-k), two 64-bit shifts in between
  const int ex = mass.e + B.c.e + lz - (int)k - 63 * 3 + 128;
  const uint64_t pn = p << lp;                                           // [2^63, 2^64)
  const int eb = ex - lp + 63 + 1023;                                    // biased exponent of 2^63 units
  if (eb < 2 || eb > 2045) {
    ok = false;
    return 0.0;
  }
  // round to 53 bits (a carry moves into the exponent)
  return of_bits(((uint64_t)(eb - 1) << 52) + ((pn >> 11) + ((pn >> 10) & 1ull)));
}

}  // namespace rtk
