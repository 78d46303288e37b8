// rt_lntab.cuh -- tables of the table-driven logarithm (rt_rng.cuh).
//
// kLn1[i - 64], i = 64..127: for f in [i/128, (i+1)/128) an integer r with f r 2^-15 = 1 - z,
// 0 <= z < 2^-5.9; L = round((ln(r 2^-15) - s ln 2) 2^64) mod 2^64 with s = 1 for i <= 90 (the
// buckets below sqrt(1/2), whose m is 2 f) and 0 above; with r: s, and two flags for the
// side on which the pinned logarithm can lie (below for m < 1, above for m > 1; both in the
// bucket that holds sqrt(1/2)).  kLn2[j], j = floor(z 2^12): t, a multiple of 2^-24 given in 2^-32,
// with (1 - z)(1 + t) = 1 - z', 0 <= z' < 2^-11.9; L = round(ln(1 + t) 2^64).  r and t were
// stepped down from the largest value that keeps z and z' >= 0 until the rounding of L was below
// 1/48 of its last place, so the tables add no error that matters.
#pragma once
#include <cstdint>

namespace rt {

struct __align__(16) Ln1Entry {
  uint64_t L;
  uint32_t r;     // r, at most 2^16
  uint32_t info;  // s | below << 1 | above << 2
};
struct __align__(16) Ln2Entry {
  uint64_t L;
  uint32_t t;  // t 2^32
  uint32_t pad;
};

constexpr int kLn2Size = 65;

__device__ const Ln1Entry kLn1[64] = {
    {0xFBF1D1F5C153B3DEull, 64506u, 5u},
    {0xF7FF4F3B370488D9ull, 63519u, 5u},
    {0xF42B121F05A31F01ull, 62576u, 5u},
    {0xF057E53B3F754810ull, 61648u, 5u},
    {0xECB248235FFFEC2Cull, 60776u, 5u},
    {0xE8EEC367D9208694ull, 59889u, 5u},
    {0xE54B8081612FC211ull, 59044u, 5u},
    {0xE1D6788EB507E4B7ull, 58252u, 5u},
    {0xDDEE981DC7EA6B48ull, 57370u, 5u},
    {0xDACB31DC2B987ADBull, 56671u, 5u},
    {0xD76599266885C32Bull, 55924u, 5u},
    {0xD3B2F30945655FA8ull, 55122u, 5u},
    {0xD0A4BDF319B57396ull, 54468u, 5u},
    {0xCD10BFECDC75C315ull, 53712u, 5u},
    {0xC9D3F03A723C5D21ull, 53037u, 5u},
    {0xC6CC4FADB8C33EB4ull, 52413u, 5u},
    {0xC3956B8CF9DE9B77ull, 51759u, 5u},
    {0xC08DBF254303AAE0ull, 51150u, 5u},
    {0xBD6AA04F7F918250ull, 50527u, 5u},
    {0xBA528CD14C123299ull, 49920u, 5u},
    {0xB74362FABA3FFC79ull, 49327u, 5u},
    {0xB4317978EC11A2C1ull, 48739u, 5u},
    {0xB164EAA8915E1832ull, 48209u, 5u},
    {0xAE7390E406339339ull, 47658u, 5u},
    {0xAB61CCB6125D0D19ull, 47090u, 5u},
    {0xA893EE52643C9C65ull, 46577u, 5u},
    {0xA56CF7752CBA7F30ull, 46007u, 7u},
    {0x547D67C442FCD39Bull, 45581u, 2u},
    {0x51BD6EE3380EB0EFull, 45094u, 2u},
    {0x4F0191BF020CC099ull, 44615u, 2u},
    {0x4C44170C3BEC70E0ull, 44140u, 2u},
    {0x48E7419FDCFA0BA4ull, 43564u, 2u},
    {0x46A60E511EC811F4ull, 43182u, 2u},
    {0x445CAA076710A9F2ull, 42798u, 2u},
    {0x41C3C9809C411A26ull, 42366u, 2u},
    {0x3F16074C05BB3862ull, 41925u, 2u},
    {0x3CA355FBEFF8F83Aull, 41526u, 2u},
    {0x3A1C3FDC06247C7Eull, 41118u, 2u},
    {0x37782B2CBCBA8439ull, 40696u, 2u},
    {0x351CBA3B31E8C113ull, 40323u, 2u},
    {0x32B031AFBBDC4C95ull, 39943u, 2u},
    {0x303221E6248F5F0Eull, 39556u, 2u},
    {0x2D27CEC8BF3C3298ull, 39089u, 2u},
    {0x2B6D6043FFF10120ull, 38826u, 2u},
    {0x28D9749D10C15636ull, 38437u, 2u},
    {0x26CBE9602AA02C5Aull, 38130u, 2u},
    {0x2474C641E9AFFF70ull, 37783u, 2u},
    {0x2220DC9EC4044376ull, 37441u, 2u},
    {0x1FC06A13E50C5CEDull, 37095u, 2u},
    {0x1D46A534DAA9E53Eull, 36738u, 2u},
    {0x1B4DA6E56B2D1E1Aull, 36456u, 2u},
    {0x18EB34326E591680ull, 36118u, 2u},
    {0x166EDD76C35B43C6ull, 35769u, 2u},
    {0x14A6E58DCD35EBDAull, 35521u, 2u},
    {0x129C884959DE3C69ull, 35239u, 2u},
    {0x1044D083F47D7204ull, 34918u, 2u},
    {0x0DFE4903BAD9373Aull, 34609u, 2u},
    {0x0C3A0C85C01AC1BDull, 34371u, 2u},
    {0x0A1671C8A20144D3ull, 34085u, 2u},
    {0x07DAD53E53BE669Cull, 33789u, 2u},
    {0x05C72E46DA889E02ull, 33516u, 2u},
    {0x03F03479111C7498ull, 33276u, 2u},
    {0x01DA4799955BD11Bull, 33006u, 2u},
    {0x0000000000000000ull, 32768u, 2u},
};

__device__ const Ln2Entry kLn2[kLn2Size] = {
    {0x0000000000000000ull, 0x00000000u, 0u},
    {0x000FF980653D17F8ull, 0x000FFA00u, 0u},
    {0x002001FFAAAEAB11ull, 0x00200400u, 0u},
    {0x002FE2853DD2E22Cull, 0x002FE700u, 0u},
    {0x003F941A3B58AD01ull, 0x003F9C00u, 0u},
    {0x00500A7B6B45034Bull, 0x00501700u, 0u},
    {0x00600EF8213FBBE5ull, 0x00602100u, 0u},
    {0x0070167297AC3DC5ull, 0x00702F00u, 0u},
    {0x00800DF3AE08A5DFull, 0x00802E00u, 0u},
    {0x008FFF78B31F07A0ull, 0x00902800u, 0u},
    {0x00A02ED83F18FCD4ull, 0x00A06100u, 0u},
    {0x00AFF07CCDAD98F5ull, 0x00B02D00u, 0u},
    {0x00C046B8D44B2C4Cull, 0x00C08F00u, 0u},
    {0x00D04530C0D3CF55ull, 0x00D09A00u, 0u},
    {0x00E05B931032E530ull, 0x00E0BE00u, 0u},
    {0x00F00656DB75212Eull, 0x00F07700u, 0u},
    {0x0100587C926EC80Dull, 0x0100D900u, 0u},
    {0x01106ADAE9ACBD6Full, 0x0110FC00u, 0u},
    {0x0120A00E86DDAD28ull, 0x01214300u, 0u},
    {0x0130B4618512B9A5ull, 0x01316A00u, 0u},
    {0x0140AED14639CE94ull, 0x01417800u, 0u},
    {0x0150CC128E20E0DAull, 0x0151AA00u, 0u},
    {0x0160A6AAEFBEB6EDull, 0x01619A00u, 0u},
    {0x0171008EBD06BC6Cull, 0x01720B00u, 0u},
    {0x018118C8C563E1F4ull, 0x01823B00u, 0u},
    {0x01912FFFD47D0D9Cull, 0x01926B00u, 0u},
    {0x01A14535AAD0AFA3ull, 0x01A29A00u, 0u},
    {0x01B15E607940FD0Cull, 0x01B2CE00u, 0u},
    {0x01C15AB92C8E98F8ull, 0x01C2E600u, 0u},
    {0x01D19B939112C562ull, 0x01D34400u, 0u},
    {0x01E1B3B0DB256137ull, 0x01E37A00u, 0u},
    {0x01F1C6D2EF2928B7ull, 0x01F3AC00u, 0u},
    {0x0201FEA6B113AE05ull, 0x02040400u, 0u},
    {0x02121EA2ED98873Eull, 0x02144500u, 0u},
    {0x02223C9D56EE4D3Bull, 0x02248500u, 0u},
    {0x02324DAE4CDB3394ull, 0x0234B900u, 0u},
    {0x02428269F3B1FB3Dull, 0x02451200u, 0u},
    {0x025274B7A1E13A47ull, 0x02552900u, 0u},
    {0x0262A56F297627C3ull, 0x02658000u, 0u},
    {0x0272F6CDC47B773Bull, 0x0275F900u, 0u},
    {0x0282C95F9C8A05F0ull, 0x0285F300u, 0u},
    {0x02934836F869EEDDull, 0x02969C00u, 0u},
    {0x02A3513414F4E187ull, 0x02A6CF00u, 0u},
    {0x02B399817C1DD24Cull, 0x02B74300u, 0u},
    {0x02C3A95FD3E48DF0ull, 0x02C77F00u, 0u},
    {0x02D3E7B5473C43D9ull, 0x02D7EB00u, 0u},
    {0x02E3F48FCBEDF0D1ull, 0x02E82600u, 0u},
    {0x02F44B8993CA9FFFull, 0x02F8AD00u, 0u},
    {0x030475FC705E0C1Bull, 0x03090800u, 0u},
    {0x0314AC4239109BAFull, 0x03197000u, 0u},
    {0x0324D1B33D056E32ull, 0x0329C800u, 0u},
    {0x033516B670FE2AB7ull, 0x033A4100u, 0u},
    {0x0345342FC0F4A0B1ull, 0x034A9300u, 0u},
    {0x035581FFD4C2973Eull, 0x035B1700u, 0u},
    {0x0365AF3227D55227ull, 0x036B7B00u, 0u},
    {0x0375F5057E918854ull, 0x037BF900u, 0u},
    {0x03861C391845F3C0ull, 0x038C5900u, 0u},
    {0x03965D07A87B5105ull, 0x039CD400u, 0u},
    {0x03A678543BE28F80ull, 0x03AD2A00u, 0u},
    {0x03B6CFB8DDAE1A0Aull, 0x03BDBE00u, 0u},
    {0x03C71359C6518114ull, 0x03CE3F00u, 0u},
    {0x03D73A5CF828D826ull, 0x03DEA400u, 0u},
    {0x03E74DA4EF8948DCull, 0x03EEF600u, 0u},
    {0x03F7CC3987593712ull, 0x03FFB600u, 0u},
    {0x0407FAFE2374749Aull, 0x04102600u, 0u},
};

// Read-only loads through L1 (the lanes of a warp read different entries).
__device__ __forceinline__ Ln1Entry ln1_entry(uint32_t i) {
  const uint4 v = __ldg((const uint4 *)(kLn1 + i));
  return {((uint64_t)v.y << 32) | v.x, v.z, v.w};
}
__device__ __forceinline__ Ln2Entry ln2_entry(uint32_t j) {
  const uint4 v = __ldg((const uint4 *)(kLn2 + j));
  return {((uint64_t)v.y << 32) | v.x, v.z, v.w};
}

}  // namespace rt
