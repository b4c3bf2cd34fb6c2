// Natural logarithm in 64 bits for the direct sums over scattered points: table
// lookup and a short polynomial (the method of P. T. P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point
// arithmetic", ACM TOMS 16, 1990).  x = 2^e m with m in [1, 2), i the nearest
// of the 129 points 1 + i / 128 to m, c ~ 1 / (1 + i / 128) rounded to 64 bits:
//     log x = e log 2 - log c + log(1 + r),  r = m c - 1, |r| <= 2^-8,
// log 2 and -log c as a part on the grid 2^-42, whose sum with e is exact,
// plus a remainder.  Near x = 1 (i = 0, or i = 128 with e = -1) those terms
// vanish exactly, so small results keep their relative accuracy.  The
// polynomial is the Taylor series of log(1 + r) to r^7 (remainder 2^-67).
//
// A GB300 scheduler takes 64 cycles for a 64-bit warp instruction, so their
// number is the time of a pair: 13 here against ~45 of the general-purpose
// function, whose error (1 ulp) this does not exceed.  The direct sum over
// scattered points takes 2.4 times less with it (direct_general_kernel).  The
// factorization keeps log(): its rank decisions at eps = 1e-9 sit on the last
// bits of the entries (the one-sided and the full proxy matrix of a symmetric
// problem have to decide alike), and its entries are a small part of its time.
#pragma once

namespace hif {

struct LogRow { double c, hi, lo; };

__device__ const LogRow kLogTab[129] = {
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0},
    {0x1.fc07f01fc07f0p-1, 0x1.fe02a6b100000p-8, 0x1.9e63f0dda40e4p-46},
    {0x1.f81f81f81f820p-1, 0x1.fc0a8b0fc0000p-7, 0x1.e1e7cf6d3a69cp-50},
    {0x1.f44659e4a4271p-1, 0x1.7b91b07d60000p-6, -0x1.3b685b602ace4p-44},
    {0x1.f07c1f07c1f08p-1, 0x1.f829b0e780000p-6, 0x1.97c267c7e09e4p-45},
    {0x1.ecc07b301ecc0p-1, 0x1.39e87b9fe8000p-5, 0x1.eb3d480ad9015p-44},
    {0x1.e9131abf0b767p-1, 0x1.77458f6330000p-5, -0x1.1807ce586af09p-44},
    {0x1.e573ac901e574p-1, 0x1.b42dd71198000p-5, -0x1.c8d7ae5d6704cp-46},
    {0x1.e1e1e1e1e1e1ep-1, 0x1.f0a30c0118000p-5, -0x1.d579e83368e91p-45},
    {0x1.de5d6e3f8868ap-1, 0x1.16536eea38000p-4, -0x1.472de768fa309p-46},
    {0x1.dae6076b981dbp-1, 0x1.341d7961bc000p-4, 0x1.1cfb299837610p-44},
    {0x1.d77b654b82c34p-1, 0x1.51b073f060000p-4, 0x1.83ba9278e686ap-44},
    {0x1.d41d41d41d41dp-1, 0x1.6f0d28ae58000p-4, -0x1.4b2241b664613p-44},
    {0x1.d0cb58f6ec074p-1, 0x1.8c345d6318000p-4, 0x1.b22b5acb42a66p-44},
    {0x1.cd85689039b0bp-1, 0x1.a926d3a4ac000p-4, 0x1.561c50bd22a9cp-44},
    {0x1.ca4b3055ee191p-1, 0x1.c5e548f5bc000p-4, 0x1.d0c97585fbe06p-46},
    {0x1.c71c71c71c71cp-1, 0x1.e27076e2b0000p-4, -0x1.a2c2c2af0003cp-45},
    {0x1.c3f8f01c3f8f0p-1, 0x1.fec9131dc0000p-4, -0x1.54455d1ae6607p-44},
    {0x1.c0e070381c0e0p-1, 0x1.0d77e7cd08000p-3, 0x1.cb6cd2ee2f482p-44},
    {0x1.bdd2b899406f7p-1, 0x1.1b72ad52f6000p-3, 0x1.e86041811a396p-45},
    {0x1.bacf914c1bad0p-1, 0x1.29552f8200000p-3, -0x1.5bd67f4471dfcp-44},
    {0x1.b7d6c3dda338bp-1, 0x1.371fc201e8000p-3, 0x1.eea079b2d8abcp-44},
    {0x1.b4e81b4e81b4fp-1, 0x1.44d2b6ccb8000p-3, -0x1.71f416135783cp-46},
    {0x1.b2036406c80d9p-1, 0x1.526e5e3a1c000p-3, -0x1.790aa37fc5238p-44},
    {0x1.af286bca1af28p-1, 0x1.5ff3070a7a000p-3, -0x1.8546f183bebf2p-44},
    {0x1.ac5701ac5701bp-1, 0x1.6d60fe719e000p-3, -0x1.bc91557134767p-44},
    {0x1.a98ef606a63bep-1, 0x1.7ab890210e000p-3, -0x1.be51072534a58p-45},
    {0x1.a6d01a6d01a6dp-1, 0x1.87fa06520c000p-3, 0x1.22130401202fcp-44},
    {0x1.a41a41a41a41ap-1, 0x1.9525a9cf46000p-3, -0x1.294937d9f158fp-44},
    {0x1.a16d3f97a4b02p-1, 0x1.a23bc1fe2c000p-3, -0x1.53d6d91dc9f0bp-44},
    {0x1.9ec8e951033d9p-1, 0x1.af3c94e80c000p-3, -0x1.92e633fcd9066p-52},
    {0x1.9c2d14ee4a102p-1, 0x1.bc286742d8000p-3, 0x1.9a873f39d121cp-44},
    {0x1.999999999999ap-1, 0x1.c8ff7c79aa000p-3, -0x1.7814f689f8434p-45},
    {0x1.970e4f80cb872p-1, 0x1.d5c216b4fc000p-3, -0x1.1b0d1bbca681bp-45},
    {0x1.948b0fcd6e9e0p-1, 0x1.e27076e2b0000p-3, -0x1.a302c2af0003cp-44},
    {0x1.920fb49d0e229p-1, 0x1.ef0adcbdc6000p-3, -0x1.b2a179c86af24p-45},
    {0x1.8f9c18f9c18fap-1, 0x1.fb9186d5e4000p-3, -0x1.d6b2aab993c87p-47},
    {0x1.8d3018d3018d3p-1, 0x1.0402594b4d000p-2, 0x1.037b89ef42d7fp-48},
    {0x1.8acb90f6bf3aap-1, 0x1.0a324e2739000p-2, 0x1.c4dee7ef4030ep-47},
    {0x1.886e5f0abb04ap-1, 0x1.1058bf9ae5000p-2, -0x1.4affd817d52cdp-44},
    {0x1.8618618618618p-1, 0x1.1675cababa000p-2, 0x1.83c0e731f55c4p-44},
    {0x1.83c977ab2beddp-1, 0x1.1c898c169a000p-2, -0x1.81260e5c62affp-44},
    {0x1.8181818181818p-1, 0x1.22941fbcf8000p-2, -0x1.a6876f5eb0963p-44},
    {0x1.7f405fd017f40p-1, 0x1.2895a13de8000p-2, 0x1.a917ad24c13f0p-44},
    {0x1.7d05f417d05f4p-1, 0x1.2e8e2bae12000p-2, -0x1.6791e99b72bd8p-45},
    {0x1.7ad2208e0ecc3p-1, 0x1.347dd9a988000p-2, -0x1.5522dd4c58092p-45},
    {0x1.78a4c8178a4c8p-1, 0x1.3a64c55694000p-2, 0x1.7a81cbcd735d0p-44},
    {0x1.767dce434a9b1p-1, 0x1.404308686a000p-2, 0x1.f8f043049f7d3p-44},
    {0x1.745d1745d1746p-1, 0x1.4618bc21c6000p-2, -0x1.3e02f484c84ccp-46},
    {0x1.724287f46debcp-1, 0x1.4be5f95778000p-2, -0x1.d7c52cd9ad824p-44},
    {0x1.702e05c0b8170p-1, 0x1.51aad872e0000p-2, -0x1.f49d8db0a7cc1p-44},
    {0x1.6e1f76b4337c7p-1, 0x1.5767717456000p-2, -0x1.650fd9524d7cap-44},
    {0x1.6c16c16c16c17p-1, 0x1.5d1bdbf581000p-2, -0x1.8d97dc9c7c238p-44},
    {0x1.6a13cd1537290p-1, 0x1.62c82f2b9c000p-2, 0x1.e57bdbd7c8a98p-44},
    {0x1.6816816816817p-1, 0x1.686c81e9b1000p-2, 0x1.2b5710af84054p-44},
    {0x1.661ec6a5122f9p-1, 0x1.6e08eaa2ba000p-2, 0x1.e390139318d71p-46},
    {0x1.642c8590b2164p-1, 0x1.739d7f6bbd000p-2, 0x1.c7389314feb50p-52},
    {0x1.623fa77016240p-1, 0x1.792a55fdd4000p-2, 0x1.e85f057691feap-44},
    {0x1.6058160581606p-1, 0x1.7eaf83b82b000p-2, -0x1.f05a62d0c25adp-49},
    {0x1.5e75bb8d015e7p-1, 0x1.842d1da1e9000p-2, -0x1.39eab13ae687cp-44},
    {0x1.5c9882b931057p-1, 0x1.89a3386c14000p-2, 0x1.2d92d38c40882p-45},
    {0x1.5ac056b015ac0p-1, 0x1.8f11e87366000p-2, 0x1.643f0bb4eab4cp-45},
    {0x1.58ed2308158edp-1, 0x1.947941c211000p-2, 0x1.bec89337451f4p-44},
    {0x1.571ed3c506b3ap-1, 0x1.99d958117e000p-2, 0x1.1367525dd88f0p-47},
    {0x1.5555555555555p-1, 0x1.9f323ecbfa000p-2, -0x1.ecc3525ca2643p-44},
    {0x1.5390948f40febp-1, 0x1.a484090e5c000p-2, -0x1.3da000d6523c5p-44},
    {0x1.51d07eae2f815p-1, 0x1.a9cec9a9a1000p-2, -0x1.ed86adec02b43p-44},
    {0x1.5015015015015p-1, 0x1.af12932478000p-2, -0x1.e53ab31eed7a9p-44},
    {0x1.4e5e0a72f0539p-1, 0x1.b44f77bcc9000p-2, -0x1.38068224aa2cep-47},
    {0x1.4cab88725af6ep-1, 0x1.b985896931000p-2, 0x1.f9831f629f11ep-47},
    {0x1.4afd6a052bf5bp-1, 0x1.beb4d9da72000p-2, -0x1.21641e78b2151p-44},
    {0x1.49539e3b2d067p-1, 0x1.c3dd7a7cdb000p-2, -0x1.5968261f5a42bp-45},
    {0x1.47ae147ae147bp-1, 0x1.c8ff7c79aa000p-2, -0x1.77acf689f8434p-44},
    {0x1.460cbc7f5cf9ap-1, 0x1.ce1af0b85f000p-2, 0x1.f5e9be95e5568p-45},
    {0x1.446f86562d9fbp-1, 0x1.d32fe7e00f000p-2, -0x1.0ab5884dcd050p-44},
    {0x1.42d6625d51f87p-1, 0x1.d83e7258a3000p-2, -0x1.83c75d48ba26dp-47},
    {0x1.4141414141414p-1, 0x1.dd46a04c1c000p-2, 0x1.283fb989a9274p-44},
    {0x1.3fb013fb013fbp-1, 0x1.e24881a7c7000p-2, -0x1.ecefa1385d356p-45},
    {0x1.3e22cbce4a902p-1, 0x1.e744261d68000p-2, 0x1.e25cdf68dbcf3p-44},
    {0x1.3c995a47babe7p-1, 0x1.ec399d2469000p-2, -0x1.9f865188d6065p-45},
    {0x1.3b13b13b13b14p-1, 0x1.f128f5faf0000p-2, 0x1.baecd720ec44cp-44},
    {0x1.3991c2c187f63p-1, 0x1.f6123fa703000p-2, -0x1.d4baaea4f0d25p-44},
    {0x1.3813813813814p-1, 0x1.faf588f78f000p-2, 0x1.8e9cd7d9f2754p-45},
    {0x1.3698df3de0748p-1, 0x1.ffd2e0857f000p-2, 0x1.25bd65f40d932p-44},
    {0x1.3521cfb2b78c1p-1, 0x1.02552a5a5d000p-1, 0x1.fe3d38d2bafddp-46},
    {0x1.33ae45b57bcb2p-1, 0x1.04bdf9da92800p-1, -0x1.2dce033eff74ep-45},
    {0x1.323e34a2b10bfp-1, 0x1.0723e5c1ce000p-1, -0x1.7e0b50d38edddp-46},
    {0x1.30d190130d190p-1, 0x1.0986f4f573800p-1, -0x1.6f937012b5806p-44},
    {0x1.2f684bda12f68p-1, 0x1.0be72e4252800p-1, 0x1.419b4c4bdd99fp-44},
    {0x1.2e025c04b8097p-1, 0x1.0e44985d1d000p-1, -0x1.ba038a8d10b4bp-44},
    {0x1.2c9fb4d812ca0p-1, 0x1.109f39e2d5000p-1, -0x1.b4c10e09b27a4p-44},
    {0x1.2b404ad012b40p-1, 0x1.12f719593f000p-1, -0x1.0cb3fb7398e0cp-47},
    {0x1.29e4129e4129ep-1, 0x1.154c3d2f4d800p-1, -0x1.0af338662e34dp-44},
    {0x1.288b01288b013p-1, 0x1.179eabbd89800p-1, 0x1.9ff1c60e6fa08p-45},
    {0x1.27350b8812735p-1, 0x1.19ee6b467c800p-1, 0x1.6ee05cbdd7782p-45},
    {0x1.25e22708092f1p-1, 0x1.1c3b81f714000p-1, -0x1.ed90b58389902p-44},
    {0x1.2492492492492p-1, 0x1.1e85f5e704000p-1, 0x1.a17bd8b34be7cp-46},
    {0x1.23456789abcdfp-1, 0x1.20cdcd192a800p-1, 0x1.b6caa81e87baep-44},
    {0x1.21fb78121fb78p-1, 0x1.23130d7bec000p-1, -0x1.7aba4392f1ba7p-46},
    {0x1.20b470c67c0d9p-1, 0x1.2555bce98f800p-1, -0x1.accfde292977ep-48},
    {0x1.1f7047dc11f70p-1, 0x1.2795e1289b000p-1, 0x1.1b6b783f3db97p-45},
    {0x1.1e2ef3b3fb874p-1, 0x1.29d37fec2b000p-1, 0x1.1680b9ad974bap-46},
    {0x1.1cf06ada2811dp-1, 0x1.2c0e9ed449000p-1, -0x1.74628563ce45dp-45},
    {0x1.1bb4a4046ed29p-1, 0x1.2e47436e40000p-1, 0x1.34212a10c3491p-44},
    {0x1.1a7b9611a7b96p-1, 0x1.307d7334f1000p-1, 0x1.7c7f6b2143eadp-46},
    {0x1.19453808ca29cp-1, 0x1.32b1339122000p-1, -0x1.4762fd54a4c27p-44},
    {0x1.1811811811812p-1, 0x1.34e289d9ce000p-1, 0x1.d22eeb92d885dp-45},
    {0x1.16e0689427379p-1, 0x1.37117b5474800p-1, -0x1.29808bf6deec9p-47},
    {0x1.15b1e5f75270dp-1, 0x1.393e0d3562800p-1, 0x1.0cd8e221301b7p-44},
    {0x1.1485f0e0acd3bp-1, 0x1.3b6844a000000p-1, -0x1.ee4738909f3d3p-44},
    {0x1.135c81135c811p-1, 0x1.3d9026a715800p-1, -0x1.04f7fbd9c2f53p-45},
    {0x1.12358e75d3033p-1, 0x1.3fb5b84d17000p-1, -0x1.79bd62c55f46bp-46},
    {0x1.1111111111111p-1, 0x1.41d8fe8467000p-1, 0x1.5742325e617a3p-44},
    {0x1.0fef010fef011p-1, 0x1.43f9fe2f9d000p-1, -0x1.98878d84649f1p-45},
    {0x1.0ecf56be69c90p-1, 0x1.4618bc21c6000p-1, -0x1.3dc2f484c84ccp-45},
    {0x1.0db20a88f4696p-1, 0x1.48353d1ea8800p-1, 0x1.bd5fabd176604p-46},
    {0x1.0c9714fbcda3bp-1, 0x1.4a4f85db04000p-1, -0x1.4575d840b8591p-45},
    {0x1.0b7e6ec259dc8p-1, 0x1.4c679afccf000p-1, -0x1.c71e971322ce8p-45},
    {0x1.0a6810a6810a7p-1, 0x1.4e7d811b75800p-1, 0x1.d7d4584c2b22cp-44},
    {0x1.0953f39010954p-1, 0x1.50913cc016800p-1, 0x1.accf2ce96c2d6p-47},
    {0x1.0842108421084p-1, 0x1.52a2d265bc800p-1, -0x1.2a68c41ba8752p-44},
    {0x1.073260a47f7c6p-1, 0x1.54b2467999800p-1, -0x1.b3c1755eba5e1p-44},
    {0x1.0624dd2f1a9fcp-1, 0x1.56bf9d5b3f000p-1, 0x1.cc888e310b9b2p-44},
    {0x1.05197f7d73404p-1, 0x1.58cadb5cd7800p-1, 0x1.895892f25d931p-45},
    {0x1.0410410410410p-1, 0x1.5ad404c35a000p-1, -0x1.a509acaab41fcp-46},
    {0x1.03091b51f5e1ap-1, 0x1.5cdb1dc6c1800p-1, -0x1.35ae12387451fp-46},
    {0x1.0204081020408p-1, 0x1.5ee02a9241800p-1, -0x1.8a6f29f6a02dcp-45},
    {0x1.0101010101010p-1, 0x1.60e32f4478800p-1, 0x1.b1d4f912b416ap-46},
    {0x1.0000000000000p-1, 0x1.62e42fefa3800p-1, 0x1.ef35793c76730p-45}};

__device__ __forceinline__ double log_tab(double x) {
    const int hi = __double2hiint(x);
    // zero, subnormal, negative, infinite or NaN
    if ((unsigned)hi - 0x00100000u >= 0x7fe00000u) return log(x);
    const int e = (hi >> 20) - 1023, man = hi & 0xfffff;
    const LogRow* t = kLogTab + ((man + 0x1000) >> 13);
    const double c = __ldg(&t->c), lh = __ldg(&t->hi), ll = __ldg(&t->lo);
    const double m = __hiloint2double(man | 0x3ff00000, __double2loint(x));
    const double r = fma(m, c, -1.0), r2 = r * r, de = (double)e;
    double p = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    p = fma(p, r, 0.2);
    p = fma(p, r, -0.25);
    p = fma(p, r, 1.0 / 3.0);
    p = fma(p, r, -0.5);
    const double a = fma(de, 0x1.62e42fefa3800p-1, lh);
    const double b = fma(de, 0x1.ef35793c76730p-45, ll);
    return a + (r + fma(r2, p, b));
}

}  // namespace hif
