// log64.cuh -- ln x in FP64 for the kernels that the FP64 pipe bounds.
//
// The pipe takes one warp instruction per 64 cycles and SM quarter, and log() spends 29 of them
// on a site that needs about 150 for the whole step.  This one spends 13, by the table method
// (P. T. P. Tang, "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990): x = 2^k m with m in [0.69, 1.38), c_j near the
// middle of the one of 128 intervals that m lies in, ln x = k ln 2 + ln c_j + ln(1 + r) with
// r = m / c_j - 1, |r| <= 2^-8, and the Taylor polynomial of degree 7.  ln 2 and ln c_j are held
// as a multiple of 2^-43, whose combination is exact, and the rest.  The interval around 1 has
// c = 1, so that ln x keeps its relative accuracy there.  Measured against 113-bit logarithms on
// 4e6 values each: at most 1.2 units in the last place (log() 0.55) and 0.25 on average as log(),
// and the same largest absolute error to 8 %.
#pragma once

#include <cuda_runtime.h>

namespace mclb {

constexpr int LOG64_ROWS = 128;
constexpr int LOG64_OFF = 0x3FE61000;   // high word where the first interval begins

struct Log64Row {
    double inv, hi, lo;
};

// Interval j is the doubles whose high words start at LOG64_OFF + j 2^13.  inv: the rounded
// reciprocal of its middle (1 where it holds 1); hi + lo = -ln inv, hi a multiple of 2^-43.
static __device__ const Log64Row log64_rows[LOG64_ROWS] = {
    {0x1.724287f46debcp+0, -0x1.79e26687cf800p-2, -0x1.9ebfd2efd1778p-45},
    {0x1.702e05c0b8170p+0, -0x1.741d876c67800p-2, -0x1.d870949dc60b3p-45},
    {0x1.6e1f76b4337c7p+0, -0x1.6e60ee6af1800p-2, -0x1.72aa57c222d87p-46},
    {0x1.6c16c16c16c17p+0, -0x1.68ac83e9c6800p-2, -0x1.0a6532756eba0p-45},
    {0x1.6a13cd1537290p+0, -0x1.630030b3ab000p-2, 0x1.dbc23e731ae00p-45},
    {0x1.6816816816817p+0, -0x1.5d5bddf596000p-2, 0x1.9de2a08a465dcp-47},
    {0x1.661ec6a5122f9p+0, -0x1.57bf753c8d000p-2, -0x1.fadadee5d40efp-46},
    {0x1.642c8590b2164p+0, -0x1.522ae0738a000p-2, -0x1.eba708164c759p-45},
    {0x1.623fa77016240p+0, -0x1.4c9e09e173000p-2, 0x1.e18891b0ad8a4p-45},
    {0x1.6058160581606p+0, -0x1.4718dc271c800p-2, 0x1.f1c4e0967d675p-45},
    {0x1.5e75bb8d015e7p+0, -0x1.419b423d5e800p-2, -0x1.8c2b6ec90e09dp-47},
    {0x1.5c9882b931057p+0, -0x1.3c25277333000p-2, -0x1.83454b606bd5cp-46},
    {0x1.5ac056b015ac0p+0, -0x1.36b6776be1000p-2, -0x1.15ecdb0f177c8p-46},
    {0x1.58ed2308158edp+0, -0x1.314f1e1d36000p-2, 0x1.8e5bad3213cb8p-45},
    {0x1.571ed3c506b3ap+0, -0x1.2bef07cdc9000p-2, -0x1.aa5ba4a5004f4p-45},
    {0x1.5555555555555p+0, -0x1.269621134d800p-2, -0x1.c8bc1df5bb3b6p-45},
    {0x1.5390948f40febp+0, -0x1.214456d0eb800p-2, -0x1.a9d5eba46baeap-47},
    {0x1.51d07eae2f815p+0, -0x1.1bf99635a6800p-2, -0x1.ca42d5147bdb7p-45},
    {0x1.5015015015015p+0, -0x1.16b5ccbacf800p-2, -0x1.b9aadf7a51681p-45},
    {0x1.4e5e0a72f0539p+0, -0x1.1178e8227e800p-2, 0x1.c2c8e63a5f01cp-45},
    {0x1.4cab88725af6ep+0, -0x1.0c42d67616000p-2, -0x1.70d4b163ceae9p-45},
    {0x1.4afd6a052bf5bp+0, -0x1.07138604d5800p-2, -0x1.8fedb16ed4e91p-48},
    {0x1.49539e3b2d067p+0, -0x1.01eae5626c800p-2, 0x1.6ec4c1485e94ap-46},
    {0x1.47ae147ae147bp+0, -0x1.f991c6cb3b000p-3, -0x1.bd1ecca0cdf30p-46},
    {0x1.460cbc7f5cf9ap+0, -0x1.ef5ade4dd0000p-3, 0x1.ad11565bb8e11p-51},
    {0x1.446f86562d9fbp+0, -0x1.e530effe71000p-3, -0x1.282276041f430p-51},
    {0x1.42d6625d51f87p+0, -0x1.db13db0d49000p-3, 0x1.afd8af715b035p-45},
    {0x1.4141414141414p+0, -0x1.d1037f2656000p-3, 0x1.8527e75b6f6e4p-47},
    {0x1.3fb013fb013fbp+0, -0x1.c6ffbc6f01000p-3, 0x1.1ed72c5962bd2p-48},
    {0x1.3e22cbce4a902p+0, -0x1.bd087383be000p-3, 0x1.d5844595412b6p-45},
    {0x1.3c995a47babe7p+0, -0x1.b31d8575bd000p-3, 0x1.c510d4eace1aap-47},
    {0x1.3b13b13b13b14p+0, -0x1.a93ed3c8ae000p-3, 0x1.86a4350562169p-45},
    {0x1.3991c2c187f63p+0, -0x1.9f6c407089000p-3, -0x1.98aad6865817ap-45},
    {0x1.3813813813814p+0, -0x1.95a5adcf70000p-3, -0x1.8262858a0ff6fp-47},
    {0x1.3698df3de0748p+0, -0x1.8beafeb390000p-3, 0x1.71154aae92cd1p-47},
    {0x1.3521cfb2b78c1p+0, -0x1.823c16551a000p-3, -0x1.e02db9a631e83p-46},
    {0x1.33ae45b57bcb2p+0, -0x1.7898d85445000p-3, 0x1.c5f9070914305p-46},
    {0x1.323e34a2b10bfp+0, -0x1.6f0128b757000p-3, 0x1.51c4de59c21e1p-45},
    {0x1.30d190130d190p+0, -0x1.6574ebe8c1000p-3, -0x1.9cb8b2c3c2e78p-46},
    {0x1.2f684bda12f68p+0, -0x1.5bf406b544000p-3, 0x1.28023eb68981cp-46},
    {0x1.2e025c04b8097p+0, -0x1.527e5e4a1b000p-3, -0x1.633c8e5697dc7p-45},
    {0x1.2c9fb4d812ca0p+0, -0x1.4913d8333b000p-3, -0x1.58b7954fdb678p-45},
    {0x1.2b404ad012b40p+0, -0x1.3fb45a5993000p-3, 0x1.cd9d87e6a354dp-45},
    {0x1.29e4129e4129ep+0, -0x1.365fcb0159000p-3, -0x1.46fa8234b7289p-51},
    {0x1.288b01288b013p+0, -0x1.2d1610c868000p-3, -0x1.3d0eccb81b4a1p-47},
    {0x1.27350b8812735p+0, -0x1.23d712a49c000p-3, -0x1.00aa38fd3df5cp-46},
    {0x1.25e22708092f1p+0, -0x1.1aa2b7e23f000p-3, -0x1.ca56e44389934p-45},
    {0x1.2492492492492p+0, -0x1.1178e8227e000p-3, -0x1.1e778ce2d07f2p-45},
    {0x1.23456789abcdfp+0, -0x1.08598b59e4000p-3, 0x1.7e5fd7009902cp-45},
    {0x1.21fb78121fb78p+0, -0x1.fe89139dbe000p-4, 0x1.536d64fa10afdp-45},
    {0x1.20b470c67c0d9p+0, -0x1.ec739830a2000p-4, 0x1.db308afe645e0p-45},
    {0x1.1f7047dc11f70p+0, -0x1.da72763844000p-4, -0x1.a79401fa71733p-46},
    {0x1.1e2ef3b3fb874p+0, -0x1.c885801bc4000p-4, -0x1.63f51c65aacd3p-45},
    {0x1.1cf06ada2811dp+0, -0x1.b6ac88dad6000p-4, 0x1.38d002bf768e5p-46},
    {0x1.1bb4a4046ed29p+0, -0x1.a4e7640b1c000p-4, 0x1.e4336b94407c8p-47},
    {0x1.1a7b9611a7b96p+0, -0x1.9335e5d594000p-4, -0x1.30f5c3abd47dap-45},
    {0x1.19453808ca29cp+0, -0x1.8197e2f40e000p-4, -0x1.f7edcf96ffdf7p-47},
    {0x1.1811811811812p+0, -0x1.700d30aeac000p-4, -0x1.d068da99ded32p-49},
    {0x1.16e0689427379p+0, -0x1.5e95a4d97a000p-4, 0x1.c66a63c5d1d1ep-45},
    {0x1.15b1e5f75270dp+0, -0x1.4d3115d208000p-4, 0x1.53e2582f4e1efp-48},
    {0x1.1485f0e0acd3bp+0, -0x1.3bdf5a7d1e000p-4, -0x1.cbc3ea5db4ed7p-45},
    {0x1.135c81135c811p+0, -0x1.2aa04a4472000p-4, 0x1.0bd28ae9c697dp-45},
    {0x1.12358e75d3033p+0, -0x1.1973bd1466000p-4, 0x1.53ebd560d9e9bp-45},
    {0x1.1111111111111p+0, -0x1.08598b59e4000p-4, 0x1.7e9dd7009902cp-46},
    {0x1.0fef010fef011p+0, -0x1.eea31c006c000p-5, 0x1.e10be4fc93b7bp-47},
    {0x1.0ecf56be69c90p+0, -0x1.ccb73cdddc000p-5, 0x1.a60f247d82807p-46},
    {0x1.0db20a88f4696p+0, -0x1.aaef2d0fb0000p-5, -0x1.1085a353bb42ep-45},
    {0x1.0c9714fbcda3bp+0, -0x1.894aa149fc000p-5, 0x1.96a95d05a267dp-46},
    {0x1.0b7e6ec259dc8p+0, -0x1.67c94f2d4c000p-5, 0x1.26afbec19afa2p-47},
    {0x1.0a6810a6810a7p+0, -0x1.466aed42e0000p-5, 0x1.c073375bdfd28p-45},
    {0x1.0953f39010954p+0, -0x1.252f32f8d0000p-5, -0x1.8401ae021b67bp-45},
    {0x1.0842108421084p+0, -0x1.0415d89e74000p-5, -0x1.101c05cf1d753p-47},
    {0x1.073260a47f7c6p+0, -0x1.c63d2ec148000p-6, -0x1.56b863f9eb2f3p-45},
    {0x1.0624dd2f1a9fcp+0, -0x1.8492528c90000p-6, 0x1.a9dba325a0c34p-45},
    {0x1.05197f7d73404p+0, -0x1.432a925980000p-6, -0x1.97739928637fep-47},
    {0x1.0410410410410p+0, -0x1.0205658938000p-6, 0x1.3e45b06e2f7d2p-45},
    {0x1.03091b51f5e1ap+0, -0x1.82448a3890000p-7, 0x1.75f37da74f640p-45},
    {0x1.0204081020408p+0, -0x1.0101575890000p-7, 0x1.0cb6b999d2be8p-46},
    {0x1.0101010101010p+0, -0x1.0080559580000p-8, -0x1.164afcb31c67bp-45},
    {0x1.0000000000000p+0, 0x0.0p+0, 0x0.0p+0},
    {0x1.fc07f01fc07f0p-1, 0x1.fe02a6b100000p-8, 0x1.9e63f0dda40e4p-46},
    {0x1.f81f81f81f820p-1, 0x1.fc0a8b0fc0000p-7, 0x1.e1e7cf6d3a69cp-50},
    {0x1.f44659e4a4271p-1, 0x1.7b91b07d58000p-6, 0x1.892f493faa639p-45},
    {0x1.f07c1f07c1f08p-1, 0x1.f829b0e780000p-6, 0x1.97c267c7e09e4p-45},
    {0x1.ecc07b301ecc0p-1, 0x1.39e87b9fec000p-5, -0x1.4c2b7f526feaap-48},
    {0x1.e9131abf0b767p-1, 0x1.77458f632c000p-5, 0x1.cff0634f2a1eep-45},
    {0x1.e573ac901e574p-1, 0x1.b42dd71198000p-5, -0x1.c8d7ae5d6704cp-46},
    {0x1.e1e1e1e1e1e1ep-1, 0x1.f0a30c0118000p-5, -0x1.d579e83368e91p-45},
    {0x1.de5d6e3f8868ap-1, 0x1.16536eea38000p-4, -0x1.472de768fa309p-46},
    {0x1.dae6076b981dbp-1, 0x1.341d7961be000p-4, -0x1.c609accf913dfp-45},
    {0x1.d77b654b82c34p-1, 0x1.51b073f062000p-4, -0x1.f115b61c65e57p-46},
    {0x1.d41d41d41d41dp-1, 0x1.6f0d28ae56000p-4, 0x1.69bb7c93373dap-45},
    {0x1.d0cb58f6ec074p-1, 0x1.8c345d631a000p-4, -0x1.375294d2f5668p-46},
    {0x1.cd85689039b0bp-1, 0x1.a926d3a4ae000p-4, -0x1.53c75e85baac8p-45},
    {0x1.ca4b3055ee191p-1, 0x1.c5e548f5bc000p-4, 0x1.d0c97585fbe06p-46},
    {0x1.c71c71c71c71cp-1, 0x1.e27076e2b0000p-4, -0x1.a2c2c2af0003cp-45},
    {0x1.c3f8f01c3f8f0p-1, 0x1.fec9131dbe000p-4, 0x1.577545ca333f2p-45},
    {0x1.c0e070381c0e0p-1, 0x1.0d77e7cd09000p-3, -0x1.a499688e85bf4p-47},
    {0x1.bdd2b899406f7p-1, 0x1.1b72ad52f6000p-3, 0x1.e86041811a396p-45},
    {0x1.bacf914c1bad0p-1, 0x1.29552f81ff000p-3, 0x1.485301771c408p-45},
    {0x1.b7d6c3dda338bp-1, 0x1.371fc201e9000p-3, -0x1.15f864d27543ap-48},
    {0x1.b4e81b4e81b4fp-1, 0x1.44d2b6ccb8000p-3, -0x1.71f416135783cp-46},
    {0x1.b2036406c80d9p-1, 0x1.526e5e3a1b000p-3, 0x1.0deab90075b8fp-45},
    {0x1.af286bca1af28p-1, 0x1.5ff3070a79000p-3, 0x1.eae439f105039p-46},
    {0x1.ac5701ac5701bp-1, 0x1.6d60fe719d000p-3, 0x1.0dbaaa3b2e266p-46},
    {0x1.a98ef606a63bep-1, 0x1.7ab890210e000p-3, -0x1.be51072534a58p-45},
    {0x1.a6d01a6d01a6dp-1, 0x1.87fa06520d000p-3, -0x1.bbd9f7fdbfa09p-45},
    {0x1.a41a41a41a41ap-1, 0x1.9525a9cf45000p-3, 0x1.ad6d904c1d4e3p-45},
    {0x1.a16d3f97a4b02p-1, 0x1.a23bc1fe2b000p-3, 0x1.58524dc46c1eap-45},
    {0x1.9ec8e951033d9p-1, 0x1.af3c94e80c000p-3, -0x1.92e633fcd9066p-52},
    {0x1.9c2d14ee4a102p-1, 0x1.bc286742d9000p-3, -0x1.95e30318bb78fp-46},
    {0x1.999999999999ap-1, 0x1.c8ff7c79aa000p-3, -0x1.7814f689f8434p-45},
    {0x1.970e4f80cb872p-1, 0x1.d5c216b4fc000p-3, -0x1.1b0d1bbca681bp-45},
    {0x1.948b0fcd6e9e0p-1, 0x1.e27076e2af000p-3, 0x1.73f4f543fff10p-46},
    {0x1.920fb49d0e229p-1, 0x1.ef0adcbdc6000p-3, -0x1.b2a179c86af24p-45},
    {0x1.8f9c18f9c18fap-1, 0x1.fb9186d5e4000p-3, -0x1.d6b2aab993c87p-47},
    {0x1.8d3018d3018d3p-1, 0x1.0402594b4d000p-2, 0x1.037b89ef42d7fp-48},
    {0x1.8acb90f6bf3aap-1, 0x1.0a324e2739000p-2, 0x1.c4dee7ef4030ep-47},
    {0x1.886e5f0abb04ap-1, 0x1.1058bf9ae4800p-2, 0x1.6a004fd055a66p-45},
    {0x1.8618618618618p-1, 0x1.1675cababa800p-2, -0x1.f0fc63382a8f0p-46},
    {0x1.83c977ab2beddp-1, 0x1.1c898c1699800p-2, 0x1.fb67c68e75404p-46},
    {0x1.8181818181818p-1, 0x1.22941fbcf7800p-2, 0x1.65e242853da76p-46},
    {0x1.7f405fd017f40p-1, 0x1.2895a13de8800p-2, -0x1.5ba14b6cfb03fp-46},
    {0x1.7d05f417d05f4p-1, 0x1.2e8e2bae12000p-2, -0x1.6791e99b72bd8p-45},
    {0x1.7ad2208e0ecc3p-1, 0x1.347dd9a988000p-2, -0x1.5522dd4c58092p-45},
    {0x1.78a4c8178a4c8p-1, 0x1.3a64c55694800p-2, -0x1.0afc686519460p-45},
    {0x1.767dce434a9b1p-1, 0x1.404308686a800p-2, -0x1.c3ef3ed820b3ap-50},
    {0x1.745d1745d1746p-1, 0x1.4618bc21c6000p-2, -0x1.3e02f484c84ccp-46},
};

// ln x with the rows at tab (in shared memory).  Zero, negative, subnormal, infinite and NaN
// arguments take log().
__device__ __forceinline__ double log64(double x, const Log64Row* tab)
{
    const int hi = __double2hiint(x);
    if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);
    const int d = hi - LOG64_OFF, k = d >> 20;
    const Log64Row t = tab[(d >> 13) & (LOG64_ROWS - 1)];
    const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
    const double r = fma(m, t.inv, -1.0);
    double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    q = fma(r, q, 1.0 / 5.0);
    q = fma(r, q, -1.0 / 4.0);
    q = fma(r, q, 1.0 / 3.0);
    q = fma(r, q, -1.0 / 2.0);
    // k as a double without a conversion: 2^52 + 2^31 + k, less 2^52 + 2^31
    const double kd = __hiloint2double(0x43300000, k ^ (int)0x80000000) -
                      __hiloint2double(0x43300000, (int)0x80000000);
    // ln 2 to 2^-43, and the rest
    return fma(kd, 0x1.62e42fefa3800p-1, t.hi) + (fma(r * r, q, r) + fma(kd, 0x1.ef35793c76730p-45, t.lo));
}

// The rows into shared memory, by all threads of the CTA; a barrier has to follow.
__device__ __forceinline__ void log64_load(Log64Row* tab)
{
    double* d = &tab[0].inv;
    const double* g = &log64_rows[0].inv;
    for (int k = threadIdx.x; k < 3 * LOG64_ROWS; k += blockDim.x) d[k] = __ldg(g + k);
}

}  // namespace mclb
