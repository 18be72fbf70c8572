// normals_f64.cuh -- the FP64 Box-Muller pair of two Philox words, in 64-bit fixed point.
//
// The FP64 lattice and graph steps are bound by the SMs' FP64 units (a warp's FP64 operation occupies them for
// 16 or more cycles, an integer one a quarter of a cycle), and the logarithm, square root, sine and cosine in
// FP64 took most of a site-update's.  The arguments are integers of 33 and 31 bits and all
// intermediate values lie in known ranges, so the whole pair needs no floating-point operation: products
// of 64-bit fractions, every value with a relative error below 2^-57, one rounding to a double at the
// end (measured over 6 million normals: at most 0.56 units in the last place, rms 0.289; with the FP64
// library functions 2.96 and 0.579).
//   48^3 volume, two chains: 80 -> 47 us per sweep.
//
//   log      table-driven (Tang, ACM TOMS 16 (1990) 378): u = m 2^-e, c ~ 1/m of 12 bits from the first seven bits of
//            m, 1 - m c = g in (0, 2^-6.9) exact; -2 ln u = 2 (e ln 2 + ln c) - 2 ln(1 - g), the last by its series.
//            For u near 1, c is 1/2, e is 1 and the table's value 0: g = 1 - u, and the product with
//            the series keeps its relative precision.
//   sqrt     a single-precision reciprocal square root and one third-order step.
//   sin, cos their Taylor series over a quarter turn centred at 0 (as in single precision), by Horner's
//            rule; the leading coefficients, which are small, in 32 bits.
#pragma once

#include <cstdint>

namespace gmrf {

struct alignas(16) LogEntry {
    uint64_t t;  // 2 (ln 2 + ln c), 63 fraction bits
    uint32_t c;  // 12 fraction bits: floor(4096 / (1 + (i + 1) / 128))
    uint32_t pad;
};

static __device__ const LogEntry kLogTable[128] = {
    {0xAF70154920B3AB87ull, 4064u, 0}, {0xAD6A0261ACF967D9ull, 4032u, 0}, {0xAB8091309457C190ull, 4002u, 0},
    {0xA982F0CB0FCA5916ull, 3971u, 0}, {0xA7A2941ACA70C882ull, 3942u, 0}, {0xA5ADEB4AB7139C6Full, 3912u, 0},
    {0xA3C6490971A24D24ull, 3883u, 0}, {0xA1EBFF97491DD125ull, 3855u, 0}, {0x9FFD208D213E08A9ull, 3826u, 0},
    {0x9E2D005C6DF237A8ull, 3799u, 0}, {0x9C48304A256DEE9Bull, 3771u, 0}, {0x9A7144ECE70E98B7ull, 3744u, 0},
    {0x98A8920E17E2F5E3ull, 3718u, 0}, {0x96DCAAB906F11632ull, 3692u, 0}, {0x950D8354EDB6D3C3ull, 3666u, 0},
    {0x933B1009A186FE69ull, 3640u, 0}, {0x917766623039354Bull, 3615u, 0}, {0x8FC2DAFE28B2C589ull, 3591u, 0},
    {0x8DF90213A96212F9ull, 3566u, 0}, {0x8C3E71DF10F22CABull, 3542u, 0}, {0x8A80DF5FC9A90C6Full, 3518u, 0},
    {0x88D30112F2B18308ull, 3495u, 0}, {0x87224C2E8E645FB7ull, 3472u, 0}, {0x856EB70A027E26D4ull, 3449u, 0},
    {0x83B837CB12C89452ull, 3426u, 0}, {0x821205CB2F2A610Cull, 3404u, 0}, {0x806916FE07085BB8ull, 3382u, 0},
    {0x7EBD623DE3CC7B67ull, 3360u, 0}, {0x7D227F9709B1E462ull, 3339u, 0}, {0x7B85054BB0181DC0ull, 3318u, 0},
    {0x79E4EAEE7402FE41ull, 3297u, 0}, {0x784227E89745A0FBull, 3276u, 0}, {0x76B0D4F8B165508Cull, 3256u, 0},
    {0x751D0902FB77562Aull, 3236u, 0}, {0x7386BC2E17CFADEEull, 3216u, 0}, {0x71EDE67B0DBABE07ull, 3196u, 0},
    {0x7067216F2B1A291Aull, 3177u, 0}, {0x6EDE0451E2FF4917ull, 3158u, 0}, {0x6D5287E52591753Eull, 3139u, 0},
    {0x6BC4A4C91DE1AC45ull, 3120u, 0}, {0x6A4974DEA3162AEAull, 3102u, 0}, {0x68CC100813E98DCDull, 3084u, 0},
    {0x674C6FA84FB4EADCull, 3066u, 0}, {0x65CA8D044D4561A6ull, 3048u, 0}, {0x6446614265754EFFull, 3030u, 0},
    {0x62D5A69CE4AC611Eull, 3013u, 0}, {0x614CF50E1A2BC335ull, 2995u, 0}, {0x5FD7E82755E928C3ull, 2978u, 0},
    {0x5E76D9A06BEB2CE7ull, 2962u, 0}, {0x5CFDA1AB90B9C8B1ull, 2945u, 0}, {0x5B823AA8AE878E30ull, 2928u, 0},
    {0x5A1B207A6C52BB11ull, 2912u, 0}, {0x58B20BCAE71E54BEull, 2896u, 0}, {0x5746F6FD60272942ull, 2880u, 0},
    {0x55D9DC5D1569B152ull, 2864u, 0}, {0x5481B7F4619C58D0ull, 2849u, 0}, {0x5310A172AB19FDC5ull, 2833u, 0},
    {0x51B4B670A0159B27ull, 2818u, 0}, {0x5056F011506D4953ull, 2803u, 0}, {0x4EF7493AC52DA84Bull, 2788u, 0},
    {0x4DAD5DDAF0445A5Eull, 2774u, 0}, {0x4C4A0757C43E91EFull, 2759u, 0}, {0x4AE4C0EAE2749277ull, 2744u, 0},
    {0x499587C4CE18B488ull, 2730u, 0}, {0x4844956618582E79ull, 2716u, 0}, {0x46F1E53F472330F4ull, 2702u, 0},
    {0x459D72AEAE98380Eull, 2688u, 0}, {0x444739000FB93372ull, 2674u, 0}, {0x4307D57622A28261ull, 2661u, 0},
    {0x41AE207E5E0BAACEull, 2647u, 0}, {0x406B78E44E7BDDB4ull, 2634u, 0}, {0x3F27389CE5AB3A04ull, 2621u, 0},
    {0x3DE15B97B8B26CA4ull, 2608u, 0}, {0x3C99DDB4C3BB4CD0ull, 2595u, 0}, {0x3B50BAC419CA00CAull, 2582u, 0},
    {0x3A1F6FE44ABCA15Bull, 2570u, 0}, {0x38D3173AFB575D38ull, 2557u, 0}, {0x379ECE6DEFAD8E17ull, 2545u, 0},
    {0x364F2FDC8C641775ull, 2532u, 0}, {0x3517D9F9105E3186ull, 2520u, 0}, {0x33DF07A4ED3467A4ull, 2508u, 0},
    {0x32A4B539E8AD68EDull, 2496u, 0}, {0x3168DF0446C4B67Dull, 2484u, 0}, {0x304602C983466376ull, 2473u, 0},
    {0x2F073AC4046AA33Aull, 2461u, 0}, {0x2DC6E3D80DDDC37Aull, 2449u, 0}, {0x2C9FDD104BF896FDull, 2438u, 0},
    {0x2B7780BE28090C49ull, 2427u, 0}, {0x2A4DCBC743686F46ull, 2416u, 0}, {0x29077999CDC7BA95ull, 2404u, 0},
    {0x27F64B4B2A5195BEull, 2394u, 0}, {0x26C8795A0B11E18Full, 2383u, 0}, {0x259941EBEBE4A10Eull, 2372u, 0},
    {0x2468A1AE03997599ull, 2361u, 0}, {0x235276FA85EC2144ull, 2351u, 0}, {0x221F1C844A736264ull, 2340u, 0},
    {0x2106715FF450533Dull, 2330u, 0}, {0x1FD05013C1429270ull, 2319u, 0}, {0x1EB518DEC04FEE36ull, 2309u, 0},
    {0x1D98A6FA604E41CDull, 2299u, 0}, {0x1C7AF7A8472D7652ull, 2289u, 0}, {0x1B5C0820E12D3EFAull, 2279u, 0},
    {0x1A3BD5933752254Aull, 2269u, 0}, {0x191A5D24C4EFB5C3ull, 2259u, 0}, {0x1814BE23F8C03647ull, 2250u, 0},
    {0x16F0D28AE56B4B9Cull, 2240u, 0}, {0x15E8FA4D8591C6FDull, 2231u, 0}, {0x14C290D4FAA503F8ull, 2221u, 0},
    {0x13B87598B1B6EDF5ull, 2212u, 0}, {0x128F83450EDA8D76ull, 2202u, 0}, {0x11831B06B9B7CBC1ull, 2193u, 0},
    {0x1075983598E47130ull, 2184u, 0}, {0x0F66F87C3DB0B422ull, 2175u, 0}, {0x0E57397DCAE10541ull, 2166u, 0},
    {0x0D4658D5D4FE1B36ull, 2157u, 0}, {0x0C34541841FB6771ull, 2148u, 0}, {0x0B2128D1282FAE5Bull, 2139u, 0},
    {0x0A2B974C0E56C7EBull, 2131u, 0}, {0x091638DE7541D282ull, 2122u, 0}, {0x081EAEC2F39F7789ull, 2114u, 0},
    {0x0707141B3BBA90D6ull, 2105u, 0}, {0x060D893EEA0EF5CEull, 2097u, 0}, {0x04F3A910D1A95D3Cull, 2088u, 0},
    {0x03F815161F807C7Aull, 2080u, 0}, {0x02FB88EBF0214EDCull, 2072u, 0}, {0x01FE02A6B1067890ull, 2064u, 0},
    {0x00FF805515885E02ull, 2056u, 0}, {0x0000000000000000ull, 2048u, 0},
};

__device__ __forceinline__ uint64_t mul_32_64(uint32_t a, uint64_t b)  // a b / 2^32
{
    return static_cast<uint64_t>(a) * static_cast<uint32_t>(b >> 32) + __umulhi(a, static_cast<uint32_t>(b));
}

// X / 2^64 * 2^e, negative if neg, rounded to nearest (X > 0; the result is a normal number).
__device__ __forceinline__ double double_of(uint64_t X, int e, bool neg)
{
    const int n = __clzll(static_cast<long long>(X));
    X <<= n;
    uint64_t b = ((X >> 11) + ((X >> 10) & 1u)) + (static_cast<uint64_t>(e - n + 1021) << 52);
    if (neg) b |= 0x8000000000000000ull;
    return __longlong_as_double(static_cast<long long>(b));
}

// sqrt(-2 ln u) = R / 2^63 * 2^e, u = (w + 1/2) / 2^32.
__device__ __forceinline__ void radius_fixed(uint32_t w, uint64_t &R, int &e)
{
    const uint64_t W = (static_cast<uint64_t>(w) << 1) | 1u;
    int n = __clzll(static_cast<long long>(W));
    const uint64_t M = W << n;  // m with 63 fraction bits; u = m 2^-(n - 30)
    const int el = n - 30, i = static_cast<int>(M >> 56) & 127;
    const uint4 te = __ldg(reinterpret_cast<const uint4 *>(&kLogTable[i]));
    const uint64_t T = (static_cast<uint64_t>(te.y) << 32) | te.x;
    const uint64_t G = ((1ull << 44) - (M >> 31) * te.z) << 20;  // g, 64 fraction bits
    // h = g / 2 + g^2 / 3 + ... + g^8 / 9, so that -ln(1 - g) = g (1 + h)
    const uint32_t g32 = static_cast<uint32_t>(G >> 32);
    uint32_t p = 0x20000000u + __umulhi(g32, 0x1C71C71Cu);
    p = 0x24924925u + __umulhi(g32, p);
    p = 0x2AAAAAABu + __umulhi(g32, p);
    p = 0x33333333u + __umulhi(g32, p);
    uint64_t h = 0x4000000000000000ull + mul_32_64(p, G);
    h = 0x5555555555555555ull + __umul64hi(G, h);
    h = 0x8000000000000000ull + __umul64hi(G, h);
    h = __umul64hi(G, h);
    const int ng = __clzll(static_cast<long long>(G));
    const uint64_t Gn = G << ng;
    const uint64_t y = (Gn >> 1) + (__umul64hi(Gn, h) >> 1);  // -ln(1 - g) 2^(63 + ng)
    // -2 ln u = X / 2^64 * 2^ex
    uint64_t X = T + (y >> (ng - 1));
    int ex = 1;
    if (el > 1) {
        X = static_cast<uint64_t>(el - 1) * 0x058B90BFBE8E7BCDull + (X >> 5);  // 2 ln 2 with 58 fraction bits
        ex = 6;
    } else if (i == 127) {
        X = y;
        ex = 2 - ng;
    }
    n = __clzll(static_cast<long long>(X));
    X <<= n;
    ex -= n;
    // A = X / 2^64 in [1/4, 1) with an even exponent, y0 ~ 1/sqrt(A)
    const int odd = ex & 1;
    const float af = __uint_as_float((static_cast<uint32_t>(126 - odd) << 23) + (static_cast<uint32_t>(X >> 40) & 0x7FFFFFu));
    X >>= odd;
    e = (ex + odd) >> 1;
    float yf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(af));
    const uint32_t y0 = __float2uint_rz(yf * 0x1p30f);
    const uint64_t s0 = mul_32_64(y0, X);                                                    // A y0, 62 fraction bits
    const int64_t r = static_cast<int64_t>((1ull << 60) - mul_32_64(y0, s0));                // 1 - A y0^2, 60 bits
    const int64_t rh = r >> 12;
    const int64_t c = (r >> 1) + ((3 * (rh * rh)) >> 39);                                    // r / 2 + 3 r^2 / 8
    R = (s0 + static_cast<uint64_t>(__mul64hi(static_cast<int64_t>(s0), c << 4))) << 1;
}

// (zc, zs) = r (cos, sin)(2 pi u_b): the angle as in box_muller_f32, quarter turn by quarter turn.
__device__ __forceinline__ void box_muller_fixed(uint32_t wa, uint32_t wb, double &zc, double &zs)
{
    uint64_t R;
    int e;
    radius_fixed(wa, R, e);
    const uint32_t ws = wb + 0x20000000u;
    const int32_t d = static_cast<int32_t>(((ws & 0x3FFFFFFFu) << 1) + 1u) - (1 << 30);  // angle pi/2 d / 2^31
    const uint32_t D = static_cast<uint32_t>(d < 0 ? -d : d);
    const uint64_t x = (static_cast<uint64_t>(D) * D) << 2;  // (d / 2^31)^2, 64 fraction bits
    const uint32_t x32 = static_cast<uint32_t>(x >> 32);
    // sin(pi/2 v) / (2 v), v = d / 2^31
    uint32_t q = 0x000B7D6Eu - __umulhi(x32, 0x00001AAFu);  // 51 fraction bits
    q = 0x03D1E86Au - __umulhi(x32, q);
    q = 0xF183A7EFu - __umulhi(x32, q);
    uint64_t S = 0x000541E0D21FB9E0ull - __umul64hi(x, static_cast<uint64_t>(q) << 13);
    S = 0x009969667315EC2Eull - __umul64hi(x, S);
    S = 0x0A335E33BAD570E9ull - __umul64hi(x, S);
    S = 0x52AEF39896F94AFBull - __umul64hi(x, S);
    S = 0xC90FDAA22168C235ull - __umul64hi(x, S);
    // cos(pi/2 v)
    q = 0x00090631u - __umulhi(x32, 0x000012A1u);  // 53 fraction bits
    q = 0x036DC49Fu - __umulhi(x32, q);
    q = 0xFCE9C51Cu - __umulhi(x32, q);
    uint64_t C = 0x0001A6D1F2A204A9ull - __umul64hi(x, static_cast<uint64_t>(q) << 11);
    C = 0x003C3EA0D1237576ull - __umul64hi(x, C);
    C = 0x05574F1F8F2FFE7Full - __umul64hi(x, C);
    C = 0x40F07C206D6B0ECDull - __umul64hi(x, C);
    C = 0x9DE9E64DF22EF2D2ull - (__umul64hi(x, C) >> 1);  // 63 fraction bits
    C = 0ull - 2 * __umul64hi(x, C);
    const int nd = __clz(static_cast<int>(D));
    const uint64_t zC = __umul64hi(R, C);                  // r cos 2^(63 - e)
    const uint64_t zS = mul_32_64(D << nd, __umul64hi(R, S));  // r |sin| 2^(61 + nd - e)
    const bool turn = (ws & 0x40000000u) != 0, half = (ws >> 31) != 0;
    // a quarter turn: (cos, sin) -> (-sin, cos); half a turn: both signs
    zc = double_of(turn ? zS : zC, (turn ? 3 - nd : 1) + e, (turn ? d > 0 : false) != half);
    zs = double_of(turn ? zC : zS, (turn ? 1 : 3 - nd) + e, (turn ? false : d < 0) != half);
}

}  // namespace gmrf
