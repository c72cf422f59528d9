// Natural logarithm of a double in integer arithmetic (sm_103a).
//
// GB300 issues an FP64 warp instruction once per 64 cycles and sub-partition; the library
// logarithm is about 30 of them (2030 cycles, 560 per warp with the multiprocessor full), and the
// FP64 forms take N + 1 logarithms per node.  This one uses the integer and FP32 pipes only: the
// table-driven reduction of P. T. P. Tang (ACM Trans. Math. Softw. 16, 1990) carried in 64-bit
// fixed point.
//
//   x = 2^k z, z in [0.6875, 1.375);  z lies in one of 128 intervals, each with a constant
//   ic / 1024 near 1 / z, so that r = z ic / 1024 - 1 is small (|r| <= 2^-7) and exact in 64 bits;
//   ln x = k ln 2 - ln(ic / 1024) + r p(r),  p(r) = ln(1 + r) / r = 1 - r/2 + r^2/3 - ...
//
// p by Horner's rule: the coefficients from 1/6 on in float, 1/5 in 32 bits, the rest in 64 bits
// (Q62), an error below 2^-61.  The sum is formed in fixed point (Q64 for k = 0, Q58 otherwise)
// and converted once; around x = 1, where it is r p(r) alone, r is normalised first, so the
// result keeps its relative accuracy.  Largest error 0.56 ulp (every interval's edges, arguments near
// 1 and 10^8 random ones against long double on the host, tests/test_log.py; CUDA documents 1 ulp for log).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace fmlbm {

struct alignas(16) LogEntry {
    long long ic;   // 1024 / z, rounded
    long long lnc;  // -ln(ic / 1024), Q64
};
#define FMLBM_LOG_TABLE \
    {1485, -6856622409918966101ll}, {1477, -6756977365064706458ll}, {1469, -6656791136050761017ll}, \
    {1460, -6543427381071246885ll}, {1452, -6442071389410675207ll}, {1444, -6340155417054629666ll}, \
    {1436, -6237673241947637361ll}, {1429, -6147531904800161429ll}, {1421, -6043970964318060933ll}, \
    {1413, -5939825343587003420ll}, {1406, -5848213088235548201ll}, {1398, -5742953207345004463ll}, \
    {1391, -5650355516661447572ll}, {1383, -5543957274616570749ll}, {1376, -5450352718192624241ll}, \
    {1369, -5356270759416466736ll}, {1362, -5261706503614631935ll}, {1355, -5166654980450020449ll}, \
    {1348, -5071111142354304413ll}, {1341, -4975069862919523938ll}, {1334, -4878525935247593925ll}, \
    {1327, -4781474070256392589ll}, {1321, -4697878410242295377ll}, {1314, -4599868913257257143ll}, \
    {1307, -4501335898734907285ll}, {1301, -4416458092206103443ll}, {1295, -4331187936949539380ll}, \
    {1288, -4231205339480400567ll}, {1282, -4145072525837730946ll}, {1276, -4058535647478120774ll}, \
    {1269, -3957060178604328672ll}, {1263, -3869634687599607112ll}, {1257, -3781792883163315921ll}, \
    {1251, -3693530781412173139ll}, {1245, -3604844341002602229ll}, {1239, -3515729462020377521ll}, \
    {1234, -3441136784262883231ll}, {1228, -3351225587219777939ll}, {1222, -3260874007046890488ll}, \
    {1216, -3170077708527314833ll}, {1211, -3094071238929963933ll}, {1205, -3002448149539718528ll}, \
    {1200, -2925746400471432400ll}, {1194, -2833281324293745646ll}, {1189, -2755871457974340717ll}, \
    {1183, -2662548776268264499ll}, {1178, -2584417596044838233ll}, {1173, -2505954083131827139ll}, \
    {1168, -2427155398279344845ll}, {1163, -2348018665696099656ll}, {1157, -2252604259485674825ll}, \
    {1152, -2172713514977912298ll}, {1147, -2092475267225756768ll}, {1142, -2011886479926060167ll}, \
    {1137, -1930944076806532158ll}, {1132, -1849644940921122012ll}, {1128, -1784346663626416374ll}, \
    {1123, -1702397421459214925ll}, {1118, -1620082496500726674ll}, {1113, -1537398610538312856ll}, \
    {1108, -1454342441078812732ll}, {1104, -1387627199918624915ll}, {1099, -1303892403058495094ll}, \
    {1095, -1236629815958875205ll}, {1090, -1152205210593624476ll}, {1085, -1067392444758829412ll}, \
    {1081, -999260348567128990ll}, {1077, -930875676835265680ll}, {1072, -845036787304660515ll}, \
    {1068, -776076916065200710ll}, {1063, -689512965221337966ll}, {1059, -619968136107063631ll}, \
    {1055, -550160128204548867ll}, {1051, -480086942047627894ll}, {1046, -392119469317874213ll}, \
    {1042, -321442202498300337ll}, {1038, -250493099368188280ll}, {1034, -179270060797655839ll}, \
    {1030, -107770963248212282ll}, {1024, 0ll}, {1024, 0ll}, \
    {1012, 217449402910135620ll}, {1004, 363852902130987047ll}, {997, 492916105791551876ll}, \
    {989, 641531161979034824ll}, {982, 772558814357976946ll}, {975, 904523821220465167ll}, \
    {967, 1056506094520383395ll}, {960, 1190525582320469641ll}, {953, 1325525880113686902ll}, \
    {946, 1461521449748507975ll}, {940, 1578892433671965565ll}, {933, 1716775839671240844ll}, \
    {926, 1855697645811877951ll}, {920, 1975611897379757024ll}, {913, 2116504244618060346ll}, \
    {907, 2238131569247314719ll}, {901, 2360566160788172870ll}, {895, 2483818806891349249ll}, \
    {889, 2607900512898827746ll}, {883, 2732822507740801840ll}, {877, 2858596250033651404ll}, \
    {871, 2985233434387237051ll}, {865, 3112745997930193658ll}, {859, 3241146127062327672ll}, \
    {854, 3348833205060016471ll}, {848, 3478893044001375095ll}, {843, 3587981144728763741ll}, \
    {838, 3697718196926968058ll}, {832, 3830270221691897566ll}, {827, 3941462505760077071ll}, \
    {822, 4053329095246964985ll}, {817, 4165878218482716586ll}, {812, 4279118255333998699ll}, \
    {807, 4393057740948001826ll}, {802, 4507705369612800438ll}, {797, 4623069998738427277ll}, \
    {792, 4739160652963219918ll}, {787, 4855986528390199858ll}, {783, 4949982879917862053ll}, \
    {778, 5068155891833629052ll}, {773, 5187090823981735259ll}, {769, 5282793991037459835ll}, \
    {764, 5403125429299924605ll}, {760, 5499958953883438787ll}, {755, 5621720082921211662ll}, \
    {751, 5719710985719572930ll}, {747, 5818225206901671492ll},

__device__ const LogEntry kLogTable[128] = {FMLBM_LOG_TABLE};

__host__ __device__ __forceinline__ long long mulhi_s64(long long a, long long b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (long long)(((__int128)a * b) >> 64);
#endif
}

// ln of a positive normal x between 2^-43 and 2^44 (log_reducible): table entry e of its
// interval (log_index).
__host__ __device__ __forceinline__ bool log_reducible(uint64_t bits) {
    return (bits >> 52) - (1023 - 43) < 87;  // sign 0, exponent within +-43
}
__host__ __device__ __forceinline__ int log_index(uint64_t bits) {
    return (int)((bits - 0x3FE6000000000000ull) >> 45) & 127;
}
__host__ __device__ __forceinline__ double log_reduced(uint64_t bits, LogEntry e) {
    const uint64_t t = bits - 0x3FE6000000000000ull;
    const int k = (int)((int64_t)t >> 52);
    const uint64_t mant = (bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    // z = mant 2^-52 for z >= 1, mant 2^-53 below; r in Q63
    const bool ge1 = (bits >> 52) == (uint64_t)(1023 + k);
    const long long r = (long long)(((mant * (uint64_t)e.ic) << (ge1 ? 1 : 0)) - 0x8000000000000000ull);
    const int r31 = (int)(r >> 32);  // Q31
    const float rf = (float)r31 * 4.656612873077393e-10f;
    const float t5 = 1.f / 6.f - rf * (1.f / 7.f - rf * (1.f / 8.f - rf * (1.f / 9.f)));
    const int t5i = (int)(t5 * 4294967296.f);  // Q32, below 2^30
    // 1/5 - r t5: (Q31 Q32) >> 32 = Q31, doubled to Q32; then to Q62
    const long long t4 = (long long)(858993459u - (unsigned)(2 * (int)(((long long)r31 * t5i) >> 32))) << 30;
    const long long r6 = r << 6;  // 2^6 r in Q63
    long long p = 1152921504606846976ll - (mulhi_s64(r6, t4) >> 5);  // 1/4 - r t4
    p = 1537228672809129301ll - (mulhi_s64(r6, p) >> 5);             // 1/3 -
    p = 2305843009213693952ll - (mulhi_s64(r6, p) >> 5);             // 1/2 -
    p = 4611686018427387904ll - (mulhi_s64(r6, p) >> 5);             // 1 -
    const bool one = k == 0 && e.ic == 1024;
#ifdef __CUDA_ARCH__
    const int lz = __clzll(r ^ (r >> 63));
#else
    const uint64_t ar = (uint64_t)(r ^ (r >> 63));
    const int lz = ar ? __builtin_clzll(ar) : 64;
#endif
    const int sh = one ? (lz > 63 ? 62 : lz - 1) : 6;
    const long long q = mulhi_s64(r << sh, p);  // r p in Q(61 + sh)
    const long long v64 = e.lnc + ((q + 4) >> 3);     // k = 0: Q64
    const long long v58 = (long long)k * 199786072581291495ll + ((v64 + 32) >> 6);
    const long long v = one ? q : (k == 0 ? v64 : v58);
    const int scale = one ? 61 + sh : (k == 0 ? 64 : 58);
    double d = (double)v;
    uint64_t db;
    memcpy(&db, &d, 8);
    db -= v == 0 ? 0 : (uint64_t)scale << 52;
    memcpy(&d, &db, 8);
    return d;
}

__device__ __forceinline__ double ln_f64(double x) {
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    if (!log_reducible(bits)) return log(x);  // zero, negative, NaN, infinite, out of range
    const longlong2 e = __ldg(reinterpret_cast<const longlong2*>(kLogTable) + log_index(bits));
    return log_reduced(bits, LogEntry{e.x, e.y});
}

}  // namespace fmlbm
