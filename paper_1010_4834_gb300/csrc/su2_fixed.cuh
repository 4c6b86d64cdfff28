// Quaternion products of FP64 links in 58-bit fixed point on the integer
// pipe.  GB300 issues FP64 at 2 lanes per clock and SM (a DFMA every 64
// clocks per warp and scheduler) and the 32 x 32 + 64 bit multiply-add
// (IMAD.WIDE) at 63 (both measured), so a product of two quaternions, 16
// FP64 multiply-adds or 48 IMAD.WIDE, takes 8 clocks per link and SM on one
// pipe and 0.75 on the other.
//
// A component v of a link is held as two signed 32-bit limbs,
//   v = h 2^-29 + l 2^-58,  |l| < 2^29,
// and a product of two components as (h h') 2^-58 + (h l' + l h') 2^-87, the
// two parts in 64-bit sums; l l' < 2^-58 is left out.  Errors, absolute, in units
// of 2^-58, for norms n <= 1.0607 (a quaternion's components then add up to 2 n at
// most): a converted component is truncated below 1; a component of a product of two
// links carries 4 n from their conversions, below 4 from four l l' and 4 from its
// rounding to 8 units, 12.3 together; a term of a staple, that product times a
// third link, 2 n 12.3 + 2 n^2 + 2 = 30.3 (the product's low limbs are centred); the
// sum of six and its rounding 186, or 2^-50.4.  Measured: a product 6.7 at most, 2.4
// rms; a staple sum 2^-53.3 at most, 2^-55.3 rms, several times closer than in FP64
// (magnitude up to 6, roundings of 2^-53 and more per addition).
//
// What a link must be for this: components |v| in [2^-31, 2) and a norm within 6%
// of one.  fix_link raises `bad` otherwise, and the thread starts again with
// fix_any_link, which takes any |v| < 2 (zeros: cold starts, Abelian fields) and
// costs twice the shifts; values other than near-unit quaternions, which a store
// set from outside may hold, are computed in FP64 (smearing does so at once).
//
// Sums.  With norms n <= 1.0607: |sum h h'| <= 2^58 n^2 per component of a
// product (Cauchy-Schwarz); |sum (h l' + l h')| <= 2^29 (sum |h| + sum |h'|)
// <= 2^59 (n + n').  A staple's six products of a product (norm <= n^2) and a
// link then stay below 6 (1.2) 2^58 < 2^61 and 6 (1.13 + 1.07) 2^59 < 2^63.
#pragma once

#include <stdint.h>

namespace su2 {

#ifdef __CUDACC__
#define SU2_HD __host__ __device__ __forceinline__
#else
#define SU2_HD inline
#endif

constexpr int kFixLow = 29;                  // bits of the low limb
constexpr int kFixFrac = 2 * kFixLow;        // fraction bits of a value

struct Fix { int h, l; };
struct FixQuat { Fix w, x, y, z; };
// Two-part 64-bit sums of a quaternion's components.
struct FixSum { int64_t hw, hx, hy, hz, mw, mx, my, mz; };

// The high word of (hi:lo) << (n mod 32).
SU2_HD uint32_t fix_funnel(uint32_t lo, uint32_t hi, uint32_t n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, n);
#else
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << (n & 31)) >> 32);
#endif
}

// The limbs of v (or -v), |v| in [2^-31, 2): the 53-bit significand is
// aligned by funnel shifts whose amount, the exponent mod 32, needs no
// arithmetic, and truncated at 2^-58.  Shifts and logic run on the ALU pipe,
// which bounds the update; the sign is a multiplication, on the other one.
// The bits of `bad` that kFixBadExp selects are raised for any other v.
constexpr uint32_t kFixBadExp = 0x7E0u;
// neg: 0, or -1 for -v.
SU2_HD Fix fix_from(uint32_t lo, uint32_t hi, int neg, uint32_t& bad) {
  const uint32_t e = hi >> 20;               // sign and exponent
  bad |= e ^ 0x3E0u;
  const uint32_t mh = (fix_funnel(lo, hi, 10) & 0x7FFFFFFFu) | 0x40000000u;
  const uint32_t ml = lo * 1024u;
  const int s = ((int32_t)hi >> 31 ^ neg) | 1;
  Fix f;
  f.h = (int)fix_funnel(mh, 0u, e) * s;
  f.l = (int)(fix_funnel(ml, mh, e) >> 3) * s;
  return f;
}

// A link's limbs, conjugated with conj = -1 (0: as it is).  bad.e collects
// exponents outside the range (kFixBadExp), bad.n >> 24 a squared norm outside
// 1 +- 1/8.
struct FixBad { uint32_t e, n; };
SU2_HD bool fix_ok(const FixBad& b) { return (b.e & kFixBadExp) == 0u && (b.n >> 24) == 0u; }

SU2_HD void fix_check_norm(const FixQuat& q, FixBad& bad) {
  // squared norm in units of 2^-58, less 1 - 1/8: in [0, 1/4) for norm^2
  // within 1 +- 1/8; components below 2 keep the sum below 2^62
  int64_t n = -((int64_t)7 << 55);
  n += (int64_t)q.w.h * q.w.h;
  n += (int64_t)q.x.h * q.x.h;
  n += (int64_t)q.y.h * q.y.h;
  n += (int64_t)q.z.h * q.z.h;
  bad.n |= (uint32_t)((uint64_t)n >> 32);
}

SU2_HD FixQuat fix_link(uint32_t w0, uint32_t w1, uint32_t x0, uint32_t x1, uint32_t y0, uint32_t y1, uint32_t z0,
                        uint32_t z1, int conj, FixBad& bad) {
  FixQuat q;
  q.w = fix_from(w0, w1, 0, bad.e);
  q.x = fix_from(x0, x1, conj, bad.e);
  q.y = fix_from(y0, y1, conj, bad.e);
  q.z = fix_from(z0, z1, conj, bad.e);
  fix_check_norm(q, bad);
  return q;
}

SU2_HD Fix fix_neg(const Fix& a) { return Fix{-a.h, -a.l}; }

// s += a b.  As an instruction, not an expression: left to itself the
// compiler reassociates the integer sums across a staple's terms and keeps
// every link of the staple alive (1.4 KB of spills a thread).
SU2_HD void fix_mad(int64_t& s, int a, int b) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
#else
  s += (int64_t)a * b;
#endif
}

SU2_HD void fix_mac(int64_t& h, int64_t& m, const Fix& a, const Fix& b) {
  fix_mad(h, a.h, b.h);
  fix_mad(m, a.h, b.l);
  fix_mad(m, a.l, b.h);
}

// s += a b
SU2_HD void fix_mac(FixSum& s, const FixQuat& a, const FixQuat& b) {
  const Fix nx = fix_neg(a.x), ny = fix_neg(a.y), nz = fix_neg(a.z);
  fix_mac(s.hw, s.mw, a.w, b.w);
  fix_mac(s.hw, s.mw, nx, b.x);
  fix_mac(s.hw, s.mw, ny, b.y);
  fix_mac(s.hw, s.mw, nz, b.z);
  fix_mac(s.hx, s.mx, a.w, b.x);
  fix_mac(s.hx, s.mx, a.x, b.w);
  fix_mac(s.hx, s.mx, ny, b.z);
  fix_mac(s.hx, s.mx, a.z, b.y);
  fix_mac(s.hy, s.my, a.w, b.y);
  fix_mac(s.hy, s.my, a.y, b.w);
  fix_mac(s.hy, s.my, nz, b.x);
  fix_mac(s.hy, s.my, a.x, b.z);
  fix_mac(s.hz, s.mz, a.w, b.z);
  fix_mac(s.hz, s.mz, a.z, b.w);
  fix_mac(s.hz, s.mz, nx, b.y);
  fix_mac(s.hz, s.mz, a.y, b.x);
}

// The limbs of v, the low one centred (|l| <= 2^28): the omitted l l' then
// averages to zero, where two low limbs of one sign would all but bias a
// product's components by 2^-60, which adds up along a chain of products.
// fix_split_raised takes v + 2^28.
constexpr int64_t kFixHalf = (int64_t)1 << (kFixLow - 1);
SU2_HD Fix fix_split_raised(int64_t v) {
  return Fix{(int)(v >> kFixLow), (int)((uint32_t)v & ((1u << kFixLow) - 1u)) - (int)kFixHalf};
}
SU2_HD Fix fix_split(int64_t v) { return fix_split_raised(v + kFixHalf); }

// An empty sum: the middle part starts at half a unit of its high word.
constexpr int64_t kFixMid = (int64_t)1 << 31;
SU2_HD FixSum fix_zero() { return FixSum{0, 0, 0, 0, kFixMid, kFixMid, kFixMid, kFixMid}; }

// The value of a sum in units of 2^-58: h + m 2^-29, from the high word of m in
// one multiply-add (rounded to 8 units, 2^-55, by the half unit fix_zero starts m
// with).
SU2_HD int64_t fix_fold(int64_t h, int64_t m) {
  fix_mad(h, (int)(m >> 32), 1 << (32 - kFixLow));
  return h;
}


// h + a . b in units of 2^-58
SU2_HD int64_t fix_dot(const FixQuat& a, const FixQuat& b, int64_t h) {
  int64_t m = kFixMid;
  fix_mac(h, m, a.w, b.w);
  fix_mac(h, m, a.x, b.x);
  fix_mac(h, m, a.y, b.y);
  fix_mac(h, m, a.z, b.z);
  return fix_fold(h, m);
}

SU2_HD FixQuat fix_one() { return FixQuat{{1 << kFixLow, 0}, {0, 0}, {0, 0}, {0, 0}}; }
SU2_HD FixQuat fix_conj(const FixQuat& a) { return FixQuat{a.w, fix_neg(a.x), fix_neg(a.y), fix_neg(a.z)}; }
SU2_HD int64_t fix_value(const Fix& a) { return (int64_t)a.h * (1 << kFixLow) + a.l; }

SU2_HD FixQuat fix_mul(const FixQuat& a, const FixQuat& b) {
  FixSum s{kFixHalf, kFixHalf, kFixHalf, kFixHalf, kFixMid, kFixMid, kFixMid, kFixMid};
  fix_mac(s, a, b);
  return FixQuat{fix_split_raised(fix_fold(s.hw, s.mw)), fix_split_raised(fix_fold(s.hx, s.mx)),
                 fix_split_raised(fix_fold(s.hy, s.my)), fix_split_raised(fix_fold(s.hz, s.mz))};
}

// The limbs of any |v| < 2 (components of a unit quaternion, however small):
// as fix_from, with a 64-bit shift in place of the funnel shifts.
SU2_HD uint64_t fix_shr(uint64_t v, uint32_t n) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));  // 0 from n = 64 on
  return r;
#else
  return n > 63 ? 0 : v >> n;
#endif
}
SU2_HD Fix fix_from_any(uint32_t lo, uint32_t hi) {
  const uint64_t m = (((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 6;
  const int64_t v = (int64_t)fix_shr(m, 1023u - ((hi >> 20) & 0x7FFu));
  const int64_t s = (int64_t)((int32_t)hi >> 31);
  return fix_split((v ^ s) - s);
}

// fix_link for components of any size, zero too: the path of links that it
// refuses for them (cold starts, Abelian fields).
SU2_HD FixQuat fix_any_link(uint32_t w0, uint32_t w1, uint32_t x0, uint32_t x1, uint32_t y0, uint32_t y1, uint32_t z0,
                            uint32_t z1, int conj, FixBad& bad) {
  FixQuat q{fix_from_any(w0, w1), fix_from_any(x0, x1), fix_from_any(y0, y1), fix_from_any(z0, z1)};
  if (conj) q.x = fix_neg(q.x), q.y = fix_neg(q.y), q.z = fix_neg(q.z);
  if ((w1 | x1 | y1 | z1) & 0x40000000u) bad.e |= kFixBadExp;   // a component of 2 or more, NaN
  fix_check_norm(q, bad);
  return q;
}

// The positive double 1.m 2^e with the given words, e < 11, in units of 2^-62
// (0 below 2^-62).
SU2_HD int64_t fix_unsigned62(uint32_t lo, uint32_t hi) {
  const uint64_t m = (((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 10;   // 1.m 2^62
  return (int64_t)fix_shr(m, 1023u - (hi >> 20));
}

// ---------------------------------------------------------------------------
// Elementary functions of a 32-bit draw x in fixed point, for the uniforms
// u = (x + 1/2) 2^-32 (z = 2 x + 1 units of 2^-33).
// ---------------------------------------------------------------------------
SU2_HD uint64_t fix_umulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
SU2_HD int64_t fix_mulhi(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}

// Table of -ln u: the leading 7 fraction bits i of the significand m select
// a 16-bit reciprocal I of the interval's centre 1 + (i + 1/2)/128, and
// t = ln(I 2^-16) in units of 2^-58 (Tang's table-driven logarithm, ACM TOMS
// 16, 1990).  Aligned for the 16-byte load of an entry.
struct alignas(16) FixLog { int64_t t; int64_t inv; };
#define SU2_FIX_LOG_TABLE                                                                                     \
  {-1123689413616504ll, 65281}, {-3357597927618363ll, 64777}, {-5573081980516173ll, 64281}, {-7774097633284494ll, 63792}, \
  {-9960179792198405ll, 63310}, {-12126270533003689ll, 62836}, {-14276411659491797ll, 62369}, {-16410121222244478ll, 61909}, \
  {-18531602068116421ll, 61455}, {-20635740466204764ll, 61008}, {-22722039064927134ll, 60568}, {-24799582025815337ll, 60133}, \
  {-26858413540281678ll, 59705}, {-28902884053536989ll, 59283}, {-30932580743649448ll, 58867}, {-32947086476193657ll, 58457}, \
  {-34945979938847877ll, 58053}, {-36933835054502750ll, 57654}, {-38910325529261412ll, 57260}, {-40870053156443740ll, 56872}, \
  {-42817683366232216ll, 56489}, {-44752878596514639ll, 56111}, {-46675297730443060ll, 55738}, {-48584596183895111ll, 55370}, \
  {-50480425999051922ll, 55007}, {-52362435944214310ll, 54649}, {-54235580169965915ll, 54295}, {-56094261258760709ll, 53946}, \
  {-57943495935180337ll, 53601}, {-59777612058294982ll, 53261}, {-61601689236295459ll, 52925}, {-63415461306664967ll, 52593}, \
  {-65218659378811176ll, 52265}, {-67005462753766376ll, 51942}, {-68786661121907461ll, 51622}, {-70556463022809603ll, 51306}, \
  {-72308937057891222ll, 50995}, {-74060758153255190ll, 50686}, {-75794685778214066ll, 50382}, {-77521841105521937ll, 50081}, \
  {-79236249038272246ll, 49784}, {-80943442831734593ll, 49490}, {-82637374327710623ll, 49200}, {-84323641262814286ll, 48913}, \
  {-85996122636574751ll, 48630}, {-87666442239035341ll, 48349}, {-89322513713852678ll, 48072}, {-90970064315697501ll, 47798}, \
  {-92602827877981356ll, 47528}, {-94232695511926415ll, 47260}, {-95853431832258605ll, 46995}, {-97464829818843168ll, 46733}, \
  {-99066680743462226ll, 46474}, {-100658774212257587ll, 46218}, {-102240898210457049ll, 45965}, {-103819144159341520ll, 45714}, \
  {-105380721177603795ll, 45467}, {-106938056994554811ll, 45222}, {-108491036470283102ll, 44979}, {-110033100610825232ll, 44739}, \
  {-111564028317700263ll, 44502}, {-113090108292244953ll, 44267}, {-114604674239412068ll, 44035}, {-116114080842717206ll, 43805}, \
  {-117618204687399774ll, 43577}, {-119110272454368929ll, 43352}, {-120596738067439682ll, 43129}, {-122077474337318462ll, 42908}, \
  {-123545601112522204ll, 42690}, {-125007671817164964ll, 42474}, {-126463555680543339ll, 42260}, {-127913120811646852ll, 42048}, \
  {-129356234214028563ll, 41838}, {-130785838262925369ll, 41631}, {-132215610446518860ll, 41425}, {-133631533202955533ll, 41222}, \
  {-135047419321088853ll, 41020}, {-136456172742086876ll, 40820}, {-137850558873334091ll, 40623}, {-139244593761669443ll, 40427}, \
  {-140631075308799936ll, 40233}, {-142009861410168356ll, 40041}, {-143380809057368345ll, 39851}, {-144751041439201743ll, 39662}, \
  {-146105913907054427ll, 39476}, {-147459849378452864ll, 39291}, {-148805434261750188ll, 39108}, {-150149925729018451ll, 38926}, \
  {-151485839844384666ll, 38746}, {-152813027613847517ll, 38568}, {-154131339324825338ll, 38392}, {-155448166422473372ll, 38217}, \
  {-156755884407054649ll, 38044}, {-158061951890219191ll, 37872}, {-159358674217786227ll, 37702}, {-160653577268204128ll, 37533}, \
  {-161938896233296224ll, 37366}, {-163222224331464060ll, 37200}, {-164495726637303404ll, 37036}, {-165767063754120698ll, 36873}, \
  {-167028330713673717ll, 36712}, {-168287255519860060ll, 36552}, {-169543783106086327ll, 36393}, {-170789903513667779ll, 36236}, \
  {-172033445978033476ll, 36080}, {-173266330615560622ll, 35926}, {-174504511490552898ll, 35772}, {-175731850222456945ll, 35620}, \
  {-176948185025791777ll, 35470}, {-178169674533618054ll, 35320}, {-179379972392946648ll, 35172}, {-180578915257295890ll, 35026}, \
  {-181782866165766112ll, 34880}, {-182983569030984713ll, 34735}, {-184172629634930104ll, 34592}, {-185358249145501941ll, 34450}, \
  {-186540364650487953ll, 34309}, {-187718912764703512ll, 34169}, {-188885359867195147ll, 34031}, {-190056546682960709ll, 33893}, \
  {-191215434605052309ll, 33757}, {-192370428085174609ll, 33622}, {-193530068469277957ll, 33487}, {-194677109675153417ll, 33354}, \
  {-195820057869899388ll, 33222}, {-196958845992691321ll, 33091}, {-198093406559548696ll, 32961}, {-199223671668903128ll, 32832}, \

#ifdef __CUDACC__
static __device__ const FixLog fix_log_table[128] = {SU2_FIX_LOG_TABLE};
#endif
static const FixLog fix_log_table_host[128] = {SU2_FIX_LOG_TABLE};

// -ln u in units of 2^-58 (at most 22.9), absolute error below 2^-57 (1 - ln u)
// (near u = 1 few digits of the logarithm itself: a0 takes it absolutely): with z =
// m 2^(63 - lz), 1 <= m < 2, -ln u = (lz - 30) ln 2 + t - ln(1 + r), where r = m
// I 2^-16 - 1 is exact in 48 bits, |r| < 2^-7.9, and ln(1 + r) = r - r q, q =
// p 2^-8 - p^2 2^-14/3 + p^3 2^-23 - ... in p = 2^7 r (Taylor to r^7).
SU2_HD int64_t fix_neg_log(uint32_t x) {
  const uint64_t z = 2 * (uint64_t)x + 1;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)z);
#else
  const int lz = __builtin_clzll(z);
#endif
  const uint64_t zn = z << lz;
  const uint32_t i = (uint32_t)(zn >> 56) & 127u;
#ifdef __CUDA_ARCH__
  static_assert(sizeof(FixLog) == sizeof(longlong2) && alignof(FixLog) >= alignof(longlong2), "one load an entry");
  const longlong2 e = __ldg(reinterpret_cast<const longlong2*>(fix_log_table) + i);
  const int64_t t = e.x;
  const uint32_t inv = (uint32_t)e.y;
#else
  const int64_t t = fix_log_table_host[i].t;
  const uint32_t inv = (uint32_t)fix_log_table_host[i].inv;
#endif
  const int64_t r = (int64_t)((zn >> 31) * inv) - ((int64_t)1 << 48);   // r 2^48
  const int64_t p = r * ((int64_t)1 << 22);                            // p 2^63
  const int ph = (int)(p >> 32);                                       // p 2^31
  // Horner, the inner terms in 32 bits: a 2^62, b 2^54, c 2^62, d 2^62
  const int a0 = (int)(((int64_t)1 << 62) / ((int64_t)6 << 35)) - (int)(((int64_t)ph * 149797) >> 31);
  const int a = (int)(((int64_t)1 << 62) / ((int64_t)5 << 28) / 2) - (int)(((int64_t)ph * a0) >> 32);     // 2^61
  const int b = (int)((int64_t)1 << 31 >> 1) - (int)(((int64_t)ph * a) >> 39);                           // 2^53
  const int64_t c = (((int64_t)1 << 48) / 3) - (((int64_t)ph * b) >> 22);                                // 2^62
  const int64_t d = ((int64_t)1 << 54) - 2 * fix_mulhi(p, c);                                            // 2^62
  const int64_t q = 2 * fix_mulhi(p, d);                                                                 // 2^62
  const int64_t rr = r * ((int64_t)1 << 12);                                                             // r 2^60
  const int64_t ln1 = (rr >> 2) - fix_mulhi(rr, q);                                                      // 2^58
  return (int64_t)(lz - 30) * 199786072581291495ll + t - ln1;
}

// The angle 2 pi u lies in quadrant q = x >> 30 at theta = (pi/4) rho from its
// middle, rho = r 2^-30, |r| < 2^30.
SU2_HD int fix_quarter(uint32_t x) { return (int)((2u * x + 1u) & 0x7FFFFFFFu) - (1 << 30); }

// cos^2(2 pi u) in units of 2^-63 = 1/2 -+ (1/2) sin 2 theta (minus in even
// quadrants); Taylor series of the sine to (2 theta)^23, in Horner form in
// t = rho^2; errors a few 2^-63.
SU2_HD uint64_t fix_cos2(uint32_t x) {
  const int r = fix_quarter(x);
  const uint64_t t = (uint64_t)((int64_t)r * r) << 4;                  // 2^64
  const uint32_t th = (uint32_t)(t >> 32);
  // terms below 2^-32 in 32 bits
  uint32_t v = 0x944u - (uint32_t)(((uint64_t)0xCu * th) >> 32);
  v = 0x62901u - (uint32_t)(((uint64_t)v * th) >> 32);
  v = 0x355D865u - (uint32_t)(((uint64_t)v * th) >> 32);
  uint64_t s = 0x000000016FADB9F1ull - (((uint64_t)v * th) >> 32);
  s = 0x0000007A3D0D3406ull - fix_umulhi(s, t);
  s = 0x00001E3074FDE887ull - fix_umulhi(s, t);
  s = 0x000541E0D21FB9E0ull - fix_umulhi(s, t);
  s = 0x009969667315EC2Eull - fix_umulhi(s, t);
  s = 0x0A335E33BAD570E9ull - fix_umulhi(s, t);
  s = 0x52AEF39896F94AFBull - fix_umulhi(s, t);
  s = 0xC90FDAA22168C235ull - fix_umulhi(s, t);                        // (sin 2 theta) / (2 rho)
  const uint64_t a = (uint64_t)(uint32_t)(r < 0 ? -r : r) << 34;       // |rho| 2^64
  const uint64_t h = fix_umulhi(s, a) >> 1;                            // |sin 2 theta| / 2, 2^-63
  const bool minus = ((x >> 30) & 1u) == (uint32_t)(r < 0);
  return minus ? ((uint64_t)1 << 62) - h : ((uint64_t)1 << 62) + h;
}

// cos and sin of 2 pi u in units of 2^-62: with C, S = sqrt(1/2) cos theta,
// sqrt(1/2) sin theta the quadrant's middle (at 45 degrees) gives
// (C - S, C + S), turned by q quarters.  Taylor series to theta^16 and
// theta^17.
SU2_HD void fix_sincos(uint32_t x, int64_t* sn, int64_t* cs) {
  const int r = fix_quarter(x);
  const uint64_t t = (uint64_t)((int64_t)r * r) << 4;
  const uint32_t th = (uint32_t)(t >> 32);
  uint32_t v = 0x4D95A0u - (uint32_t)((0x330Cull * th) >> 32);
  v = 0x596B1624u - (uint32_t)(((uint64_t)v * th) >> 32);
  uint64_t c = 0x0000004ABEA760DEull - (((uint64_t)v * th) >> 32);
  c = 0x00002A9971EA0F44ull - fix_umulhi(c, t);
  c = 0x000F1B558609C5CFull - fix_umulhi(c, t);
  c = 0x02DEB493652FC3C4ull - fix_umulhi(c, t);
  c = 0x37D4B6C0E564C456ull - fix_umulhi(c, t);
  c = 0xB504F333F9DE6484ull - fix_umulhi(c, t);
  uint32_t w = 0x40FF4u - (uint32_t)((0x25Cull * th) >> 32);
  w = 0x566F877u - (uint32_t)(((uint64_t)w * th) >> 32);
  uint64_t s = 0x00000005563609DEull - (((uint64_t)w * th) >> 32);
  s = 0x000003B7ADFAAD60ull - fix_umulhi(s, t);
  s = 0x0001B1E9F34CA91Full - fix_umulhi(s, t);
  s = 0x007368418E083860ull - fix_umulhi(s, t);
  s = 0x0E9DD2E0E2FA3EEFull - fix_umulhi(s, t);
  s = 0x8E2C18D6EB17214Full - fix_umulhi(s, t);
  const uint64_t a = (uint64_t)(uint32_t)(r < 0 ? -r : r) << 34;
  const int64_t S = (int64_t)(fix_umulhi(s, a) >> 2), C = (int64_t)(c >> 2);
  const int64_t Sn = r < 0 ? -S : S;
  const int64_t d = C - Sn, u = C + Sn;
  const uint32_t q = x >> 30;
  const int64_t cc = (q & 1u) ? u : d, ss = (q & 1u) ? d : u;
  *cs = (q == 1u || q == 2u) ? -cc : cc;
  *sn = (q & 2u) ? -ss : ss;
}

#ifdef __CUDACC__
// v 2^-FRAC in FP64: the conversion rounds once, the scale is an exponent step.
template <int FRAC = kFixFrac> __device__ __forceinline__ double fix_to_double(int64_t v) {
  const double d = __ll2double_rn(v);
  return __hiloint2double(v ? __double2hiint(d) - (FRAC << 20) : 0, __double2loint(d));
}
#endif

}  // namespace su2
