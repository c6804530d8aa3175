// rewl_sweep.cu -- the fast WL sweep (Sec. 2 of arXiv:1312.3004) for sm_103a.
//
// Same states as the binary64 reference sweep in rewl_kernels.cu, bit for
// bit, organised for a GPU whose FP64 pipe is narrow and slow (GB300: one DADD
// has ~64 cycles of latency and ~2 per clock per SM of throughput):
//
//  * A group of S lanes (S = 2 .. 32, a power of two) owns one walker.  Each
//    lane prepares one of the next S proposals in parallel: Philox block,
//    site, new value, energy change against the lattice at the start of the
//    batch, and an integer acceptance bracket.
//  * Tagged fixed-point shadow of ln g: for the launch, every ln g value v of
//    the walker is also held as F(v) = 2 floor(v / u) + (1 if the floor
//    dropped bits), u = 2^(e_w - 1075), e_w seven binades below the largest
//    value the launch can reach.  The reference test
//    "u_rnd < exp(ln g(E) - ln g(E'))" is decided by D = F(ln g(E')) -
//    F(ln g(E)): D < T_lo (accept) or D >= T_hi (reject), with [T_lo, T_hi)
//    bracketing -ln(u_rnd) with a proven margin.  Only D inside the bracket
//    (about 1e-5 of the decisions) takes the binary64 path exp(a - b) -- the
//    operation the reference does.
//  * ln g(E) += ln f is an integer add on the shadow (ln f = 2^-k is a whole
//    number of half-units; another ln f adds the same whole number of last places
//    inside a binade, see whole_steps); a value whose shadow dropped bits and
//    steps that integers do not give exactly take binary64 adds.
//  * The S proposals of a batch are resolved together, by fixed-point
//    iteration over the whole batch (walker_sweep below).
//  * S = 1: a thread per walker, one step after another (walker_sweep_1).
#include <algorithm>
#include <cstdint>

#include "rewl_internal.cuh"

namespace rewl {
namespace fast {

// Philox4x32-10 with prepared round keys (rk[2 r], rk[2 r + 1] in round r; constant
// operands in lane groups): 20 wide multiplies and 20 three-input logic operations.
__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const uint32_t (&rk)[20]) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned long long a = 0xD2511F53ull * c0, b = 0xCD9E8D57ull * c2;  // (one wide multiply each)
        c0 = (uint32_t)(b >> 32) ^ c1 ^ rk[2 * r];
        c2 = (uint32_t)(a >> 32) ^ c3 ^ rk[2 * r + 1];
        c1 = (uint32_t)b;
        c3 = (uint32_t)a;
    }
    return make_uint4(c0, c1, c2, c3);
}
// C blocks of one key, counter words t[c] (low, high) and c2, interleaved so that
// the rounds of one hide the latency of another.
template <int C>
__device__ __forceinline__ void philox_blocks(const unsigned long long (&t)[C], uint32_t c2, uint32_t c3,
                                              const uint32_t (&rk)[20], uint4 (&x)[C]) {
#pragma unroll
    for (int c = 0; c < C; ++c) x[c] = make_uint4((uint32_t)t[c], (uint32_t)(t[c] >> 32), c2, c3);
#pragma unroll
    for (int r = 0; r < 10; ++r) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const unsigned long long a = 0xD2511F53ull * x[c].x, b = 0xCD9E8D57ull * x[c].z;
            x[c] = make_uint4((uint32_t)(b >> 32) ^ x[c].y ^ rk[2 * r], (uint32_t)b,
                              (uint32_t)(a >> 32) ^ x[c].w ^ rk[2 * r + 1], (uint32_t)a);
        }
    }
}
template <int BITS>
__device__ __forceinline__ int spin_get(const uint32_t *w, int s) {
    if (BITS == 8) return reinterpret_cast<const uint8_t *>(w)[s];
    return (int)((w[s >> 3] >> ((s & 7) << 2)) & 15u);
}
struct Site4 { int r, l, d, u; };
__device__ __forceinline__ Site4 nbrs(int s, int L, int N, uint32_t divL) {
    const int y = (int)__umulhi((uint32_t)s, divL);
    const int x = s - y * L;
    Site4 n;
    n.r = (x == L - 1) ? s - (L - 1) : s + 1;
    n.l = (x == 0) ? s + (L - 1) : s - 1;
    n.d = (y == L - 1) ? s - (N - L) : s + L;
    n.u = (y == 0) ? s + (N - L) : s - L;
    return n;
}

// 53-bit integer of the uniform u = U * 2^-53 (27 bits of hi, 26 of lo).
__device__ __forceinline__ unsigned long long u53(uint32_t hi, uint32_t lo) {
    return ((unsigned long long)(hi >> 5) << 26) | (lo >> 6);
}

// Upper bracket end that never rejects inside a window (in-window |D| < 2^62).
constexpr long long kNoReject = 1LL << 62;
// Shadow value of the bins beyond each end of a window: every proposal there
// has D >= 2^62 >= t_hi and is rejected like an out-of-window move.  The
// padding also covers the bins that a wrong guess inside a batch can reach
// (walker_sweep holds them within it).
constexpr long long kOutside = 0x7fffffffffffffffLL;
constexpr int kPad = kShadowPad;
constexpr long long kMant = (1LL << 52) - 1, kHidden = 1LL << 52;

// floor / ceil of x * 2^k as a 64-bit integer, saturating at 2^61 (x >= 0).
__device__ __forceinline__ long long scaled_floor(float x, int k) {
    if (x <= 0.0f) return 0;
    if (k > 120) return 1LL << 61;
    const float y = x * __int_as_float((k + 127) << 23);
    return y >= 0x1p61f ? (1LL << 61) : __float2ll_rd(y);
}
__device__ __forceinline__ long long scaled_ceil(float x, int k) {
    if (x <= 0.0f) return 0;
    if (k > 120) return 1LL << 61;
    const float y = x * __int_as_float((k + 127) << 23);
    return y >= 0x1p61f ? (1LL << 61) : __float2ll_ru(y);
}

// Bracket of T = -ln(u) / unit, unit = 2^-k: accept for sure if D < t_lo,
// reject for sure if D >= t_hi, where D is within three units of the true
// difference (the shadow's floors and inexact tags, see shadow_of); a lane
// group widens it by kSlack for the roundings inside a batch.  uf = u with relative error <= 2^-23 (24 + 24 bits, one
// rounding; top >= 1 makes the 5 dropped bits <= 2^-24 relative); logf is
// within 1 ulp; so |Lf - (-ln u)| <= (Lf + 1) 2^-22.9, and the margin
// (Lf + 1) 2^-18 leaves a factor > 8 for that, for exp's own error (1 ulp of
// binary64) and for the rounding of Lf -/+ margin.
__device__ __forceinline__ void accept_bracket(unsigned long long U, int k, long long &t_lo, long long &t_hi) {
    const uint32_t top = (uint32_t)(U >> 29);
    if (top == 0u) {  // u < 2^-24: only D < 0 is decided here
        t_lo = 0;
        t_hi = kNoReject;
        return;
    }
    const float uf = fmaf((float)top, 0x1p-24f, (float)((uint32_t)(U >> 5) & 0xffffffu) * 0x1p-48f);
    const float Lf = -logf(uf);
    const float margin = (Lf + 1.0f) * 0x1p-18f;
    const long long lo = scaled_floor(Lf - margin, k) - 3;
    t_lo = lo > 0 ? lo : 0;
    t_hi = scaled_ceil(Lf + margin, k) + 4;
}

// Shadow of a non-negative binary64 bit pattern v in half-units of
// u = 2^(ew - 1075): 2 floor(v / u) + (1 if the floor dropped bits).  A value
// whose tag bit is 0 is exactly (shadow / 2) u.  The exponent of v is at most
// ew + 8, so the shadow stays below 2^62.
__device__ __forceinline__ long long shadow_of(long long v, int ew) {
    if (v == 0) return 0;
    const int s = (int)(v >> 52) - ew;
    const long long mf = (v & kMant) | kHidden;
    if (s >= 0) return (mf << s) << 1;
    if (s <= -53) return 1;
    return ((mf >> -s) << 1) | (long long)((mf & ((1LL << -s) - 1)) != 0);
}

// v / 2^(e - 1075) for the binary64 value v = ln f if that is an integer below
// 2^52 (ln f is an exact multiple of the unit and one step cannot span a
// binade); ok = false otherwise.
__device__ __forceinline__ long long exact_units(long long v, int e, bool &ok) {
    ok = true;
    if (v == 0) return 0;
    const int el = (int)(v >> 52);
    if (el == 0 || e <= 0) {
        ok = false;
        return 0;
    }
    const long long mf = (v & kMant) | kHidden;
    const int s = el - e;
    if (s >= 0) {
        if (s > 9) {
            ok = false;
            return 0;
        }
        const long long r = mf << s;
        ok = r < (1LL << 52);
        return r;
    }
    if (s <= -53 || (mf & ((1LL << -s) - 1)) != 0) {
        ok = false;
        return 0;
    }
    return mf >> -s;
}

// The reference decision in binary64: accept iff d >= 0 or u < exp(d), d = a - b.
// A draw with |u - exp(d)| < 1e-14 is a near tie: counted, and its step index
// kept (the first two of the walker's launch) for the tie log.
struct TieRec {
    unsigned long long n, t[2];
};
__device__ __noinline__ bool exact_accept(long long A, long long B, unsigned long long U, TieRec *tie,
                                          unsigned long long step) {
    const double d = __dsub_rn(__longlong_as_double(A), __longlong_as_double(B));
    if (d >= 0.0) return true;
    const double u = __ull2double_rn(U) * 0x1p-53;
    const double e = exp(d);
    if (fabs(u - e) < 1e-14) {
        if (tie->n < 2ull) tie->t[tie->n] = step;
        tie->n += 1ull;
    }
    return u < e;
}

// The walker's near ties of this launch into the control block and the log.
__device__ __forceinline__ void flush_ties(const State &S, int g, const TieRec &tie) {
    if (!tie.n) return;
    for (unsigned long long i = 0; i < tie.n && i < 2ull; ++i) record_tie(S.ctl, S.tlog, TIE_WL, (unsigned int)g, tie.t[i]);
    if (tie.n > 2ull) atomicAdd(&S.ctl->ties, tie.n - 2ull);
}

template <int S>
__device__ __forceinline__ unsigned group_mask() {
    if (S >= 32) return 0xffffffffu;
    const unsigned lane = threadIdx.x & 31u;
    return ((1u << (S & 31)) - 1u) << (lane & ~(unsigned)(S - 1));
}

// Per-walker scratch of the lane group in shared memory (S > 1 only).
struct Stage {
    uint2 *ring;     // [kAhead S] proposals drawn ahead: site | new value index << 20; -ln u
    uint32_t *pk;    // [2 S] proposal k as touched lanes read it: site | new value << 20; lanes at its mark
    uint32_t *tab;   // [8 S] lanes that start from bin x, at x mod 8 S; zero between uses
    uint8_t *bm;     // [marks] a lane of the batch that proposes a site, at the site's entry (kNoLane: none)
    uint32_t mmask;  // all bits, or entries - 1 where sites share entries (that costs comparisons only)
    // fixed-weight production only
    int *cnt;                 // [q] spins of each value
    unsigned long long *heo;  // [B][n_obins] visits H(E, class) of the walker's window
    int n_obins;
};
// Entries of the conflict marks: one per site up to kMarks sites.
constexpr int kMarks = 8192;
// Lattices in global memory: fewer, so that more walkers fit an SM (q = 10, L = 300,
// 717 windows of 3: all resident at once, 1.05 -> 0.84 ms a round).
constexpr int kMarksFar = 2048;
// Narrow lane groups: a CTA holds 256 / S walkers, and their memory is what limits it.
// Eight lanes take at most 2048 entries (1024 beside lattices in global memory) and
// leave larger lattices packed, two and four take the bytes that a walker is granted
// anyway (make_layout).  q = 10, L = 80, 64 windows of 32, 1000 steps, with an entry
// and a byte per site -> so: 8 lanes 0.90 -> 0.54 ms, 4 lanes 2.34 -> 1.30, 2 lanes 5.5 -> 3.0
// (windows of 16, where all fit: 0.507 -> 0.523).
constexpr int kMarksNarrow = 2048;
constexpr uint32_t kNoLane = 255u;
// ln f from which a lane group counts the batch's own ln f steps in every
// evaluation (about 60 cycles each) instead of leaving the steps they could
// decide, about 500 ln f a batch of 32, to the full comparison (about 1000 cycles).
constexpr double kCountLnf = 0x1p-12;
constexpr int kCrowded = 300;
constexpr int kAhead = 2;  // batches drawn at a time (as fast as 4)
// Half-units by which D in a batch can miss the true difference beyond the
// floors of shadow_of: up to 32 adds on either bin, each rounded by at most
// half a last place (2^8 half-units for values below 2^61 units) and, for an
// ln f that is no whole number of units, known to 2 half-units.
constexpr long long kSlack = 1LL << 15;

struct Tally {
    TieRec tie;
    unsigned long long slow;
    unsigned int acc, seq;
#ifdef REWL_DEBUG_CHECKS
    unsigned int bad = 0;  // failed bounds checks
#endif
};

// Binary64 bits of F * 2^(ew - 1075) for an integer F >= 0 that has at most
// 53 significant bits (a value the shadow holds exactly).
__device__ __forceinline__ long long from_units(long long F, int ew) {
    if (F == 0) return 0;
    const int sh = 11 - __clzll(F);  // top bit position - 52
    const long long m = sh >= 0 ? (F >> sh) : (F << -sh);
    return ((long long)(ew + sh) << 52) | (m & kMant);
}

// 64-bit access to the shadow array by 32-bit shared address.  Lanes of a
// group see each other's writes only across a __syncwarp.
__device__ __forceinline__ long long lds64(uint32_t a) {
    return *reinterpret_cast<const long long *>(__cvta_shared_to_generic(a));
}
__device__ __forceinline__ void sts64(uint32_t a, long long v) {
    *reinterpret_cast<long long *>(__cvta_shared_to_generic(a)) = v;
}

// What both forms of the sweep share: the fixed-point frame of a launch and the
// brackets of -ln u on it.
//
// T = -ln u in 2^-26 (kTiny: u < 2^-24, only D < 0 is decided by it): as
// accept_bracket, in integers -- u from its leading 27 bits and the rest (relative
// error below 2^-23), -ln u from lg2.approx (absolute or relative error at most
// 2^-22, times ln 2) and rounded to 2^-26: together below (Lf + 1) 2^-21; the
// margin is (Lf + 1) 2^-18.
constexpr int kTiny = 0x7fffffff;
__device__ __forceinline__ int minus_ln(uint32_t hi, uint32_t lo) {
    const float uf = fmaf((float)(hi & ~31u), 0x1p-32f, (float)lo * 0x1p-59f);
    float l2;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l2) : "f"(uf));
    return hi < 256u ? kTiny : __float2int_rn(l2 * -0x1.62e43p+25f);  // below 2^31 for u >= 2^-24
}
// Decisions are first taken on the leading 32-bit words of the shadows, in units
// of 2^(32 - k): [blo, blo + bw) are the differences of leading words that do not
// decide (the true difference D 2^-32 lies strictly within 1 of the difference of
// the leading words, kSlack is far below a leading word's unit, and out of the
// window the difference is at least 2^30 - 2, above every T at tsh = 58 - k >= 1).
// small_k: leading_words(k); loose: more units.
__device__ __forceinline__ void lead_bracket(int T, bool small_k, int tsh, int loose, int &blo, uint32_t &bw) {
    const int mg = (T >> 18) + 260;  // (Lf + 1) 2^-18, rounded up
    blo = ((T - mg) >> tsh) - 1 - loose;
    const int up = (int)((uint32_t)T + (uint32_t)mg);  // (kTiny: not used)
    bw = (uint32_t)((up >> tsh) + 3 + loose - blo);
    if (T == kTiny || !small_k) {
        blo = small_k ? -2 : -0x7fffffff;
        bw = 0xfffffff0u;
    }
}

// The exact binary64 value of a bin after `count` more ln f steps of the batch:
// its bits before the batch (kept in lgb when the shadow F dropped bits), then
// the reference's adds one by one.
__device__ __noinline__ long long exact_steps(long long F, const long long *lgb, int b, int ew, double lnf, int count) {
    double a = __longlong_as_double((F & 1) ? lgb[b] : from_units(F >> 1, ew));
    for (int i = 0; i < count; ++i) a = __dadd_rn(a, lnf);
    return __double_as_longlong(a);
}

// The shadow after c ln f steps from F where integers give the reference's
// binary64 sums although the plain add does not apply; false where they do not.
// F2: on entry F + c ln f in whole units.
//  - ln f a multiple of the largest last place (int_add): only a step into the
//    next binade can round, and only if the sum has bits below that binade's last
//    place; the steps leave those bits as they are, so the last sum shows them.
//  - another ln f (the 1/t rule's bins / steps): inside a binade every step adds
//    the same whole number of last places, ln f rounded to them, unless ln f lies
//    half-way between two (then the sum's parity decides).
__device__ __forceinline__ bool whole_steps(long long F, int c, long long LNF, int ew, bool int_add, long long &F2) {
    if (F & 1) return false;
    if (int_add) {
        const int sh = 11 - __clzll(F2 >> 1);
        return sh <= 0 || ((F2 >> 1) & ((1LL << sh) - 1)) == 0;
    }
    const int sh = 11 - __clzll(F >> 1);  // the last place of F's binade is 2^sh units
    if (F == 0 || sh < 0 || LNF < (1LL << 52)) return false;
    const int s = sh + ew - (int)(LNF >> 52);  // and 2^s last places of ln f
    const long long mf = (LNF & kMant) | kHidden;
    long long inc = 0;
    if (s >= 0 && s <= 54) {
        const long long rest = mf & ((1LL << s) - 1), half = s > 0 ? 1LL << (s - 1) : 1;
        if (rest == half) return false;
        inc = (mf >> s) + (rest > half ? 1 : 0);
    } else if (s < 0) {
        if (s < -8) return false;
        inc = mf << -s;
    }
    if (inc >= 1LL << 52) return false;
    F2 = F + ((inc << sh) * c << 1);
    return __clzll(F2) == __clzll(F);
}

// One lane per walker, its state in global memory: the steps one after another,
// the next proposal drawn (and its spins read) while the present step waits for
// its ln g shadow; a flip of the present step is put into the words read.
//
// What bounds it: a step's chain of latencies (a read that misses L1 in some lane,
// the random words, the decision: 1100 cycles with a warp per scheduler) and, with
// three warps per scheduler, its 280 instructions (issue 44 % busy).  Hence
// leading-word decisions, brackets in 32-bit integers, round keys kept in
// registers, the proposal held as the five words of its spins (a plain store to
// the lattice, which the thread owns, and one change per word for a flip, taken
// over only when the proposal is looked at: nothing waits for the reads in the
// step that issues them) and the current bin's shadow and visits in registers
// until the walker leaves the bin.  The passes over all bins before and after the
// steps are taken by the warp together, one walker after another, so that the
// lanes' loads lie side by side (3.1 -> 1.0 ms on 2048 instances; so a walker's ln g
// has more than one name, and lgb is not __restrict__).  Every thread
// of a warp calls, live or not.  10^4 steps: 2048 instances (56,784 walkers)
// 16.1 -> 8.4 ms a round (8-bit spins 9.1), 700 instances 7.9 -> 5.5 ms with words
// instead of spins.
// Lattices in shared memory (a word of each lane side by side) were slower, 10.2
// and 6.9 ms: less L1 for the shadows and fewer warps; so were reads two
// steps ahead and both possible shadow reads of the next step issued early.
struct Slow1 {  // what the rare parts of a step need
    long long *lgb;
    double lnf;
    int ew, k;
    bool small_k;
    unsigned int slow = 0, seq = 0;
};
// The decision with all 64 bits, then in binary64; r: the step's random words.
__device__ __noinline__ bool decide_1(Slow1 &s, long long AF, long long BF, int a, int b, int T, uint4 r, TieRec *tie,
                                      unsigned long long t) {
    long long blo, bhi;
    if (s.small_k && T != kTiny) {
        const int mg = (T >> 18) + 260;
        blo = (long long)(T - mg) << (s.k - 26);
        bhi = (long long)(T + mg) << (s.k - 26);
    } else {
        accept_bracket(u53(r.z, r.w), s.k, blo, bhi);
    }
    const long long D = BF - AF;
    if (D < blo - kSlack) return true;
    if (D >= bhi + kSlack) return false;
    s.slow += 1;
    return exact_accept(exact_steps(AF, s.lgb, a, s.ew, 0.0, 0), exact_steps(BF, s.lgb, b, s.ew, 0.0, 0), u53(r.z, r.w), tie,
                        t);
}
__device__ __noinline__ long long add_1(Slow1 &s, long long F, int b, long long F2, bool int_add) {
    if (whole_steps(F, 1, __double_as_longlong(s.lnf), s.ew, int_add, F2)) return F2;
    s.seq += 1;
    const long long v = exact_steps(F, s.lgb, b, s.ew, s.lnf, 1);
    s.lgb[b] = v;
    return shadow_of(v, s.ew);
}

constexpr int kInFlight = 8;  // loads of such a pass in flight per lane

template <int BITS, bool GLOBAL>
__device__ void walker_sweep_1(const Model &M, uint32_t *__restrict__ lat, long long *lgb, long long *lgf,
                               uint32_t *__restrict__ hg, int g, int lo, double lnf, int &E_io,
                               unsigned long long &t_io, Tally &tally, bool live) {
    const int N = M.N, L = M.L;
    const uint32_t qm1 = (uint32_t)(M.q - 1), divL = M.divL;
    const long long LNF = __double_as_longlong(lnf);
    if (GLOBAL) {
        __builtin_assume(__isGlobal(lat));
        __builtin_assume(__isGlobal(lgf));
    }
    __builtin_assume(__isGlobal(lgb));
    __builtin_assume(__isGlobal(hg));
    const int lane = (int)(threadIdx.x & 31u);
    const unsigned lanes = __ballot_sync(0xffffffffu, live);
    auto of = [&](auto *p, int w) {  // lane w's pointer
        return reinterpret_cast<decltype(p)>(__shfl_sync(0xffffffffu, (unsigned long long)p, w));
    };
    long long vmax = 0;
    for (unsigned rest = lanes; rest; rest &= rest - 1u) {
        const int w = __ffs((int)rest) - 1, B = __shfl_sync(0xffffffffu, M.B, w);
        const long long *v = of(lgb, w);
        __builtin_assume(__isGlobal(v));
        long long top = 0;
        for (int b0 = lane; b0 < B; b0 += 32 * kInFlight) {
            long long x[kInFlight];
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) x[i] = b0 + 32 * i < B ? v[b0 + 32 * i] : 0;
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) top = max(top, x[i]);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (lane == w) vmax = top;
    }
    const double reach = __dadd_rn(__longlong_as_double(vmax), __dmul_rn((double)M.K, lnf));
    Slow1 rare;
    rare.lgb = lgb;
    rare.lnf = lnf;
    rare.ew = max(1, (int)(__double_as_longlong(reach) >> 52) - 7);
    rare.k = 1076 - rare.ew;
    rare.small_k = leading_words(rare.k);
    const bool small_k = rare.small_k;
    const int tsh = small_k ? 58 - rare.k : 0;
    for (unsigned rest = lanes; rest; rest &= rest - 1u) {
        const int w = __ffs((int)rest) - 1, B = __shfl_sync(0xffffffffu, M.B, w), e = __shfl_sync(0xffffffffu, rare.ew, w);
        const long long *v = of(lgb, w);
        long long *f = of(lgf, w);
        __builtin_assume(__isGlobal(v));
        if (GLOBAL) __builtin_assume(__isGlobal(f));
        for (int b0 = lane; b0 < B; b0 += 32 * kInFlight) {
            long long x[kInFlight];
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) x[i] = b0 + 32 * i < B ? v[b0 + 32 * i] : 0;
#pragma unroll
            for (int i = 0; i < kInFlight; ++i)
                if (b0 + 32 * i < B) f[b0 + 32 * i] = shadow_of(x[i], e);
        }
        if (lane < kPad) {
            f[-1 - lane] = kOutside;
            f[B + lane] = kOutside;
        }
    }
    __syncwarp();
    bool addF;
    const long long incU = exact_units(LNF, rare.ew, addF);
    const unsigned long long incF = (unsigned long long)(addF ? incU << 1 : shadow_of(LNF, rare.ew) & ~1LL);
    const bool int_add = addF && (incU & 255) == 0;
    uint32_t rk[20];
#pragma unroll
    for (uint32_t r = 0; r < 10; ++r) {
        rk[2 * r] = M.key0 + r * 0x9E3779B9u;
        rk[2 * r + 1] = M.key1 + r * 0xBB67AE85u;
    }
#pragma unroll
    for (int r = 0; r < 20; ++r) asm("" : "+r"(rk[r]));  // kept, not added up again in every block

    struct Prop {
        int site, v, T, blo;
        uint32_t bw, here, wr, wl, wd, wu;  // the words that hold the site and its neighbours
        Site4 nb;
    };
    // sites as bit offsets in the lattice: word s >> 5, bit s (mod 32, as a funnel shift takes it)
    auto same = [](int a, int b) { return (a >> 5) == (b >> 5); };
    auto field = [](uint32_t w, int s) { return (int)(__funnelshift_r(w, 0u, (uint32_t)s) & ((1u << BITS) - 1u)); };
    const int row = L * BITS, all = N * BITS;
    auto random = [&](unsigned long long t) {
        return philox((uint32_t)t, (uint32_t)(t >> 32), (uint32_t)g, DOM_WL, rk);
    };
    auto draw = [&](unsigned long long t, Prop &p) {
        const uint4 r = random(t);
        const int s = (int)__umulhi(r.x, (uint32_t)N), y = (int)__umulhi((uint32_t)s, divL), x = s - y * L;
        p.site = s * BITS;
        p.v = (int)__umulhi(r.y, qm1);
        p.nb.r = p.site + (x == L - 1 ? BITS - row : BITS);  // (nbrs)
        p.nb.l = p.site + (x == 0 ? row - BITS : -BITS);
        p.nb.d = p.site + (y == L - 1 ? row - all : row);
        p.nb.u = p.site + (y == 0 ? all - row : -row);
        p.here = lat[p.site >> 5];
        p.wr = lat[p.nb.r >> 5];
        p.wl = lat[p.nb.l >> 5];
        p.wd = lat[p.nb.d >> 5];
        p.wu = lat[p.nb.u >> 5];
        p.T = minus_ln(r.z, r.w);
        lead_bracket(p.T, small_k, tsh, 0, p.blo, p.bw);
    };
    if (live) {
    // The current bin's shadow AF and its visits since the walker came are kept
    // in registers, and written when the walker leaves the bin.
    int Eo = E_io - lo;
    long long AF = lgf[REWL_IDX(Eo, 0, M.B, tally.bad)];
    uint32_t visits = 0;
    unsigned int nacc = 0;
    unsigned long long t = t_io;
    const unsigned long long t_end = t_io + (unsigned long long)M.K;
    // The next proposal is drawn and its words read while a step waits for its
    // ln g shadow; it takes over the step's flip when it is looked at.
    auto flipped = [&](Prop &p, int site, uint32_t x) {
        p.here ^= same(p.site, site) ? x : 0u;
        p.wr ^= same(p.nb.r, site) ? x : 0u;
        p.wl ^= same(p.nb.l, site) ? x : 0u;
        p.wd ^= same(p.nb.d, site) ? x : 0u;
        p.wu ^= same(p.nb.u, site) ? x : 0u;
    };
    int fsite = 0;  // the last step's flip: its site, and its change of the word (0: none)
    uint32_t fx = 0;
    auto step = [&](Prop &cp, Prop &n1) {
        flipped(cp, fsite, fx);
        const int curs = field(cp.here, cp.site);
        const int sr = field(cp.wr, cp.nb.r), sl = field(cp.wl, cp.nb.l);
        const int sd = field(cp.wd, cp.nb.d), su = field(cp.wu, cp.nb.u);
        const int nw = cp.v + (cp.v >= curs);
        const int dE = (int)(sr == curs) + (int)(sl == curs) + (int)(sd == curs) + (int)(su == curs) -
                       (int)(sr == nw) - (int)(sl == nw) - (int)(sd == nw) - (int)(su == nw);
        const int En = Eo + dE;
        long long BF = AF;  // (a proposal that keeps the energy reads nothing)
        if (dE != 0) BF = lgf[REWL_IDX(En, -kPad, M.B + kPad, tally.bad)];  // beyond the window: kOutside
        draw(t + 1ull, n1);  // (past the last step: drawn, never taken)
        const int D = (int)(BF >> 32) - (int)(AF >> 32);
        bool acc = D < cp.blo;
        if ((uint32_t)(D - cp.blo) < cp.bw)  // the leading words do not decide
            acc = decide_1(rare, AF, BF, REWL_IDX(Eo, 0, M.B, tally.bad), REWL_IDX(En, 0, M.B, tally.bad), cp.T, random(t),
                           &tally.tie, t);
        const int Eb = acc ? En : Eo;
        const long long cur = acc ? BF : AF;
        if (Eb != Eo) {  // leaving the bin: its value and visits go to memory
            lgf[REWL_IDX(Eo, 0, M.B, tally.bad)] = AF;
            atomicAdd(&hg[REWL_IDX(Eo, 0, M.B, tally.bad)], visits);  // (result not used: the walker does not wait)
            visits = 0;
        }
        ++visits;
        Eo = Eb;
        AF = (long long)((unsigned long long)cur + incF);  // ln g(E) += ln f
        const uint32_t hc = (uint32_t)((unsigned long long)cur >> 32), h2 = (uint32_t)((unsigned long long)AF >> 32);
        if (!int_add || (cur & 1) || (h2 ^ hc) > hc) {
            const int sh = 11 - __clzll(AF >> 1);  // (whole_steps, its usual case)
            if (!int_add || (cur & 1) || (sh > 0 && ((AF >> 1) & ((1LL << sh) - 1)) != 0))
                AF = add_1(rare, cur, REWL_IDX(Eb, 0, M.B, tally.bad), AF, int_add);
        }
        fsite = cp.site;
        fx = acc ? __funnelshift_l(0u, (uint32_t)(curs ^ nw), (uint32_t)cp.site) : 0u;
        if (acc) lat[cp.site >> 5] = cp.here ^ fx;
        nacc += acc;
        return ++t == t_end;
    };
    Prop a, b;
    draw(t, a);
    while (!step(a, b) && !step(b, a)) {
    }
    lgf[Eo] = AF;
    atomicAdd(&hg[Eo], visits);
    t_io = t_end;
    E_io = Eo + lo;
    tally.acc += nacc;
    tally.slow += rare.slow;
    tally.seq += rare.seq;
    }
    __syncwarp();
    for (unsigned rest = lanes; rest; rest &= rest - 1u) {
        const int w = __ffs((int)rest) - 1, B = __shfl_sync(0xffffffffu, M.B, w), e = __shfl_sync(0xffffffffu, rare.ew, w);
        const long long *f = of(lgf, w);
        long long *v = of(lgb, w);
        __builtin_assume(__isGlobal(v));
        if (GLOBAL) __builtin_assume(__isGlobal(f));
        for (int b0 = lane; b0 < B; b0 += 32 * kInFlight) {
            long long x[kInFlight];
#pragma unroll
            for (int i = 0; i < kInFlight; ++i) x[i] = b0 + 32 * i < B ? f[b0 + 32 * i] : 1;
#pragma unroll
            for (int i = 0; i < kInFlight; ++i)
                if (!(x[i] & 1)) v[b0 + 32 * i] = from_units(x[i] >> 1, e);
        }
    }
}

// S > 1 lanes per walker: batches of S steps, lane j owning step j.
//
// A step's outcome depends on the earlier steps of its batch only through the
// bin they have led to, the ln f steps they have added to the two bins it
// compares, and the spins they have flipped around its site.  So every lane
// evaluates its step under the present decisions of the lanes before it, all
// at once, and the evaluations are repeated until no decision changes.  Such a
// fixed point is unique and is the serial result: step 0 depends on nothing,
// and if steps 0 .. j - 1 agree with the serial run, so does step j.  Each
// evaluation makes at least one more leading step final, so at most S + 1 are
// needed; the decisions depend on each other weakly, and the measured number
// per batch of 32 is 1.0 .. 1.7 at a late ln f and 2 .. 7 at ln f = 1,
// confirming evaluation included.
//
// What bounds it: the latency of one dependent chain per walker, so every part is
// chosen for its latency; with 7 walkers per SM the instructions count as well
// (60 more in an evaluation cost 20 %).  At ln f = 1 a batch of 32 takes 580 warp
// instructions (18 a step), the SM issues in 35 % of its cycles, and of the
// cycles between two instructions of a warp 1.5 are fixed latencies, 1.3 shared
// memory and the vote units.  Measured on GB300, in cycles with their use:
// popcount 24 (four of them 56), ballot 17 (four 33), match 41 and 11 more per
// distinct value, shared load 34, store-then-load 42, atomic-then-load 99,
// leading-zero count 27, a branch on a vote about 45.  Hence ballots and plain
// stores instead of shared atomics, one branch per evaluation, flips without
// branches, and the random numbers of two batches at a time (four: no faster, and
// more shared memory).  q = 10, L = 80, 1024 walkers, 10^4 steps each, the
// sweep alone: 1.10 -> 0.57 ms in the first rounds (ln f = 1) and 1.03 -> 0.39 ms
// at ln f = 2^-20, against the step trees that were here before (the decisions of
// the next five steps at a time, 275 cycles a step).
//
//  * The bin before step j: the batch's start plus the accepted energy changes
//    of the lanes before it; from four ballots (the bit planes of the changes,
//    two's complement) and popcounts instead of a five-step shuffle scan.
//  * ln f steps added inside the batch: at a large ln f every evaluation counts
//    them, otherwise only when one of the at most j that precede step j could
//    decide.  The steps before j that ended in a bin are the lanes 1 .. j that
//    start from it: from the bit planes of the lanes' bins, by ballots.
//  * Flips: a byte per site names a lane that proposes it, and every lane reads
//    its own site's and those of its four neighbours; the energy change of a
//    lane that others touch is recomputed from the spins at the
//    start of the batch and the flips of the accepted touching lanes, in order,
//    whenever those change.
//  * A draw inside its bracket is settled when everything before it is final:
//    the reference's binary64 test on the exact values, then the lane keeps
//    that decision.
//  * Commit: one add of count x ln f per distinct bin (binary64 adds one by one
//    where the integer add is not exact), one histogram add per distinct bin,
//    one store per flipped site.
//
// PROD, fixed-weight production (Sec. 3.2: once g(E) is known, configurations
// are sampled with the fixed weights 1/g(E) and distributions H(E, O)
// recorded): ln f = 0 and ln g stays, any sign; the shadow is
// floor((v - min) 2^k), and the binary64 values themselves settle what it does
// not decide.  After every step H(E, O) counts the bin and the class of the
// majority count O = max_v #{i : s_i = v}: for each value v, two ballots give
// the steps that gain and lose a spin of it, popcounts its number after each
// step.  Same workload, 64 classes: 8.4 -> 0.65 ms a round (1024 walkers, reads included) against one thread per
// walker (1690 cycles a step: the binary64 decision and the counts on one chain).
template <int BITS, int S, bool PROD = false>
__device__ __forceinline__ void walker_sweep(const Model &M, uint32_t *__restrict__ lat, long long *__restrict__ lgb,
                                             long long *lgf, uint32_t *__restrict__ hg, const Stage &st, int g, int lo,
                                             double lnf, int &E_io, unsigned long long &t_io, Tally &tally) {
    static_assert(S > 1, "walker_sweep_1");
    const int j = (int)(threadIdx.x & (unsigned)(S - 1));
    const unsigned gm = group_mask<S>();
    const unsigned gbase = S == 32 ? 0u : threadIdx.x & 31u & ~(unsigned)(S - 1);
    const unsigned bit = 1u << j, lt = bit - 1u, le = lt | bit;  // lane j; the lanes before it; both
    const unsigned le1 = le & ~1u;  // (the bins before steps 1 .. j are those after steps 0 .. j - 1)
    const int N = M.N, L = M.L;
    constexpr int per = 32 / BITS;  // sites per lattice word
    const uint32_t qm1 = (uint32_t)(M.q - 1);
    const long long LNF = __double_as_longlong(lnf);
    auto ballot = [&](bool p) { return __ballot_sync(gm, p) >> gbase; };

    // ---- fixed-point frame of this launch --------------------------------------
    int k;  // half-unit = 2^-k
    int ew = 0;
    bool int_add = false, blind = false;  // blind: no shadow (values that are no numbers), every step in binary64
    unsigned long long incF = 0;          // ln f in half-units
    if constexpr (PROD) {
        double vmin = __longlong_as_double(lgb[0]), vmax = vmin;
        bool finite = true;
        for (int b = j; b < M.B; b += S) {
            const double v = __longlong_as_double(lgb[b]);
            finite = finite && fabs(v) < 0x1p1000;
            vmin = fmin(vmin, v);
            vmax = fmax(vmax, v);
        }
#pragma unroll
        for (int o = 1; o < S; o <<= 1) {
            vmin = fmin(vmin, __shfl_xor_sync(gm, vmin, o));
            vmax = fmax(vmax, __shfl_xor_sync(gm, vmax, o));
        }
        blind = !__all_sync(gm, finite);
        // shadows below 2^61; v - vmin is off by at most 2^-53 of it, 2^8 half-units
        const int e = (int)(__double_as_longlong(__dsub_rn(vmax, vmin)) >> 52) - 1022;  // vmax - vmin < 2^e
        k = min(61 - e, 57);
        blind = blind || k < -100;  // (draws scaled by 2^k are kept in single precision)
        for (int b = j; b < M.B; b += S) {
            const double d = __dsub_rn(__longlong_as_double(lgb[b]), vmin);
            lgf[b] = blind ? 0 : __double2ll_rd(d * __longlong_as_double((long long)(k + 1023) << 52));
        }
    } else {
        long long vmax = 0;
        for (int b = j; b < M.B; b += S) vmax = max(vmax, lgb[b]);
#pragma unroll
        for (int o = 1; o < S; o <<= 1) vmax = max(vmax, __shfl_xor_sync(gm, vmax, o));
        const double reach = __dadd_rn(__longlong_as_double(vmax), __dmul_rn((double)M.K, lnf));
        // values stay below 2^(e_reach + 2 - 1023): below 2^61 units of
        // u = 2^(ew - 1075), shadows (half-units) below 2^62
        ew = max(1, (int)(__double_as_longlong(reach) >> 52) - 7);
        k = 1076 - ew;
        for (int b = j; b < M.B; b += S) lgf[b] = shadow_of(lgb[b], ew);
        bool addF;
        const long long incU = exact_units(LNF, ew, addF);
        // (ln f rounded down to whole units where it is none)
        incF = (unsigned long long)(addF ? incU << 1 : shadow_of(LNF, ew) & ~1LL);
        // every integer step inside a binade is exact when ln f is a multiple of the
        // largest last place (2^8 units for values below 2^61 units)
        int_add = addF && (incU & 255) == 0;
    }
    for (int p = j; p < kPad; p += S) {
        lgf[-1 - p] = kOutside;
        lgf[M.B + p] = kOutside;
    }
    // Decisions are first taken on the leading 32-bit words of the shadows, in
    // units of 2^(32 - k); where those cannot decide, on all 64 bits (see
    // `bracket` below).
    const bool small_k = __all_sync(gm, leading_words(k) && !blind);
    const int tsh = small_k ? 58 - k : 0;
    // At a large ln f many evaluations have to count the batch's own ln f steps:
    // they all do, in leading words (loose: with up to 32 units for what those cut off).
    const bool heavy = !PROD && __all_sync(gm, small_k && lnf >= kCountLnf);
    const int incH = (int)(incF >> 32), loose = heavy && (uint32_t)incF != 0u ? 32 : 0;
    // ln f steps that can precede step j, in leading words (rounded up)
    const uint32_t kinc = heavy || !small_k ? 0u : (uint32_t)((incF * (unsigned)j + 0xffffffffull) >> 32);
    __syncwarp(gm);

    const uint32_t pbase = (uint32_t)__cvta_generic_to_shared(lgf);
    const uint32_t tbase = (uint32_t)__cvta_generic_to_shared(st.tab);
    const uint32_t mbase = (uint32_t)__cvta_generic_to_shared(st.bm);
    const int pmin = (int)pbase - (kPad - 4) * 8, pmax = (int)pbase + (M.B + kPad - 5) * 8;
    uint32_t pcur = pbase + (uint32_t)(E_io - lo) * 8u;  // shared address of the current bin's shadow
    unsigned int nacc = 0, nseq = 0;
    auto lds32 = [](uint32_t a) { return *reinterpret_cast<const uint32_t *>(__cvta_shared_to_generic(a)); };
    auto lead = [&](uint32_t a) { return (int)lds32(a + 4u); };  // leading word of a shadow
    auto sts32 = [](uint32_t a, uint32_t v) { *reinterpret_cast<uint32_t *>(__cvta_shared_to_generic(a)) = v; };
    // the entry of tab that stands for the bin whose shadow is at shared address a
    auto tab_at = [&](uint32_t a) { return tbase + ((a >> 1) & (uint32_t)(32 * S - 4)); };
    // Lanes whose x has the low seven bits of this lane's y, from bit planes by
    // ballots.  Bins a path of one batch visits, or proposes from its second step
    // on, are less than 128 apart.
    auto planes = [&](uint32_t x, unsigned (&p)[7]) {
#pragma unroll
        for (int b = 0; b < 7; ++b) p[b] = ballot((x >> b) & 1u);
    };
    auto equal = [&](const unsigned (&p)[7], uint32_t y) {
        unsigned eq = ~0u;
#pragma unroll
        for (int b = 0; b < 7; ++b) eq &= (y >> b) & 1u ? p[b] : ~p[b];
        return eq;
    };
    auto mark_at = [&](int s) { return mbase + ((uint32_t)s & st.mmask); };
    const bool shared_marks = st.mmask != 0xffffffffu;
    // On small lattices most batches propose some site twice: the lanes of each
    // site are matched ahead, with the draws (300 cycles for about 25 sites, under
    // the waits of a batch); elsewhere they are compared one by one when it occurs.
    const bool crowded = N <= kCrowded;
    auto lds8 = [](uint32_t a) { return (uint32_t)*reinterpret_cast<const uint8_t *>(__cvta_shared_to_generic(a)); };
    auto sts8 = [](uint32_t a, uint32_t v) { *reinterpret_cast<uint8_t *>(__cvta_shared_to_generic(a)) = (uint8_t)v; };

    // The part of a proposal that needs no state: site, neighbours, new value,
    // T = -ln u and the leading words' bracket of it.
    struct Draw {
        int site, v, T, blo;
        uint32_t bw;
        unsigned twins;  // lanes that propose the same site (found ahead on small lattices)
        Site4 nb;
    };
    auto random = [&](unsigned long long t) {
        return philox((uint32_t)t, (uint32_t)(t >> 32), (uint32_t)g, DOM_WL, M.rk);
    };
    // The random part of the next kAhead batches (from step t on), into the ring.
    auto draw_ahead = [&](unsigned long long t0) {
        unsigned long long t[kAhead];
        uint4 r[kAhead];
#pragma unroll
        for (int c = 0; c < kAhead; ++c) t[c] = t0 + (unsigned long long)(c * S + j);
        philox_blocks<kAhead>(t, (uint32_t)g, DOM_WL, M.rk, r);
#pragma unroll
        for (int c = 0; c < kAhead; ++c) {
            const int T = minus_ln(r[c].z, r[c].w);
            st.ring[c * S + j] = make_uint2(__umulhi(r[c].x, (uint32_t)N) | __umulhi(r[c].y, qm1) << 20, (uint32_t)T);
        }
    };
    auto drawn = [&](int c) {  // this lane's proposal of batch c of the ring
        const uint2 w = st.ring[c * S + j];
        Draw d;
        d.site = (int)(w.x & 0xfffffu);
        d.v = (int)(w.x >> 20);
        d.T = (int)w.y;
        d.nb = nbrs(d.site, L, N, M.divL);
        d.twins = bit;
        if (crowded) d.twins = __match_any_sync(gm, d.site) >> gbase;
        lead_bracket(d.T, small_k, tsh, loose, d.blo, d.bw);
        return d;
    };
    // the same bracket in half-units, from step t's draw
    auto bracket = [&](int T, unsigned long long t, long long &blo, unsigned long long &width) {
        long long bhi;
        if (small_k && T != kTiny) {
            const int mg = (T >> 18) + 260;
            blo = (long long)(T - mg) << (k - 26);
            bhi = (long long)(T + mg) << (k - 26);
        } else {
            const uint4 r = random(t);
            accept_bracket(u53(r.z, r.w), k, blo, bhi);
            if (PROD && blind) {  // every shadow in the window is 0: nothing decided
                blo = -(1LL << 61);
                bhi = 1LL << 61;
            }
        }
        width = (unsigned long long)(bhi - blo) + 2ull * kSlack;
        blo -= kSlack;
    };

    draw_ahead(t_io);
    Draw next = drawn(0);  // (a lane reads back its own entries only)
    int ahead = 0;         // the batch of the ring that `next` holds
    int cur0, sr0, sl0, sd0, su0;
    auto read_spins = [&]() {
        cur0 = spin_get<BITS>(lat, next.site);
        sr0 = spin_get<BITS>(lat, next.nb.r);
        sl0 = spin_get<BITS>(lat, next.nb.l);
        sd0 = spin_get<BITS>(lat, next.nb.d);
        su0 = spin_get<BITS>(lat, next.nb.u);
    };
    read_spins();
    sts8(mark_at(next.site), (uint32_t)j);
    __syncwarp(gm);
    const int qlo = PROD ? (N + M.q - 1) / M.q : 0;  // the smallest majority count
    const uint32_t span = (uint32_t)(N - qlo + 1);
    const bool narrow = PROD && (unsigned long long)span * (unsigned)st.n_obins < 0x100000000ull;
    int nmax = 0;
    for (int v = 0; PROD && v < M.q; ++v) nmax = max(nmax, st.cnt[v]);

    long long left = M.K;
    for (;;) {
        const int n = left < S ? (int)left : S;
        // ---- lane j prepares proposal t + j against the lattice as it is --------
        // (its spins were read, and its site marked, at the end of the last batch)
        Draw d = next;
        const int site = d.site;
        const Site4 nb = d.nb;
        int cur = cur0, nw = d.v + (d.v >= cur0);
        int dE = (int)(sr0 == cur) + (int)(sl0 == cur) + (int)(sd0 == cur) + (int)(su0 == cur) - (int)(sr0 == nw) -
                 (int)(sl0 == nw) - (int)(sd0 == nw) - (int)(su0 == nw);
        // earlier lanes whose flip would change this proposal
        unsigned touch = 0u, twins = d.twins;  // ... ; lanes that propose the same site
        unsigned t0 = 0u, tr = 0u, tl = 0u, td = 0u, tu = 0u;  // touch, by the site touched
        const uint32_t m0 = lds8(mark_at(site)), mr = lds8(mark_at(nb.r)), ml = lds8(mark_at(nb.l)), md = lds8(mark_at(nb.d)), mu = lds8(mark_at(nb.u));
        if (n < S && j >= n) {  // past the launch's last step: never accepted
            d.blo = (int)0x80000000;
            d.bw = 0u;
        }
        // with up to kinc ln f steps on either side (kTiny: already everything from -2 up)
        const int blo2 = d.blo - (int)kinc;
        const uint32_t bw2 = d.bw == 0xfffffff0u || d.bw == 0u ? d.bw : d.bw + 2u * kinc;
        // first evaluation: as if every step started from the batch's first bin
        const int D0 = lead(pcur + (uint32_t)(dE * 8)) - lead(pcur);
        // bit planes of the energy changes (two's complement)
        unsigned q0 = ballot(dE & 1), q1 = ballot(dE & 2), q2 = ballot(dE & 4), q3 = ballot(dE & 8);
        unsigned A = ballot(D0 < d.blo);  // the steps that accept, as presently known
        // (without two lanes at one entry every mark names the only lane there)
        unsigned fl = ballot(m0 != (uint32_t)j || min(min(mr, ml), min(md, mu)) < (uint32_t)j);
        // the state-free part of the next batch's proposals: independent
        // instructions for the waits of this batch
        if (++ahead == kAhead) {
            draw_ahead(t_io + S);
            ahead = 0;
        }
        next = drawn(ahead);
        __syncwarp(gm);
        sts8(mark_at(site), kNoLane);
        if (fl) {
            unsigned there = twins;  // lanes at this site's entry
            for (unsigned rest = crowded ? 0u : ballot(m0 != (uint32_t)j); rest;) {
                const int f = __ffs((int)rest) - 1;
                const int sf = __shfl_sync(gm, site, f, S);
                const unsigned t = ballot(site == sf);
                const unsigned e = shared_marks ? ballot(mark_at(site) == mark_at(sf)) : t;
                if (t & bit) twins = t;
                if (e & bit) there = e;
                rest &= ~t;
            }
            st.pk[j] = (uint32_t)site | ((uint32_t)nw << 20);
            st.pk[S + j] = there;
            __syncwarp(gm);
            auto at_mark = [&](uint32_t id) {  // (loads without branches)
                const unsigned x = st.pk[S + (id & (S - 1))] & lt;
                return id != kNoLane ? x : 0u;
            };
            t0 = twins & lt;
            tr = at_mark(mr);
            tl = at_mark(ml);
            td = at_mark(md);
            tu = at_mark(mu);
            if (shared_marks) {  // keep the lanes that propose the site itself
                const unsigned all = tr | tl | td | tu;
                tr = tl = td = tu = 0u;
                for (unsigned rest = all; rest; rest &= rest - 1u) {
                    const int ps = (int)(st.pk[__ffs((int)rest) - 1] & 0xfffffu);
                    const unsigned low = rest & (0u - rest);
                    tr |= ps == nb.r ? low : 0u;
                    tl |= ps == nb.l ? low : 0u;
                    td |= ps == nb.d ? low : 0u;
                    tu |= ps == nb.u ? low : 0u;
                }
            }
            touch = t0 | tr | tl | td | tu;
            fl = ballot(touch != 0u);
        }

        // ---- evaluations until nothing changes -----------------------------------
        unsigned moved = 0u, last = 0u;
        uint32_t pre, to;  // the bins step j compares, as addresses of their shadows
        // energy changes under the present flips of the touching lanes, where those changed
        auto reflip = [&]() {
            const unsigned ta = touch & A;
            const bool need = ta != last || (touch & moved) != 0u;
            moved = 0u;
            if (ballot(need)) {
                __syncwarp(gm);
                // a site's spin: the last accepted flip of it, or as read (for every
                // lane, without branches: the five chains side by side)
                auto flip = [&](unsigned t, int was) {
                    const unsigned a = t & A;
                    const int x = (int)(st.pk[(31 - __clz((int)a)) & (S - 1)] >> 20);
                    return a ? x : was;
                };
                const int c = flip(t0, cur0), sr = flip(tr, sr0), sl = flip(tl, sl0), sd = flip(td, sd0), su = flip(tu, su0);
                last = ta;
                cur = c;
                const int w = d.v + (d.v >= c);
                const bool ch = w != nw;
                nw = w;
                dE = (int)(sr == c) + (int)(sl == c) + (int)(sd == c) + (int)(su == c) - (int)(sr == w) - (int)(sl == w) -
                     (int)(sd == w) - (int)(su == w);
                __syncwarp(gm);
                if (ch) st.pk[j] = (uint32_t)site | ((uint32_t)nw << 20);
                moved = ballot(ch);
                q0 = ballot(dE & 1);
                q1 = ballot(dE & 2);
                q2 = ballot(dE & 4);
                q3 = ballot(dE & 8);
            }
        };
        // the bins of step j under the decisions A (a wrong guess can lie outside the window)
        auto place = [&]() {
            const uint32_t p = pcur + 8u * __popc(q0 & A & lt) + 16u * __popc(q1 & A & lt) +
                               32u * __popc(q2 & A & lt) - 64u * __popc(q3 & A & lt);
            pre = (uint32_t)max(pmin, min((int)p, pmax));
            to = pre + (uint32_t)(dE * 8);
        };
        // ln f steps the path adds to step j's new bin before it, and to its old
        // one: the lanes 1 .. j that start from them
        auto counted = [&](int &cA, int &cB) {
            unsigned p[7];
            planes((pre - pcur) >> 3, p);
            cA = __popc(equal(p, (pre - pcur) >> 3) & le1);
            cB = __popc(equal(p, (to - pcur) >> 3) & le1);
        };
        // the same for every evaluation at a large ln f: in a fifth of the
        // instructions, by a match (11 cycles per distinct bin) and a table
        auto counted_now = [&]() {
            if (S == 2) return j == 1 ? (int)(to == pre) - 1 : 0;  // (the second step starts from the first one's bin)
            const unsigned here = __match_any_sync(gm, pre) >> gbase;
            const uint32_t slot = tab_at(pre);
            __syncwarp(gm);
            sts32(slot, here);
            __syncwarp(gm);
            const unsigned there = lds32(tab_at(to));
            __syncwarp(gm);
            sts32(slot, 0u);
            return __popc(there & le1) - __popc(here & le1);
        };
        unsigned open;  // steps that the leading words do not decide
        if (heavy) {
            for (;;) {
                if (fl) reflip();
                place();
                const int D = lead(to) - lead(pre) + incH * counted_now();
                const unsigned A2 = ballot(D < d.blo);
                open = ballot((uint32_t)(D - d.blo) < d.bw);
                if (A2 == A && moved == 0u) break;
                A = A2;
            }
        } else {
            for (;;) {
                if (fl) reflip();
                place();
                const int D = lead(to) - lead(pre);
                const unsigned A2 = ballot(D < d.blo);
                open = ballot((uint32_t)(D - blo2) < bw2);
                if (A2 == A && moved == 0u) break;
                A = A2;
            }
        }
        if (open) {
            // on from here with all 64 bits and the batch's own ln f steps
            long long b64;
            unsigned long long w64;
            bracket(d.T, t_io + (unsigned long long)j, b64, w64);
            unsigned fm = 0u, fv = 0u;  // steps settled in binary64, and those of them that accept
            for (;;) {
                if (fl) reflip();
                place();
                int cA, cB;
                counted(cA, cB);
                const unsigned long long D64 = (unsigned long long)lds64(to) - (unsigned long long)lds64(pre) +
                                               incF * (unsigned long long)(long long)(cB - cA);
                const unsigned A2 = (ballot(j < n && (long long)D64 < b64) & ~fm) | fv;
                const unsigned um = ballot(j < n && D64 - (unsigned long long)b64 < w64) & ~fm;
                if (A2 != A || moved != 0u) {
                    A = A2;
                    continue;
                }
                if (um == 0u) break;
                // the first undecided step: the reference's test in binary64
                const int f = __ffs((int)um) - 1;
                long long Ab = 0, Bb = 0;
                if (j == f) {
                    const int ia = REWL_IDX((int)(pre - pbase) / 8, 0, M.B, tally.bad);
                    const int ib = REWL_IDX((int)(to - pbase) / 8, 0, M.B, tally.bad);
                    Ab = PROD ? lgb[ia] : exact_steps(lds64(pre), lgb, ia, ew, lnf, cA);
                    Bb = PROD ? lgb[ib] : exact_steps(lds64(to), lgb, ib, ew, lnf, cB);
                }
                Ab = __shfl_sync(gm, Ab, f, S);
                Bb = __shfl_sync(gm, Bb, f, S);
                const unsigned long long tf = t_io + (unsigned long long)f;
                const uint4 r = random(tf);
                tally.slow += 1;
                const bool ok = ballot(exact_accept(Ab, Bb, u53(r.z, r.w), &tally.tie, tf)) != 0u;
                fm |= 1u << f;
                if (ok) fv |= 1u << f;
                A = (A & ~fm) | fv;
            }
        }

        // ---- commit ---------------------------------------------------------------
        // the lattice, and at once the next proposals' spins and marks, whose
        // reads run under the ln g updates
        const bool acc = (A & bit) != 0u;
        if (BITS == 8) {  // the site's last accepted value stays
            if (acc && (twins & A & ~le) == 0u) reinterpret_cast<uint8_t *>(lat)[site] = (uint8_t)nw;
        } else if (acc) {
            atomicXor(&lat[site / per], (uint32_t)(cur ^ nw) << ((site & (per - 1)) * BITS));
        }
        const uint32_t at = acc ? to : pre;  // the bin after the step
        unsigned steps = 0u;  // those that ended in this lane's bin
        if (!PROD) steps = __match_any_sync(gm, j < n ? at : 0u) >> gbase;
        __syncwarp(gm);
        read_spins();
        sts8(mark_at(next.site), (uint32_t)j);
        if constexpr (PROD) {
            int most = nmax;  // the majority count after the step
            if (A) {
                most = 0;
#pragma unroll 2
                for (int v = 0; v < M.q; ++v) {
                    const int c = st.cnt[v];
                    const unsigned up = ballot(acc && nw == v), down = ballot(acc && cur == v);
                    most = max(most, c + __popc(up & le) - __popc(down & le));
                    if ((up | down) != 0u && j == 0) st.cnt[v] = c + __popc(up) - __popc(down);
                }
                nmax = __shfl_sync(gm, most, n - 1, S);
            }
            // class = (O - ceil(N / q)) n_obins / (N - ceil(N / q) + 1)
            const uint32_t x = (uint32_t)(most - qlo);
            const int cls = narrow ? (int)(x * (uint32_t)st.n_obins / span)
                                   : (int)((unsigned long long)x * (unsigned)st.n_obins / span);
            const int b = REWL_IDX((int)(at - pbase) / 8, 0, M.B, tally.bad);
            const long long key = heo_index(b, st.n_obins, cls);
            // one add per run of equal keys, by its last step (keys of neighbouring
            // steps lie within 5 n_obins < 2^23: the low words tell them apart)
            const int after = __shfl_down_sync(gm, (int)key, 1, S);
            const bool ends = j < n && (j == n - 1 || after != (int)key);
            const unsigned before = ballot(ends) & lt;
            if (ends) atomicAdd(&st.heo[key], (unsigned long long)(before ? j - 31 + __clz((int)before) : j + 1));
        } else {
            const long long F = lds64(at);
            const int c = __popc(steps);
            const bool writer = j < n && (steps & ~le) == 0u;  // the bin's last step: its lane writes for all of them
            const int b = REWL_IDX((int)(at - pbase) / 8, 0, M.B, tally.bad);
            const long long F2 = (long long)((unsigned long long)F + incF * (unsigned)c);
            const uint32_t h1 = (uint32_t)((unsigned long long)F >> 32), h2 = (uint32_t)((unsigned long long)F2 >> 32);
            const bool plain = int_add && !(F & 1) && (h2 ^ h1) <= h1;
            if (writer) {  // (predicated: no branch)
                sts64(at, F2);
                atomicAdd(&hg[b], (uint32_t)c);  // (result not used: the walker does not wait)
            }
            if (writer && !plain) {
                long long F3 = F2;
                if (!whole_steps(F, c, LNF, ew, int_add, F3)) {  // binary64 adds
                    const long long v = exact_steps(F, lgb, b, ew, lnf, c);
                    F3 = shadow_of(v, ew);
                    if (F3 & 1) lgb[b] = v;
                    nseq += (unsigned)c;
                }
                sts64(at, F3);
            }
        }
        pcur = __shfl_sync(gm, at, n - 1, S);
        nacc += acc ? 1u : 0u;
        t_io += (unsigned long long)n;
        left -= n;
        __syncwarp(gm);
        if (left <= 0) break;
    }
    // the binary64 array from the authoritative shadow
    for (int b = j; !PROD && b < M.B; b += S) {
        const long long F = lgf[b];
        if (!(F & 1)) lgb[b] = from_units(F >> 1, ew);
    }
#pragma unroll
    for (int o = 1; o < S; o <<= 1) {
        nseq += __shfl_xor_sync(gm, nseq, o);
        nacc += __shfl_xor_sync(gm, nacc, o);
    }
    tally.seq += nseq;
    tally.acc += nacc;
    E_io = (int)(pcur - pbase) / 8 + lo;
}

// P walkers g0 .. g0 + P - 1 of one instance: stage their lattices in shared
// memory (LG = false; LG = true keeps large lattices in global memory), run K
// steps (one lane group per walker), write the lattices back.  The binary64
// ln g and the histogram of each walker stay in global memory: the launch
// reads ln g once to build the shadow and writes it back once at the end.
// BITS is the packing while the sweep runs: 4-bit configurations are staged as
// bytes where BITS = 8.
template <int BITS>
__device__ __forceinline__ void stage_lattice(const Model &M, uint32_t *lat, const uint32_t *src) {
    if (BITS == 8 && M.bits == 4) {
        for (int i = threadIdx.x; i < M.wpc; i += blockDim.x) {  // eight 4-bit fields to eight bytes
            const uint32_t w = src[i];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t x = (w >> (16 * h)) & 0xffffu;
                x = (x | (x << 8)) & 0x00ff00ffu;
                x = (x | (x << 4)) & 0x0f0f0f0fu;
                if (8 * i + 4 * h < M.N) lat[2 * i + h] = x;
            }
        }
    } else {
        for (int i = threadIdx.x; i < M.wpc; i += blockDim.x) lat[i] = src[i];
    }
}
template <int BITS>
__device__ __forceinline__ void unstage_lattice(const Model &M, uint32_t *dst, const uint32_t *lat) {
    if (BITS == 8 && M.bits == 4) {
        for (int i = threadIdx.x; i < M.wpc; i += blockDim.x) {
            uint32_t w = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t x = 8 * i + 4 * h < M.N ? lat[2 * i + h] : 0u;
                x = (x | (x >> 4)) & 0x00ff00ffu;
                x = (x | (x >> 8)) & 0xffffu;
                w |= x << (16 * h);
            }
            dst[i] = w;
        }
    } else {
        for (int i = threadIdx.x; i < M.wpc; i += blockDim.x) dst[i] = lat[i];
    }
}

// A walker's state and counters after its launch (one thread per walker).
__device__ __forceinline__ void end_walker(const Model &M, const State &Sg, int g, uint32_t c, int E, unsigned long long t,
                                           const Tally &tally) {
    Sg.cfg_E[c] = E;
    Sg.t[g] = t;
    atomicAdd(&Sg.ctl->flips, (unsigned long long)M.K);
    atomicAdd(&Sg.ctl->accepted, (unsigned long long)tally.acc);
    if (tally.slow) atomicAdd(&Sg.ctl->slow, tally.slow);
    flush_ties(Sg, g, tally.tie);
    if (tally.seq) atomicAdd(&Sg.ctl->seq, (unsigned long long)tally.seq);
#ifdef REWL_DEBUG_CHECKS
    if (tally.bad) atomicOr(&Sg.ctl->error, ERR_BOUNDS);
#endif
}

template <int BITS, int S, bool LG>
__device__ __forceinline__ void sweep_block(const Model &M, const State &Sg, int g0, int P, const Layout &lay,
                                            unsigned char *smem) {
    // (votes and the broadcast of the group index tell the compiler that whole
    // warps take each branch, which spares a divergence check at every ballot)
    if (__any_sync(0xffffffffu, *(volatile unsigned int *)&Sg.ctl->all_done)) return;
    for (int p = 0; p < P; ++p) {
        const int g = g0 + p;
        if (g >= M.G || Sg.done[g / M.m]) continue;
        unsigned char *base = smem + (size_t)p * lay.stride;
        if (!LG)
            stage_lattice<BITS>(M, reinterpret_cast<uint32_t *>(base + lay.off_lat),
                                Sg.spins + (size_t)Sg.slot_cfg[g] * M.wpc);
        if (S > 1) {
            uint32_t *bm = reinterpret_cast<uint32_t *>(base + lay.off_bm);
            for (int i = threadIdx.x; i < lay.marks / 4; i += blockDim.x) bm[i] = 0xffffffffu;
            uint32_t *tab = reinterpret_cast<uint32_t *>(base + lay.off_tab);
            for (int i = threadIdx.x; i < 8 * S; i += blockDim.x) tab[i] = 0u;
        }
    }
    __syncthreads();

    const int grp = S == 32 ? __shfl_sync(0xffffffffu, (int)threadIdx.x / S, 0) : (int)threadIdx.x / S;
    const int g = g0 + grp;
    Tally tally{};
    bool live = grp < P && g < M.G;
    if (live) live = !Sg.done[g / M.m];
    if (S == 32) live = __any_sync(0xffffffffu, live);
    if constexpr (S == 1) {
        unsigned char *base = smem + (size_t)(live ? grp : 0) * lay.stride;
        const int gl = live ? g : g0, w = gl / M.m;
        const uint32_t c = Sg.slot_cfg[gl];
        int E = Sg.cfg_E[c];
        unsigned long long t = Sg.t[gl];
        // with global lattices the shadow is in global memory too
        walker_sweep_1<BITS, LG>(M, LG ? Sg.spins + (size_t)c * M.wpc : reinterpret_cast<uint32_t *>(base + lay.off_lat),
                             reinterpret_cast<long long *>(Sg.lng + (size_t)gl * M.B),
                             LG ? Sg.shadow + (size_t)gl * (M.B + 2 * kPad) + kPad
                                : reinterpret_cast<long long *>(base + lay.off_lgf) + kPad,
                             Sg.H + (size_t)gl * M.B, gl, Sg.e_lo[w], Sg.lnf[w], E, t, tally, live);
        if (live) end_walker(M, Sg, gl, c, E, t, tally);
    } else if (live) {
        unsigned char *base = smem + (size_t)grp * lay.stride;
        Stage st;
        st.ring = reinterpret_cast<uint2 *>(base + lay.off_ring);
        st.pk = reinterpret_cast<uint32_t *>(base + lay.off_pk);
        st.tab = reinterpret_cast<uint32_t *>(base + lay.off_tab);
        st.bm = base + lay.off_bm;
        st.mmask = lay.marks >= M.N ? 0xffffffffu : (uint32_t)(lay.marks - 1);
        const int w = g / M.m;
        const uint32_t c = Sg.slot_cfg[g];
        int E = Sg.cfg_E[c];
        unsigned long long t = Sg.t[g];
        uint32_t *lat = LG ? Sg.spins + (size_t)c * M.wpc : reinterpret_cast<uint32_t *>(base + lay.off_lat);
        long long *lgf = reinterpret_cast<long long *>(base + lay.off_lgf) + kPad;
        walker_sweep<BITS, S>(M, lat, reinterpret_cast<long long *>(Sg.lng + (size_t)g * M.B), lgf,
                              Sg.H + (size_t)g * M.B, st, g, Sg.e_lo[w], Sg.lnf[w], E, t, tally);
        if ((threadIdx.x & (S - 1)) == 0) end_walker(M, Sg, g, c, E, t, tally);
#ifdef REWL_DEBUG_CHECKS
        if (tally.bad) atomicOr(&Sg.ctl->error, ERR_BOUNDS);
#endif
    }
    __syncthreads();

    if (!LG) {
        for (int p = 0; p < P; ++p) {
            const int gg = g0 + p;
            if (gg >= M.G || Sg.done[gg / M.m]) continue;
            unstage_lattice<BITS>(M, Sg.spins + (size_t)Sg.slot_cfg[gg] * M.wpc,
                                  reinterpret_cast<const uint32_t *>(smem + (size_t)p * lay.stride + lay.off_lat));
        }
    }
}

template <int BITS, int S, bool LG>
__global__ void __launch_bounds__(256, 1) sweep_fast_kernel(Model M, State Sg, int P, Layout lay) {
    extern __shared__ __align__(16) unsigned char smem[];
    sweep_block<BITS, S, LG>(M, Sg, blockIdx.x * P, P, lay, smem);
}

// Fixed-weight production: P walkers per CTA, a lane group of 32 each; every
// window runs, finished or not, with the walkers' own ln g.
template <int BITS, bool LG>
__global__ void __launch_bounds__(256) production_fast_kernel(Model M, State Sg, int P, Layout lay, int off_cnt) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int g0 = blockIdx.x * P;
    for (int p = 0; p < P && g0 + p < M.G; ++p) {
        unsigned char *base = smem + (size_t)p * lay.stride;
        const uint32_t c = Sg.slot_cfg[g0 + p];
        if (!LG)
            stage_lattice<BITS>(M, reinterpret_cast<uint32_t *>(base + lay.off_lat), Sg.spins + (size_t)c * M.wpc);
        uint32_t *bm = reinterpret_cast<uint32_t *>(base + lay.off_bm);
        for (int i = threadIdx.x; i < lay.marks / 4; i += blockDim.x) bm[i] = 0xffffffffu;
        int *cnt = reinterpret_cast<int *>(base + off_cnt);
        for (int i = threadIdx.x; i < M.q; i += blockDim.x) cnt[i] = Sg.cnt[(size_t)c * M.q + i];
    }
    __syncthreads();

    const int grp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0);
    const int g = g0 + grp;
    Tally tally{};
    if (__any_sync(0xffffffffu, grp < P && g < M.G)) {
        unsigned char *base = smem + (size_t)grp * lay.stride;
        const int w = g / M.m;
        const uint32_t c = Sg.slot_cfg[g];
        Stage st;
        st.ring = reinterpret_cast<uint2 *>(base + lay.off_ring);
        st.pk = reinterpret_cast<uint32_t *>(base + lay.off_pk);
        st.tab = reinterpret_cast<uint32_t *>(base + lay.off_tab);
        st.bm = base + lay.off_bm;
        st.mmask = lay.marks >= M.N ? 0xffffffffu : (uint32_t)(lay.marks - 1);
        st.cnt = reinterpret_cast<int *>(base + off_cnt);
        st.heo = Sg.heo + (size_t)w * M.B * M.n_obins;
        st.n_obins = M.n_obins;
        int E = Sg.cfg_E[c];
        unsigned long long t = Sg.t[g];
        walker_sweep<BITS, 32, true>(M, LG ? Sg.spins + (size_t)c * M.wpc : reinterpret_cast<uint32_t *>(base + lay.off_lat),
                                     reinterpret_cast<long long *>(Sg.lng + (size_t)g * M.B),
                                     reinterpret_cast<long long *>(base + lay.off_lgf) + kPad, nullptr, st, g, Sg.e_lo[w],
                                     0.0, E, t, tally);
        if ((threadIdx.x & 31) == 0) {
            Sg.cfg_E[c] = E;
            Sg.t[g] = t;
            atomicAdd(&Sg.ctl->flips, (unsigned long long)M.K);
            atomicAdd(&Sg.ctl->accepted, (unsigned long long)tally.acc);
            if (tally.slow) atomicAdd(&Sg.ctl->slow, tally.slow);
            flush_ties(Sg, g, tally.tie);
        }
#ifdef REWL_DEBUG_CHECKS
        if (tally.bad) atomicOr(&Sg.ctl->error, ERR_BOUNDS);
#endif
    }
    __syncthreads();

    for (int p = 0; p < P && g0 + p < M.G; ++p) {
        const unsigned char *base = smem + (size_t)p * lay.stride;
        const uint32_t c = Sg.slot_cfg[g0 + p];
        if (!LG)
            unstage_lattice<BITS>(M, Sg.spins + (size_t)c * M.wpc, reinterpret_cast<const uint32_t *>(base + lay.off_lat));
        const int *cnt = reinterpret_cast<const int *>(base + off_cnt);
        for (int i = threadIdx.x; i < M.q; i += blockDim.x) Sg.cnt[(size_t)c * M.q + i] = cnt[i];
    }
}

// Persistent batched sweep by lane groups of 32: each CTA takes the next item from *queue.
template <int BITS>
__global__ void __launch_bounds__(256) batch_sweep_kernel(const InstDev *inst, const SweepItem *items, int n_items,
                                                          unsigned int *queue) {
    extern __shared__ __align__(16) unsigned char smem[];
    // The item's number passes through the first walker's shadow padding, which
    // sweep_block writes only behind its first barrier: walkers may take all the
    // shared memory that a CTA can have.
    volatile int *next = reinterpret_cast<volatile int *>(smem);
    for (;;) {
        if (threadIdx.x == 0) *next = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int i = __shfl_sync(0xffffffffu, *next, 0);
        if (i >= n_items) break;
        const SweepItem it = items[i];
        const Model M = inst[it.inst].M;
        const State Sg = inst[it.inst].S;
        const Layout lay = inst[it.inst].lay;
        sweep_block<BITS, 32, false>(M, Sg, it.g0, it.P, lay, smem);
        __syncthreads();
    }
}

// Batched one-lane sweep with every walker's state in global memory: thread i
// runs walker items[i] (any instance of this spin packing) for K steps.
template <int BITS>
__global__ void __launch_bounds__(256) batch_walker_kernel(const InstDev *inst, const WalkerItem *items, int n_items) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const WalkerItem it = items[min(i, n_items - 1)];
    const Model M = inst[it.inst].M;
    const State Sg = inst[it.inst].S;
    const int g = it.g, w = g / M.m;
    const bool live = i < n_items && !*(volatile unsigned int *)&Sg.ctl->all_done && !Sg.done[w];
    Tally tally{};
    const uint32_t c = Sg.slot_cfg[g];
    int E = Sg.cfg_E[c];
    unsigned long long t = Sg.t[g];
    walker_sweep_1<BITS, true>(M, Sg.spins + (size_t)c * M.wpc, reinterpret_cast<long long *>(Sg.lng + (size_t)g * M.B),
                         Sg.shadow + (size_t)g * (M.B + 2 * kPad) + kPad, Sg.H + (size_t)g * M.B, g, Sg.e_lo[w],
                         Sg.lnf[w], E, t, tally, live);
    if (live) end_walker(M, Sg, g, c, E, t, tally);
}

// Bits per spin of a lattice staged in shared memory: bytes, one load per spin
// (4-bit fields take a shift and a mask more for each of a proposal's five
// spins), up to this many bytes for the walker; narrow lane groups: see kMarksNarrow.
constexpr int kByteStageMax = 96 * 1024;

Layout make_layout(const Model &M, int S, bool lat_global, int bits);

int stage_bits(const Model &M, int S, bool lat_global) {
    if (M.bits == 8 || lat_global || S <= 4 || (S == 8 && M.N > kMarksNarrow)) return M.bits;
    return make_layout(M, S, false, 8).stride <= kByteStageMax ? 8 : 4;
}

Layout make_layout(const Model &M, int S, bool lat_global, int bits) {
    auto al = [](int x) { return (x + 15) & ~15; };
    Layout l{};
    int off = 0;
    if (S == 1 && lat_global) {  // every part of the walker's state in global memory
        l.off_lgf = l.off_lat = l.off_ring = l.off_pk = l.off_tab = l.off_bm = -1;
        l.stride = 0;
        return l;
    }
    l.off_lgf = off;  // (first: batch_sweep_kernel passes an item number through its padding)
    off += al((M.B + 2 * kPad) * 8);
    l.off_lat = -1;
    if (!lat_global) {
        l.off_lat = off;
        off += al((M.N * bits + 31) / 32 * 4);
    }
    // (at least the bytes per walker that decide which windows fit, so that the
    // set of accepted configurations does not depend on the scratch below)
    const int least = S > 1 ? al((S + 8) * 16) + al((S + 8) * 4) + al(2 * ((min(M.N, 8192) + 31) / 32) * 4) : 0;
    const int fits = off + least;
    const int queues = al(kAhead * S * 8) + al(2 * S * 4) + al(8 * S * 4);
    int most = lat_global ? kMarksFar : kMarks;
    if (S == 8) most = lat_global ? kMarksNarrow / 2 : kMarksNarrow;
    if (S <= 4)
        for (most = 512; 2 * most <= least - queues;) most *= 2;
    l.marks = M.N <= (S > 8 ? kMarks : most) ? al(M.N) : most;
    if (off > kByteStageMax) l.marks = 512;
    if (S > 1) {
        l.off_ring = off;
        off += al(kAhead * S * 8);
        l.off_pk = off;
        off += al(2 * S * 4);
        l.off_tab = off;
        off += al(8 * S * 4);
        l.off_bm = off;
        off += l.marks;
    }
    off = off > fits ? off : fits;
    l.stride = al(off);
    return l;
}

template <int BITS, int S, bool LG>
cudaError_t launch_lg(const Model &M, const State &St, const SweepPlan &p, cudaStream_t s, bool prepare) {
    const Layout lay = make_layout(M, S, LG, BITS);
    if (prepare) return allow_shared((const void *)sweep_fast_kernel<BITS, S, LG>);
    sweep_fast_kernel<BITS, S, LG><<<p.grid, p.threads, p.smem, s>>>(M, St, p.P, lay);
    return cudaGetLastError();
}

template <int BITS, int S>
cudaError_t launch_t(const Model &M, const State &St, const SweepPlan &p, cudaStream_t s, bool prepare) {
    return p.lat_global ? launch_lg<BITS, S, true>(M, St, p, s, prepare)
                        : launch_lg<BITS, S, false>(M, St, p, s, prepare);
}

template <int BITS>
cudaError_t dispatch_s(const Model &M, const State &St, const SweepPlan &p, cudaStream_t s, bool prepare) {
    switch (p.lanes) {
    case 1: return launch_t<BITS, 1>(M, St, p, s, prepare);
    case 2: return launch_t<BITS, 2>(M, St, p, s, prepare);
    case 4: return launch_t<BITS, 4>(M, St, p, s, prepare);
    case 8: return launch_t<BITS, 8>(M, St, p, s, prepare);
    case 16: return launch_t<BITS, 16>(M, St, p, s, prepare);
    default: return launch_t<BITS, 32>(M, St, p, s, prepare);
    }
}

}  // namespace fast

int sweep_bits(const Model &M, int lanes, bool lat_global) { return fast::stage_bits(M, lanes, lat_global); }

size_t fast_smem_per_walker(const Model &M, int lanes, bool lat_global) {
    return (size_t)fast_layout(M, lanes, lat_global).stride;
}

Layout fast_layout(const Model &M, int lanes, bool lat_global) {
    return fast::make_layout(M, lanes, lat_global, fast::stage_bits(M, lanes, lat_global));
}

namespace {
const void *batch_sweep(int bits) {
    return bits == 8 ? (const void *)fast::batch_sweep_kernel<8> : (const void *)fast::batch_sweep_kernel<4>;
}
}  // namespace

cudaError_t launch_batch_sweep(int bits, const InstDev *inst, const SweepItem *items, int n_items, unsigned int *queue,
                               int grid, int threads, size_t smem, cudaStream_t s, bool prepare) {
    if (prepare) return allow_shared(batch_sweep(bits));
    if (n_items <= 0) return cudaSuccess;
    if (bits == 8) fast::batch_sweep_kernel<8><<<grid, threads, smem, s>>>(inst, items, n_items, queue);
    else fast::batch_sweep_kernel<4><<<grid, threads, smem, s>>>(inst, items, n_items, queue);
    return cudaGetLastError();
}

int batch_sweep_ctas_per_sm(int bits, int threads, size_t smem) {
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_sweep(bits), threads, smem) == cudaSuccess ? n : 0;
}

// Production by lane groups or by a thread per walker: which is faster, from what both
// took on GB300 (q = 3 .. 255, L = 16 .. 200, 3 to 860 walkers per SM; estimates in
// microseconds per 1000 steps of every walker, most within 10 %).
//  * Lane groups go in waves of the CTAs that are resident together.  A wave of r
//    walkers per SM takes 43 + 1.1 q (each value's count is looked at by every batch:
//    latency up to about 10 walkers per SM, issue slots above), and 20 to set up.
//  * A thread per walker takes one chain of steps, 700 for a few walkers per SM; in
//    full warps the lanes diverge (to 1700 at 40 walkers per SM), more warps share the
//    SM, and large lattices and many counts leave the caches.
// q = 10, L = 80: groups up to 340 walkers per SM (7.47 against 9.18 ms a round of 3000
// steps; at 674 14.3 against 13.2); q = 80: up to 110 (5.8 / 6.6; at 168 8.7 / 7.8);
// q = 255: up to 27 (4.1 / 4.9; at 54 7.3 / 6.1, at 674 84.8 / 21.2).
bool production_lane_groups(const Model &M, int num_sms, int P, int ctas_per_sm) {
    auto wave = [&](double r) {
        return 43.0 + 20e3 / M.K + std::max(0.0, 0.9 * (r - 8.0)) + M.q * std::max(1.1, 0.112 * r);
    };
    const long long ctas = (M.G + P - 1) / P, at_once = (long long)num_sms * ctas_per_sm, rest = ctas % at_once;
    double groups = (double)(ctas / at_once) * wave((double)P * ctas_per_sm);
    if (rest) groups += wave((double)P * (double)((rest + num_sms - 1) / num_sms));
    const double w = (double)M.G / num_sms;
    const double chain = 700.0 + 25.0 * std::min(w, 40.0) + 3.6 * w;
    const double counts = 1.0 + 0.0015 * M.q * std::min(std::max(0.0, (w - 30.0) / 120.0), 1.0);
    const double lattices = 0.85 + M.wpc * 4 / 42000.0;
    return groups <= chain * counts * lattices;
}

// If a walker's production state fits a CTA's shared memory and lane groups are the
// faster form, queue the sweep (P walkers a CTA, one CTA per SM while the walkers
// last: their chains, not a pipe, set the rate).
bool launch_production_fast(const Model &M, const State &S, int num_sms, size_t smem_optin, cudaStream_t s,
                            cudaError_t *err) {
    const bool lg = M.wpc * 4 > kSharedLatticeMax;
    const int bits = sweep_bits(M, 32, lg);
    Layout lay = fast::make_layout(M, 32, lg, bits);
    const int off_cnt = lay.stride;
    lay.stride += (M.q * 4 + 15) & ~15;
    int P = (int)(smem_optin / (size_t)lay.stride);
    P = min(min(P, 8), (M.G + num_sms - 1) / num_sms);
    if (P < 1) return false;
    const size_t smem = (size_t)P * (size_t)lay.stride;
    bool queued = true;
    auto go = [&](auto kernel) {
        *err = allow_shared((const void *)kernel);
        if (*err != cudaSuccess) return;
        int per_sm = 1;
        if ((M.G + P - 1) / P > num_sms)
            *err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, P * 32, smem);
        if (*err != cudaSuccess) return;
        queued = production_lane_groups(M, num_sms, P, max(per_sm, 1));
        if (!queued) return;
        kernel<<<(M.G + P - 1) / P, P * 32, smem, s>>>(M, S, P, lay, off_cnt);
        *err = cudaGetLastError();
    };
    if (lg) bits == 8 ? go(fast::production_fast_kernel<8, true>) : go(fast::production_fast_kernel<4, true>);
    else bits == 8 ? go(fast::production_fast_kernel<8, false>) : go(fast::production_fast_kernel<4, false>);
    return queued;
}

cudaError_t launch_batch_walkers(int bits, const InstDev *inst, const WalkerItem *items, int n_items, int grid,
                                 int threads, cudaStream_t s, bool prepare) {
    if (prepare) return cudaSuccess;
    if (n_items <= 0) return cudaSuccess;
    if (bits == 8) fast::batch_walker_kernel<8><<<grid, threads, 0, s>>>(inst, items, n_items);
    else fast::batch_walker_kernel<4><<<grid, threads, 0, s>>>(inst, items, n_items);
    return cudaGetLastError();
}

int batch_walkers_ctas_per_sm(int bits, int threads) {
    int n = 0;
    cudaError_t e = bits == 8 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fast::batch_walker_kernel<8>, threads, 0)
                              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fast::batch_walker_kernel<4>, threads, 0);
    return e == cudaSuccess ? n : 0;
}

cudaError_t launch_sweep_fast(const Model &M, const State &S, const SweepPlan &p, cudaStream_t s, bool prepare) {
    return sweep_bits(M, p.lanes, p.lat_global != 0) == 8 ? fast::dispatch_s<8>(M, S, p, s, prepare)
                                                          : fast::dispatch_s<4>(M, S, p, s, prepare);
}

}  // namespace rewl
