// Exact Gram pass on tcgen05 (C = X^T X) with a fixed-point Cholesky behind it: R in one pass
// over X, in the 4-, 8-, 16-, 32- and 64-column classes, for TSQR calls and, while their further
// passes could not change R, for the Gram methods.
//
// Measured against the double-float Householder tiles (which stay for calls that lose light rows,
// see light_floor, and those that exact_route leaves them) and the Gram methods' own passes (which
// stay beyond the limits in xg_finish): TSQR m = 2^25, n = 4 917 -> 383 us; m = 2^23, n = 8, 16, 32
// 213, 406, 783 us (2.5, 2.6, 2.7 TB/s of X); m = 2^22, n = 64 21.1 -> 2.11 ms, Cholesky-QR2
// 8.30 -> 2.11 ms; SVQB2 10^6 x 32 3.89 -> 0.20 ms; shifted Cholesky-QR3 300007 x 24 871 ->
// 114 us; least squares 2^24 x 31, FP32-stored, 19.3 -> 1.48 ms; 131072 x 8 145 -> 42 us.
// ||R - R_ref|| / ||R_ref|| against 64-bit references: 3.5e-16 -> 1.9e-16 (n = 64), 1.1e-15 ->
// 1.9e-16 (Cholesky-QR2), 1e-14 -> 3.3e-16 (SVQB2), 4.2e-15 -> 1.2e-16 (Cholesky-QR3).
// Up to 32 columns the integer pipe bounds it (75 % busy: some 37 instructions of it per element
// to cut and pack the digits); at 64 columns the MMAs do (36 of 128 x 64 x 16 per 16 rows: each
// reads 6 KB of shared memory for 32 cycles of work) and the read-out every 8 tiles.
//
// Every value is rounded to a signed 56-bit fixed point N relative to a running per-column
// scale 2^e (|x| < 2^e, x ~ N 2^(e - 55)) and cut into EIGHT balanced base-128 digits, which
// bf16 holds exactly.  ALL 64 digit-plane products are formed, every FP32 sum of the tensor
// core stays an integer of at most 2^24 (exact), the read-outs fold them into 128-bit
// integers and the CTAs add those into one integer accumulator of 320 bits per entry of C.
// The Gram matrix of the rounded X is therefore exact: no product is dropped, no sum rounds,
// and the sums do not depend on the order of tiles, CTAs or atomics (the rounding follows the
// running maxima of each CTA, so it does on the partition into CTAs).  That is what lets
// one pass serve TSQR: with C exact, a Cholesky factorisation in 125-bit fixed point
// (xg_cholesky) loses kappa^2 2^-99, 2^-111 when refined, instead of kappa^2 2^-53, so the R it
// gives is limited by the rounding of X: a scale stands 2 to 3 bits above the maximum that set it,
// so half a step is 2^-54 to 2^-53 of the largest entry that the CTA has met in the column, a
// columnwise backward error of up to sqrt(m) max|x| 2^-53.  (It is not a rowwise one: light_floor.)
//
//  * Roles and tiles: 16 slicer warps cut tiles of 4096 elements (KT = 4096 / NC rows) into
//    digit planes and read the accumulators out; one warp issues the tensor-map copies two
//    tiles ahead (a whole tile per instruction), one the MMAs, in warp-uniform code with one
//    elected lane so that descriptors stay in uniform registers.  Two raw stages and two
//    digit buffers alternate.
//  * The slicers form two groups of eight warps: one takes the even tiles (stage and buffer 0),
//    the other the odd ones, so that one group cuts while the other waits for its tile or
//    votes; cutting is bound by the integer pipe, and with all sixteen warps in step that pipe
//    idled 40 % of the time.  Each group votes once per tile whether a column outgrew its scale
//    (the groups' votes alternate in tile order, so neither can hand a tile over that the
//    tensor core would wait on the other for); a full group of tiles, such a column or the end
//    brings both groups together for the read-out, with their next tiles already cut.
//    Mbarriers: "MMAs done" and "digits ready" per digit buffer, "tile landed" and "stage
//    read" per raw stage, "vote passed" per group.  All waits are bounded; the first that gives
//    up sets a flag that ends the others at once.
//  * The planes lie one after the other in the K-major core-matrix layout, so all planes
//    together are one operand of 8 NC columns (plane p, column c at 8-column group
//    (p NC + c) / 8).
//      NC = 16:  one MMA 128 x 128 x 16 per 16 rows; lane p 16 + i, column q 16 + j.
//      NC = 4, 8: the tile is cut into 16 / NC row segments that stand side by side as 16
//                virtual columns; the products of different segments are never read.  (MMAs
//                of 8 NC columns took as long each: n = 4 was bound by their number.)
//      NC = 32:  two MMAs 128 x 256 x 16 (planes 0..3, 4..7): 512 tensor-memory columns.
//      NC = 64:  512 x 512 sums do not fit, so pairs of equal weight w = p + q share one of
//                16 half blocks: block b holds weight 2 b in lanes 0..63 and 2 b + 1 in lanes
//                64..127.  Plane q even meets the stacked planes (p, p + 1), p even, and q
//                odd those with p odd (from -1 to 7; plane -1 and plane 8 are zeros), so
//                every product lands on its own weight: 36 MMAs 128 x 64 x 16.
//  * G tiles add up in one set of tensor-memory sums: G KT rows x (pairs per sum) x 64^2 <=
//    2^24.  The classes up to 16 columns fill NS sets in turn before a read-out (64 tiles).
#pragma once

#include "gram_launch.cuh"

namespace ql {

using u64 = unsigned long long;
using u128 = unsigned __int128;
using i128 = __int128;

template <int NC>
struct XgShape {
  static constexpr int TS = 512;             // slicer threads, in two groups of TG
  static constexpr int TG = 256;
  static constexpr int T = TS + 64;          // and the copy warp and the MMA warp
  static constexpr int KT = 4096 / NC;       // rows per tile
  static constexpr int VC = NC < 16 ? 16 : NC;      // columns of a digit plane: SEG segments x NC
  static constexpr int SEG = VC / NC;
  static constexpr int KV = KT / SEG;        // rows of a digit plane
  static constexpr int PLANE = VC * KV * 2;  // bytes per digit plane (8 KB)
  static constexpr int DBUF = 8 * PLANE;     // digit planes of a tile (64 KB)
  static constexpr int PAD = NC == 64 ? PLANE : 0;  // zero planes before, between and after the buffers
  static constexpr int LBO = 128;            // bytes between core matrices along the rows
  static constexpr int SBO = KV * 16;        // bytes between 8-column groups
  static constexpr int SCOLS = VC == 16 ? 128 : 512;        // tensor-memory columns of one set of sums
  static constexpr int NS = 512 / SCOLS;                    // sets: 4, 4, 4, 1, 1
  static constexpr int PAIRS = NC == 64 ? 8 : 1;     // products per sum (weight 7 has eight)
  static constexpr int G = 4096 / (KV * PAIRS);      // tiles per set: 16, 16, 16, 32, 8
  static constexpr int GT = G * NS;                  // tiles per read-out: 64, 64, 64, 32, 8
  static constexpr int SLACK = 2;            // bits of headroom above a new column maximum
  static constexpr int HALF = NC / 4;        // columns of C per slicer thread at a read-out
  static constexpr int LG = 128 / VC;        // lane groups (planes, or weight parities)
  // the 128-bit sums of an entry's lane groups come together below 1.02 2^110 per row (NC = 64:
  // 2^111 per row in the odd weights' one): emptied before 2^126
  static constexpr int MAX_READS = (NC == 64 ? 1 << 15 : 1 << 16) / (GT * KT);
  static_assert(NC == 4 || NC == 8 || NC == 16 || NC == 32 || NC == 64, "column classes");
  static_assert((long long)G * KV * PAIRS * 4096 <= (1LL << 24), "exact FP32 digit sums");
};

template <int NC, typename S>
struct XgSmem {
  using Sh = XgShape<NC>;
  // a staged tile: blocks of 128 bytes of rows x NC columns, column c of block k in the
  // 128-byte line k NC + c, whose 16-byte chunk q sits at q ^ (line & 7) (128-byte swizzle);
  // the right-hand side of least squares is staged apart, its rows in order
  static constexpr int RPB = 128 / (int)sizeof(S);
  static constexpr size_t kDig = 2 * (size_t)Sh::DBUF + 3 * (size_t)Sh::PAD;
  static constexpr size_t kRaw = sizeof(S) * (size_t)NC * Sh::KT;
  static constexpr size_t kOffRaw = kDig;
  static constexpr size_t kStageB = sizeof(S) * (size_t)Sh::KT;
  static constexpr size_t kOffB = kOffRaw + 2 * kRaw;
  static constexpr size_t kOffScale = kOffB + 2 * kStageB;
  static constexpr size_t kOffColmax = kOffScale + 4 * NC;
  static constexpr size_t kOffBal = kOffColmax + 4 * NC;  // per column: light entries less the others,
  static constexpr size_t kOffLit = kOffBal + 4 * NC;     // whether a unit of eight rows was light
  static constexpr size_t kOffMisc = kOffLit + 4 * NC;
  // barriers and the tensor-memory slot: the same place in every class, so that a grouped
  // launch sets them up once
  static constexpr size_t kOffBar = 231424;
  static constexpr size_t kOffSlot = kOffBar + 80;
  static constexpr size_t kBytes = kOffSlot + 32;
  static_assert(kOffMisc + 64 * 4 <= kOffBar, "the tile areas end below the barriers");
  static constexpr size_t kEpi = 8 * (4 * (size_t)NC * (NC + 1) + 8 * (NC + 1)) + 64 * 4 + 16;
  static_assert(kBytes <= 232448, "shared memory of one SM");
  static_assert(kEpi <= kOffScale, "the epilogue's shared memory stays below the scales and barriers");
  static_assert(16 * (size_t)(Sh::LG * Sh::SEG - 1) * NC * NC <= (size_t)Sh::DBUF, "lane-group sums fit in a digit buffer");
};

// Integer accumulators of C: entry (i <= j) at index i + j (j + 1) / 2, kLimbs limbs of 40 bits
// in 64-bit words.  The unit is 2^(2 (kEsMin - 1022) - 110): N_i N_j of columns at scale
// exponents Es_i, Es_j (>= kEsMin) weighs 2^(Es_i + Es_j - 2 kEsMin) units, at most 2^184, so
// 128-bit sums end below bit 312 of 320; a limb takes 2^23 additions before it could overflow.
constexpr int kEsMin = kDfEminLimit;
constexpr int kEsMax = kDfEmaxLimit + 2;
constexpr int kXgUnitExp = 2 * (kEsMin - 1022) - 110;  // -188
QL_DEV int tri_index(int i, int j) { return i + j * (j + 1) / 2; }

// ---------------------------------------------------------------------------------------
// Cutting.  Nb2 = Q + 1 + 2 kDigitBias8 with Q = floor(2 |x| 2^(55 - e)): field p, (Nb2 >> (1 +
// 7 (7 - p))) & 127 (& 255 for p = 0), is digit p of |x| (rounded to nearest, ties away from
// zero) plus 64.  Q is one funnel shift of the significand aligned at bit 62, by s = Es - E + 7.
// Shift counts are formed without masking the sign bit off the exponent (modulo 2048, or 256
// for FP32), which the shifter's own modulo 32 makes exact for elements less than 2^24 below
// the scale; FAR covers the others.
// ---------------------------------------------------------------------------------------
constexpr u64 kCutBias = 2 * kDigitBias8 + 1;

QL_DEV unsigned sig_hi(unsigned hw, unsigned lw) { return (__funnelshift_l(lw, hw, 10) & 0x3fffffffu) | 0x40000000u; }

template <bool FAR>
QL_DEV u64 cut56(unsigned h, unsigned l, int s) {
  unsigned ql = __funnelshift_r(l, h, s), qh = h >> (s & 31);
  if constexpr (FAR) {
    if (s > 31) {
      ql = __funnelshift_rc(h, 0u, (unsigned)(s - 32));
      qh = 0u;
    }
  }
  return (((u64)qh << 32) | ql) + kCutBias;
}

// Planes 7 - 2 K and 6 - 2 K of eight elements: two adjacent 7-bit fields per element and
// shift, packed for rows (r, r + 1) into one word each; bf16(128 + f) sg - 192 sg = sg (f - 64)
// in one packed multiply-add gives the signed digit.
template <int PLANE, int K>
QL_DEV void put_plane_pairs(unsigned char* base, const u64 (&Nb)[8], const unsigned (&sg)[4]) {
  unsigned lo[4], hi[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const unsigned fa = (unsigned)(Nb[2 * e] >> (1 + 14 * K)), fb = (unsigned)(Nb[2 * e + 1] >> (1 + 14 * K));
    const unsigned t = __byte_perm(fa, fb, 0x5410);
    const unsigned wl = (t & 0x007f007fu) | 0x43004300u;
    const unsigned wh = ((t >> 7) & (K == 3 ? 0x00ff00ffu : 0x007f007fu)) | 0x43004300u;
    const unsigned one = sg[e] | 0x3f803f80u, off = sg[e] ^ 0xc340c340u;  // +-1, -+192
    const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162*>(&one);
    const __nv_bfloat162 c = *reinterpret_cast<const __nv_bfloat162*>(&off);
    const __nv_bfloat162 rl = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&wl), m, c);
    const __nv_bfloat162 rh = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&wh), m, c);
    lo[e] = *reinterpret_cast<const unsigned*>(&rl);
    hi[e] = *reinterpret_cast<const unsigned*>(&rh);
  }
  *reinterpret_cast<uint4*>(base + (7 - 2 * K) * PLANE) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  *reinterpret_cast<uint4*>(base + (6 - 2 * K) * PLANE) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  if constexpr (K < 3) put_plane_pairs<PLANE, K + 1>(base, Nb, sg);
}

// Eight rows of one column as raw words.
template <typename S>
struct Rows8;
template <>
struct Rows8<double> {
  unsigned hw[8], lw[8];
  QL_DEV unsigned amax() const {  // largest |x|, as its high word
    unsigned a = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) a = max(a, hw[j] & 0x7fffffffu);
    return a;
  }
  QL_DEV static int exponent(unsigned amax) { return (int)(amax >> 20); }
  // the scale's shift base (an all-zero column: far for every element), an element's shift
  // modulo kWrap, and the bits of it that are zero unless the element is far
  static constexpr int kWrap = 2048, kFar = 0x7e0;
  QL_DEV static int base(int Es) { return Es > 0 ? Es + 7 : 2000; }
  QL_DEV int shift(int j, int base) const { return base - (int)(hw[j] >> 20); }
  QL_DEV unsigned h(int j) const { return sig_hi(hw[j], lw[j]); }
  QL_DEV unsigned l(int j) const { return lw[j] << 10; }
  QL_DEV void set(int j, double x) {
    hw[j] = (unsigned)__double2hiint(x);
    lw[j] = (unsigned)__double2loint(x);
  }
  QL_DEV void chunk(int q, const uint4& t) {
    lw[2 * q] = t.x;
    hw[2 * q] = t.y;
    lw[2 * q + 1] = t.z;
    hw[2 * q + 1] = t.w;
  }
};
template <>
struct Rows8<float> {
  unsigned hw[8];
  QL_DEV unsigned amax() const {
    unsigned a = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) a = max(a, hw[j] & 0x7fffffffu);
    return a;
  }
  QL_DEV static int exponent(unsigned amax) {
    const int ef = (int)(amax >> 23);
    return ef == 0 ? 0 : ef + 896;
  }
  static constexpr int kWrap = 256, kFar = 0xe0;
  QL_DEV static int base(int Es) { return Es > 0 ? Es + 7 - 896 : 200; }
  QL_DEV int shift(int j, int base) const { return base - (int)(hw[j] >> 23); }
  QL_DEV unsigned h(int j) const { return ((hw[j] << 7) & 0x3fffffffu) | 0x40000000u; }
  QL_DEV unsigned l(int) const { return 0u; }
  QL_DEV void set(int j, float x) { hw[j] = __float_as_uint(x); }
  QL_DEV void chunk(int q, const uint4& t) {
    hw[4 * q] = t.x;
    hw[4 * q + 1] = t.y;
    hw[4 * q + 2] = t.z;
    hw[4 * q + 3] = t.w;
  }
};

// One lane of the (converged) warp: 1 in it, 0 in the others.
QL_DEV uint32_t elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p;
}
QL_DEV void umma_bf16_if(uint32_t leader, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(leader));
}
QL_DEV void umma_commit_if(uint32_t leader, uint64_t* mbar) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %1, 0;\n"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_addr(mbar)),
      "r"(leader));
}
// Wait for a phase, at most 2^32 clocks (about 2 s).  The wait that gives up records `code` in
// *fail; once that is set every other wait that would block gives up at once, so the roles of
// the CTA run through with whatever the buffers hold and the call is redone.
QL_DEV bool xg_wait(uint64_t* mbar, uint32_t parity, volatile int* fail, int code) {
  if (mbar_try_wait(mbar, parity)) return true;
  const long long t0 = clock64();
  do {
    if (mbar_try_wait(mbar, parity)) return true;
    if (*fail) return false;
  } while (clock64() - t0 <= (1ll << 32));
  *fail = code;
  return false;
}
// Whether a phase is over (never suspends the thread).
QL_DEV bool mbar_test_wait(uint64_t* mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred P1;\nmbarrier.test_wait.parity.shared::cta.b64 P1, [%1], %2;\n"
      "selp.b32 %0, 1, 0, P1;\n}\n"
      : "=r"(done)
      : "r"(smem_addr(mbar)), "r"(parity)
      : "memory");
  return done != 0;
}
// Named barriers of the slicers: 1 and 2 one group each (with a vote), 3 both.
QL_DEV bool group_or(int g, bool p) {
  uint32_t r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, 256, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)p), "r"(g + 1)
      : "memory");
  return r != 0;
}
QL_DEV void joint_sync() { asm volatile("bar.sync 3, 512;\n" ::: "memory"); }
// One box of a rank-3 tensor map (x = row in its 128-byte block, y = column, z = block).
QL_DEV void tma_load_3d(void* dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* mbar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];\n" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(mbar))
      : "memory");
}

// The MMAs of one tile (whole warp, issued by the elected lane): d0 is the descriptor of
// plane 0, k-step 0.
template <int NC>
QL_DEV void xg_issue_mmas(uint32_t leader, uint32_t tbase, uint64_t d0, bool fresh) {
  using Sh = XgShape<NC>;
  constexpr uint64_t PL = Sh::PLANE >> 4;
#pragma unroll 1
  for (int kk = 0; kk < Sh::KV / 16; ++kk) {
    const uint64_t dk = d0 + (uint64_t)((kk * 2 * Sh::LBO) >> 4);
    const uint32_t first = (!fresh || kk > 0) ? 1u : 0u;
    if constexpr (NC <= 16) {
      umma_bf16_if(leader, tbase, dk, dk, umma_idesc_bf16(128, 128), first);
    } else if constexpr (NC == 32) {
      umma_bf16_if(leader, tbase, dk, dk, umma_idesc_bf16(128, 256), first);
      umma_bf16_if(leader, tbase + 256, dk + 4 * PL, dk, umma_idesc_bf16(128, 256), first);
    } else {
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        bool opened = false;
#pragma unroll
        for (int p = -1; p <= 7; ++p) {
          const int q = 2 * b - p;
          if (q >= 0 && q <= 7) {
            umma_bf16_if(leader, tbase + (uint32_t)(b * 64), dk + (uint64_t)(int64_t)(p * (int64_t)PL),
                         dk + (uint64_t)q * PL, umma_idesc_bf16(128, 64), opened ? 1u : first);
            opened = true;
          }
        }
      }
    }
  }
}

// tcgen05.ld of one and two columns (the narrow classes).
QL_DEV void tmem_ld(uint32_t taddr, uint32_t (&v)[1]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(v[0]) : "r"(taddr));
}
QL_DEV void tmem_ld(uint32_t taddr, uint32_t (&v)[2]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];\n" : "=r"(v[0]), "=r"(v[1]) : "r"(taddr));
}

// c + a b, 32 x 32 bits into 64
QL_DEV long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
QL_DEV void store_i128(ulonglong2* p, i128 v) {
  __stcg(p, make_ulonglong2((u64)(u128)v, (u64)((u128)v >> 64)));
}

// Add v 2^s (0 <= s <= 184) to the limbs of one entry.
QL_DEV void sacc_add(long long* limbs, i128 v, int s) {
  if (v == 0) return;
  const bool neg = v < 0;
  u128 mag = neg ? (u128)(-v) : (u128)v;
  constexpr u64 kMask = (1ull << kLimbBits) - 1ull;
  int k = s / kLimbBits;
  const int off = s - k * kLimbBits;
  u64 c = ((u64)mag << off) & kMask;
  u128 rem = mag >> (kLimbBits - off);
  for (;;) {
    if (c) atomicAdd(reinterpret_cast<u64*>(limbs + k), neg ? (u64)0 - c : c);
    if (rem == 0) break;
    c = (u64)rem & kMask;
    rem >>= kLimbBits;
    ++k;
  }
}

// Magnitude (320 bits, little-endian words) and sign of an entry.
struct Wide320 {
  u64 w[5];
  bool neg;
};
QL_DEV Wide320 sacc_load(const long long* limbs) {
  long long l[kLimbs];
#pragma unroll
  for (int k = 0; k < kLimbs; k += 2) {
    const longlong2 t = __ldcg(reinterpret_cast<const longlong2*>(limbs + k));
    l[k] = t.x;
    l[k + 1] = t.y;
  }
  constexpr u64 kMask = (1ull << kLimbBits) - 1ull;
  u64 d[kLimbs];
  long long carry = 0;
#pragma unroll
  for (int k = 0; k < kLimbs; ++k) {
    const long long t = l[k] + carry;
    d[k] = (u64)t & kMask;
    carry = t >> kLimbBits;
  }
  Wide320 r;
  r.neg = carry < 0;
  if (r.neg) {  // two's complement over the eight limbs
    u64 c = 1;
#pragma unroll
    for (int k = 0; k < kLimbs; ++k) {
      const u64 t = ((~d[k]) & kMask) + c;
      d[k] = t & kMask;
      c = t >> kLimbBits;
    }
  }
  r.w[0] = d[0] | (d[1] << 40);
  r.w[1] = (d[1] >> 24) | (d[2] << 16) | (d[3] << 56);
  r.w[2] = (d[3] >> 8) | (d[4] << 32);
  r.w[3] = (d[4] >> 32) | (d[5] << 8) | (d[6] << 48);
  r.w[4] = (d[6] >> 16) | (d[7] << 24);
  return r;
}
QL_DEV int bit_length(const Wide320& a) {
#pragma unroll
  for (int k = 4; k >= 0; --k)
    if (a.w[k]) return 64 * k + 64 - __clzll((long long)a.w[k]);
  return 0;
}
// Bits [r, r + 128) of the magnitude (0 <= r).
QL_DEV u128 bits_at(const Wide320& a, int r) {
  const int wi = r >> 6, bi = r & 63;
  u64 x[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if (i == wi + k) x[k] = a.w[i];
  const u128 lo = ((u128)x[1] << 64) | x[0];
  if (bi == 0) return lo;
  return (lo >> bi) | ((u128)x[2] << (128 - bi));
}
// Signed magnitude times 2^e as a double (one rounding; mag fits in 128 bits).
QL_DEV double ldexp_pow2(double v, int e) {  // |e| may exceed one normal power of two
  while (e > 1000) {
    v *= 0x1p1000;
    e -= 1000;
  }
  while (e < -1000) {
    v *= 0x1p-1000;
    e += 1000;
  }
  return v * __longlong_as_double((long long)(e + 1023) << 52);
}
QL_DEV double mag_to_double(u128 mag, int e) {
  const u64 hi = (u64)(mag >> 64);
  if (hi == 0) {
    const u64 lo = (u64)mag;
    return lo ? ldexp_pow2(__ull2double_rn(lo), e) : 0.0;
  }
  const int z = __clzll((long long)hi);
  const u128 t = mag << z;
  const u64 top = (u64)(t >> 64) | ((u64)t != 0 ? 1ull : 0ull);  // sticky bit below the 64
  return ldexp_pow2(__ull2double_rn(top), e + 64 - z);
}
QL_DEV double wide_to_double(const Wide320& a, int e) {
  const int bl = bit_length(a);
  if (bl == 0) return 0.0;
  const int r = bl > 128 ? bl - 128 : 0;
  const double v = mag_to_double(bits_at(a, r), e + r);
  return a.neg ? -v : v;
}

// ---------------------------------------------------------------------------------------
// Cholesky factorisation of the exact Gram matrix in 125-bit fixed point, by one CTA.
// Column j is scaled by 2^-s_j so that 1/4 <= C_jj < 1; every later quantity (Schur
// complements, rows of R) stays below 1 in magnitude, so fixed point loses 2^-122 per
// operation and nothing to cancellation.  Integer multiplies run on the ALUs at full rate,
// where FP64 (1/64 of the FP32 rate) or double-double would not: a double-double version of
// the same factorisation needs about 0.9 M FP64 operations at n = 64, 0.2 ms on one SM.
// (The divisions lose 2^-99, see fx_div_pivot, where they are not refined.)
// 1 / sqrt(pivot) is formed in integers too, by one lane, while the other warps update the
// trailing rows (a chain of dependent FP64 instructions took several times as long).  A pivot below
// 2^-min_bits of its column, zero or negative stops the factorisation; a column that is zero
// altogether gives a zero row of R.  (What then happens is in xg_finish.)
// ---------------------------------------------------------------------------------------
constexpr int kFx = 125;

QL_DEV u64 umul_hi(u64 a, u64 b) { return __umul64hi(a, b); }
// (a b) 2^-kFx for |a|, |b| < 2^(kFx + 1); error below 2^4 units
QL_DEV i128 fx_mul(i128 a, i128 b) {
  const long long ah = (long long)(a >> 64), bh = (long long)(b >> 64);
  const u64 al = (u64)a, bl = (u64)b;
  i128 p = (i128)ah * bh;
  p += (i128)(u128)umul_hi((u64)ah, bl) - (ah < 0 ? (i128)(u128)bl : (i128)0);
  p += (i128)(u128)umul_hi((u64)bh, al) - (bh < 0 ? (i128)(u128)al : (i128)0);
  return p * 8;  // 2^128 / 2^125
}

// What a step needs of its pivot d = 2^-2z f, f in [1/4, 1): c ~ 1 / f in units of 2^-61
// (single precision and one Newton step: 2^-44) and the correction 1 / f = c (1 + eps), eps in
// units of 2^-102 (error 2^-102).
struct FxPivot {
  u64 c;
  long long eps;
  int z;
  int ok;  // 1: usable; 0: zero column; -1: pivot too small
};
QL_DEV int fx_half_lead(i128 d) {  // z with d 4^z in [1/4, 1)
  const u64 hi = (u64)((u128)d >> 64);
  const int lead = hi ? __clzll((long long)hi) : 64 + __clzll((long long)(u64)d);  // of 128 bits
  return (lead - (128 - kFx)) >> 1;
}
QL_DEV FxPivot fx_pivot(i128 d, bool zero_column, int min_bits) {
  FxPivot pv{0, 0, 0, 0};
  if (zero_column) return pv;
  if (d < ((i128)1 << (kFx - min_bits))) {
    pv.ok = -1;
    return pv;
  }
  pv.ok = 1;
  pv.z = fx_half_lead(d);
  const u128 f = (u128)d << (2 * pv.z);
  const u64 f64 = (u64)(f >> (kFx - 64));  // f 2^64
  const float y0 = __fdividef(1.0f, (float)(unsigned)(f64 >> 40) * 0x1p-24f);  // in [1, 4]
  const u64 c0 = (u64)(unsigned)(y0 * 0x1p21f) << 40;
  const long long e = (long long)((1ull << 61) - umul_hi(f64, c0));  // (1 - f y) 2^61
  const u64 de = umul_hi(c0, e < 0 ? (u64)-e : (u64)e) << 3;
  pv.c = e < 0 ? c0 - de : c0 + de;
  const u128 p = (u128)(u64)(f >> 64) * pv.c + umul_hi((u64)f, pv.c);  // f c 2^122
  const long long eps = (long long)((i128)(((u128)1 << 122) - p) >> 20);  // 2^102 (1 - f c)
  pv.eps = eps + (__mul64hi(eps, eps) >> 38);                              // + eps^2
  return pv;
}
// s / f in units of 2^-122 for s in units of 2^-kFx, |s / f| <= 2
QL_DEV i128 fx_div_pivot(i128 s, const FxPivot& pv) {
  const long long sh = (long long)(s >> 64);
  i128 w = (i128)(u128)umul_hi((u64)s, pv.c);
  // sh c, sh signed and c unsigned
  w += (i128)((u128)(u64)sh * pv.c) - (sh < 0 ? (i128)((u128)pv.c << 64) : (i128)0);
  return w + (i128)__mul64hi((long long)(w >> 61), pv.eps) * ((i128)1 << 23);
}
// w = s / f of fx_div_pivot with its residual divided once more: 2^-99 -> 2^-117.
QL_DEV i128 fx_div_refine(i128 w, i128 s, i128 f, const FxPivot& pv) {
  const long long r = (long long)((s >> 3) - fx_mul(f, w));  // units of 2^-122, below 2^-97
  return w + (((i128)r * (i128)(u128)pv.c) >> 61);
}
// 1 / (2 sqrt(f)) for f in [1/4, 1): single precision, one Newton step in 64-bit fixed point
// (2^-44), then one third-order step y (1 + e / 2 + 3 e^2 / 8), e = 1 - f y^2, in 128 bits.
QL_DEV i128 fx_half_rsqrt(i128 f) {
  const u64 f64 = (u64)(f >> (kFx - 64));  // f 2^64
  const float y0 = rsqrtf((float)(unsigned)(f64 >> 40) * 0x1p-24f);
  const u64 y = (u64)(unsigned)(y0 * 0x1p23f) << 39;  // y 2^62
  const long long e1 = (long long)((1ull << 60) - umul_hi(f64, umul_hi(y, y)));  // (1 - f y^2) 2^60
  const u64 d1 = umul_hi(y, e1 < 0 ? (u64)-e1 : (u64)e1) << 3;                   // |y e / 2| 2^62
  const u64 y1 = e1 < 0 ? y - d1 : y + d1;
  const i128 t = (i128)(((u128)y1 * y1) >> 1);  // y^2 / 4
  const i128 e = ((i128)1 << kFx) - fx_mul(f, t) * 4;
  const long long e64 = (long long)(e >> 20);         // e 2^105
  const i128 e2 = (i128)(__mul64hi(e64, e64) >> 21);  // e^2
  const i128 h = (i128)y1 << 62;                      // y / 2
  return h + fx_mul(h, (e >> 1) + (e2 * 3 >> 3));
}

// sacc -> Rout (n x n upper triangle, row-major, ld LE, in shared memory).  Shared memory from
// smem: two arrays of NC x LE words, then the scratch.  A pivot below 2^-min_bits of its
// column stops it, as does a zero column unless zero_ok.  Returns 0, or the 1-based index of
// the pivot that stopped it (to every thread).
//
// dependent: the second attempt of a call that a small pivot has stopped (of Cholesky-QR2 only if
// its own Cholesky would have answered).  The divisions are
// refined, which leaves Schur complements good to n 2^-117 (2^-99 otherwise), and a pivot below
// kDependentBits, half of what the Householder tiles' 48 bits could tell from zero, is the zero that
// they make of it: R_kk and its row vanish.  lstsq: a pivot of A between the limits (not the last
// one, the squared residual norm) stops the attempt, since the tiles may answer such a call or
// report it, depending on the order of the rows.
//
// Step k with pivot d = 2^-2z f keeps row k as s_j = S_kj 2^z and w_j = s_j / f, subtracts
// s_i w_j from the trailing entries and leaves 1 / sqrt(f) to the end (R_kj = s_j / sqrt(f),
// R_kk = 2^-z f / sqrt(f), all rows at once): the chain from one pivot to the next is a reciprocal and three multiplies.
constexpr int kDependentBits = 96;
template <int NC, int T, bool dependent>
QL_DEV int xg_cholesky(const long long* sacc, int n, unsigned char* smem, double* Rout, int min_bits, bool zero_ok,
                       bool lstsq) {
  constexpr int LE = NC + 1;
  u64* Slo = reinterpret_cast<u64*>(smem);
  long long* Shi = reinterpret_cast<long long*>(Slo + NC * LE);
  u64* Wlo = reinterpret_cast<u64*>(Shi + NC * LE);
  long long* Whi = reinterpret_cast<long long*>(Wlo + NC);
  FxPivot* piv = reinterpret_cast<FxPivot*>(Whi + NC);  // [2]
  int* sj = reinterpret_cast<int*>(piv + 2);            // column exponents
  int* zk = sj + NC;                                    // z of each pivot
  u64* fk = reinterpret_cast<u64*>(zk + NC);            // [2] f of the pivot, low and high word (dependent)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = T / 32;
  auto get = [&](int i, int j) -> i128 { return (i128)(((u128)(u64)Shi[i * LE + j] << 64) | Slo[i * LE + j]); };
  auto put = [&](int i, int j, i128 v) {
    Slo[i * LE + j] = (u64)(u128)v;
    Shi[i * LE + j] = (long long)(v >> 64);
  };
  for (int j = tid; j < n; j += T) {
    const Wide320 a = sacc_load(sacc + (size_t)tri_index(j, j) * kLimbs);
    const int bl = a.neg ? 0 : bit_length(a);
    sj[j] = bl ? (bl + 1) >> 1 : -1;
  }
  __syncthreads();
  const int ne = n * (n + 1) / 2;
#pragma unroll 2
  for (int e = tid; e < ne; e += T) {
    int j = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
    if (j * (j + 1) / 2 > e) --j;
    if ((j + 1) * (j + 2) / 2 <= e) ++j;
    const int i = e - j * (j + 1) / 2;
    const Wide320 a = sacc_load(sacc + (size_t)e * kLimbs);
    const int r = sj[i] + sj[j] - kFx;
    u128 mag = r > 0 ? (bits_at(a, r - 1) + 1) >> 1 : (((u128)a.w[1] << 64) | a.w[0]) << (-r);
    if (sj[i] < 0 || sj[j] < 0) mag = 0;
    put(i, j, a.neg ? -(i128)mag : (i128)mag);
  }
  __syncthreads();
  auto pivot = [&](int k, i128 d) {
    int limit = min_bits;
    bool zero = sj[k] < 0;
    if (dependent) {
      zero |= d < ((i128)1 << (kFx - kDependentBits));
      if (!lstsq || k == n - 1) limit = kFx;
    }
    FxPivot pv = fx_pivot(d, zero, limit);
    if (pv.ok == 0 && !zero_ok) pv.ok = -1;
    piv[k & 1] = pv;
    if (dependent) {
      const u128 f = (u128)d << (2 * pv.z);
      fk[2 * (k & 1)] = (u64)f;
      fk[2 * (k & 1) + 1] = (u64)(f >> 64);
    }
  };
  if (tid == 0) pivot(0, get(0, 0));
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    const FxPivot pv = piv[k & 1];
    if (pv.ok < 0) return k + 1;  // uniform
    for (int j = k + tid; j < n; j += T) {
      const i128 v = pv.ok ? get(k, j) << (j == k ? 2 * pv.z : pv.z) : (i128)0;  // S_kk becomes f
      put(k, j, v);
      if (j == k) zk[k] = pv.z;
      i128 w = j == k ? (i128)0 : fx_div_pivot(v, pv);
      if (dependent && j != k && pv.ok != 0) {
        const i128 f = (i128)(((u128)fk[2 * (k & 1) + 1] << 64) | fk[2 * (k & 1)]);
        w = fx_div_refine(w, v, f, pv);
      }
      Wlo[j] = (u64)(u128)w;
      Whi[j] = (long long)(w >> 64);
    }
    __syncthreads();
    auto update_row = [&](int i) {
      const i128 si = get(k, i);
      i128 first = 0;
      for (int j = i + lane; j < n; j += 32) {
        const i128 w = (i128)(((u128)(u64)Whi[j] << 64) | Wlo[j]);
        const i128 v = get(i, j) - fx_mul(si, w) * 8;  // units 2^-125 2^-122 2^128 / 2^3
        put(i, j, v);
        if (j == i) first = v;
      }
      return first;
    };
    if (warp == 0) {  // the next row, then its pivot
      if (k + 1 < n) {
        const i128 d = update_row(k + 1);
        if (lane == 0) pivot(k + 1, d);
      }
    } else {
      for (int i = k + 1 + warp; i < n; i += NW - 1) update_row(i);
    }
    __syncthreads();
  }
  for (int k = tid; k < n; k += T) {  // 1 / (2 sqrt(f))
    const i128 f = get(k, k), r = f == 0 ? (i128)0 : fx_half_rsqrt(f);
    Wlo[k] = (u64)(u128)r;
    Whi[k] = (long long)(r >> 64);
  }
  __syncthreads();
  for (int i = warp; i < n; i += NW)
    for (int j = lane; j < n; j += 32) {
      double r = 0.0;
      if (j >= i) {
        const i128 h = (i128)(((u128)(u64)Whi[i] << 64) | Wlo[i]);
        const i128 v = fx_mul(get(i, j), h);
        r = mag_to_double(v < 0 ? (u128)-v : (u128)v, sj[j] + 1 - (j == i ? zk[i] : 0) - kFx + kXgUnitExp / 2);
        if (v < 0) r = -r;
      }
      Rout[i * LE + j] = r;
    }
  __syncthreads();
  return 0;
}

// The second attempt, apart from the kernel's code: small calls feel its instruction cache.  (One
// copy with a switch at run time took 2 us of 35 at 131072 x 8.)
template <int NC, int T>
__device__ __noinline__ bool xg_cholesky_dependent(const long long* sacc, int n, unsigned char* smem, double* Rout, int min_bits,
                                                   bool zero_ok, bool lstsq) {
  return xg_cholesky<NC, T, true>(sacc, n, smem, Rout, min_bits, zero_ok, lstsq) == 0;
}

// Whether SVQB would keep every eigenvalue of C = R^T R: lambda_min > tol lambda_max, shown by
// tol trace(C) ||R^{-1}||_F^2 <= 1/16 (trace >= lambda_max, ||R^{-1}||_F^2 >= 1 / lambda_min).  R in
// shared memory (ld LE), scaled by rows of its inverse in FP32: good to a few per cent up to
// the condition numbers (about 10^6) where the answer can be yes.  One warp per column.
template <int NC, int T>
QL_DEV bool svqb_full_rank(const double* R, int n, double tol, float* sums) {
  constexpr int LE = NC + 1, NW = T / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // scale by the largest column norm so that FP32 covers the range
  if (threadIdx.x < 2) sums[threadIdx.x] = 0.0f;
  double big = 0.0;
  for (int i = 0; i < n; ++i) big = fmax(big, fabs(R[i * LE + i]));
  if (!(big > 0.0) || !isfinite(big)) return false;  // uniform
  const double inv = 1.0 / big;
  __syncthreads();
  float tr = 0.0f, fr = 0.0f;
  for (int c = warp; c < n; c += NW) {
    float x0 = 0.0f, x1 = 0.0f;  // rows lane, lane + 32 of the right-hand side, e_c at the start
    if (lane == (c & 31)) (c < 32 ? x0 : x1) = 1.0f;
    for (int i = c; i >= 0; --i) {
      const float xi =
          __shfl_sync(0xffffffffu, i < 32 ? x0 : x1, i & 31) / (float)(R[i * LE + i] * inv);
      fr = fmaf(xi, xi, fr);
      if (lane < i) x0 = fmaf(-(float)(R[lane * LE + i] * inv), xi, x0);
      if (NC > 32 && lane + 32 < i) x1 = fmaf(-(float)(R[(lane + 32) * LE + i] * inv), xi, x1);
    }
    for (int i = lane; i <= c; i += 32) {
      const float v = (float)(R[i * LE + c] * inv);
      tr = fmaf(v, v, tr);
    }
  }
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
  if (lane == 0) {
    atomicAdd(&sums[0], tr);
    atomicAdd(&sums[1], fr);
  }
  __syncthreads();
  const double bound = tol * (double)sums[0] * (double)sums[1];
  return bound <= 0.0625;
}

// Whether the fixed point has lost rows that R depends on.  An entry is held to 2^-54 to 2^-53 of
// the largest entry that its CTA has met in the column, not to 48 bits of its own as in the
// Householder tiles and the SIMT Gram passes.  That matters where a few heavy rows (weighted or
// constraint rows of a least-squares problem) stand above light ones and do not determine every
// column: then R_kk, made of light rows, is small against the column's largest entry, and its
// error of about 2^-56 of that entry is not (m = 2^14, n = 3, first row 2^30 times the others: R was
// 3e-11 off, the Householder tiles 2e-15).  So: column k has light entries (kLightBits below its
// scale in a CTA's last two tiles, for eight rows together or for most of the rows), and R_kk is below four times its
// largest entry.  Neither alone would do: Gaussian columns of any condition number show no light
// units, and light rows beside a large R_kk change nothing.
constexpr int kLightBits = 8;
// E: largest exponent of column k, mask: the word of flags[6], [7] with its bit.
QL_DEV double light_floor(int E, int mask, int k) {  // R_kk below it: lost (0: column k has no light entries)
  return E > 0 && ((mask >> (k & 31)) & 1) ? __longlong_as_double((long long)(E + 2) << 52) : 0.0;
}

// One unit of a column: with bal, its nonzero entries below the light limit count 1 and the others
// -1; a unit that is light in all eight rows sets *lit.
template <typename S>
QL_DEV void count_light(const Rows8<S>& v, int limit, int* bal, int* lit) {
  int below = 0, above = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned ax = v.hw[j] & 0x7fffffffu;
    if (ax) ++(Rows8<S>::exponent(ax) < limit ? below : above);
  }
  if (bal && below != above) atomicAdd(bal, below - above);
  if (below == 8) *lit = 1;
}

// Range verdict, election of the last CTA and, in it, R from the fixed-point Cholesky.  The
// Gram methods end here as well when their further passes could not change R: with C exact
// and factored to 2^-90, Y = X R1^{-1} is orthonormal to working precision and R2 the identity.
// flags[5] then tells the later launches of the call.  What a method answers beyond that
// range is left to its passes: Cholesky-QR2 where its first Cholesky, FP64 of C, breaks down (asked
// below pivots of 2^-46; the R it accepts is then factored again in fixed point), shifted Cholesky-QR3 from 2^-66, SVQB2 when an eigenvalue could be
// truncated or Z is wanted; a zero column breaks down there.  A TSQR call whose pivots fall below
// 2^-80 is factored again as dependent (see xg_cholesky).  One that this does not answer is redone
// by the Householder launch (flags[1]), as is one that has lost light rows; so are
// Gram calls of up to 8 columns by their passes (of 48-bit entries; those of 9 columns and more hold
// X in fixed point themselves).
template <int NC, int T, typename S>
QL_DEV void xg_finish(const GramArgs<S>& a, unsigned char* smem, const int* colmax, int* misc, int k) {
  if (!gram_elect<S, ArithDF>(a, colmax, misc, k)) return;
  const int tid = threadIdx.x, n = a.n;
  constexpr int LE = NC + 1;
  const bool tsqr = a.method == QL_TSQR;
  if (tsqr && *(volatile int*)&a.w.flags[1] != 0) {  // a bounded wait gave up: Householder redoes the call
    if (a.redo && tid == 0) gram_request_redo(a.redo, a.redo_any, *(volatile int*)&a.w.flags[4], kRedoDF);
    return;
  }
  double* Rs = reinterpret_cast<double*>(smem);
  double* vec = Rs + NC * LE;
  int* sflag = reinterpret_cast<int*>(vec + 2 * LE);
  unsigned char* scratch = smem + ((NC + 3) * LE * 8 + 255) / 256 * 256;
  const int min_bits = tsqr ? 80 : (a.method == QL_SCHOLQR3 ? 66 : 46);
  const bool check_light = tid < n && (tsqr || NC <= 8);
  const int E = check_light ? __ldcg(&a.w.flags[64 + tid]) : 0, mask = check_light ? __ldcg(&a.w.flags[6 + (tid >> 5)]) : 0;
  auto load_c = [&]() {  // C in FP64 (Rs)
    __syncthreads();
    for (int i = tid >> 5; i < n; i += T / 32)
      for (int j = i + (tid & 31); j < n; j += 32) {
        const double v = wide_to_double(sacc_load(a.w.sacc + (size_t)tri_index(i, j) * kLimbs), kXgUnitExp);
        Rs[i * LE + j] = v;
        Rs[j * LE + i] = v;
      }
    __syncthreads();
  };
  bool done = false;
  if (a.method != QL_SVQB2 || !a.Z) {
    done = xg_cholesky<NC, T, false>(a.w.sacc, n, scratch, Rs, min_bits, tsqr, false) == 0;
    if (!done && (tsqr || a.method == QL_CHOLQR2)) {
      __syncthreads();  // the scratch is written again
      bool again = true;
      if (!tsqr) {  // would its own first Cholesky answer?
        load_c();
        again = chol_upper_inplace<T>(Rs, LE, n, sflag) == 0;
        __syncthreads();
      }
      if (again) done = xg_cholesky_dependent<NC, T>(a.w.sacc, n, scratch, Rs, min_bits, tsqr, tsqr && a.epilogue == kEpiLstsq);
    }
    if (done && a.method == QL_SVQB2)
      done = svqb_full_rank<NC, T>(Rs, n, a.rank_tol > 0.0 ? a.rank_tol : (double)n * 2.220446049250313e-16,
                                   reinterpret_cast<float*>(sflag));
  }
  // (the barrier: the scratch is reused)
  if (__syncthreads_or(done && check_light && fabs(Rs[tid * LE + tid]) < light_floor(E, mask, tid))) done = false;
  if (done) {
    if (!tsqr && tid == 0) a.w.flags[5] = 1;
    if (a.epilogue == kEpiR)
      epilogue_r<T>(Rs, LE, n, a.R, a.ldr, a.info, sflag);
    else
      epilogue_lstsq<T>(Rs, LE, n, a.x, a.resnorm, a.Rext, a.info, vec, sflag);
    return;
  }
  if (tsqr) {
    if (tid == 0) {
      a.w.flags[1] = 1;
      if (a.redo) gram_request_redo(a.redo, a.redo_any, 0, kRedoDF);
    }
    return;
  }
  load_c();
  gram_epilogue<NC, T, S, ArithDF>(a, smem);
}

// Row tiles [tiles bid / k, tiles (bid + 1) / k) of one problem; tensor memory at tbase and
// barriers set up by xg_cta_begin, phases carried in bars (see gram_pipe_body).
template <int NC, typename S>
QL_DEV void xgram_body(GramArgs<S> a, int bid, int k, uint32_t tbase, PipeBars& bars, const CUtensorMap* map,
                       int slot) {
  using Sh = XgShape<NC>;
  using Sm = XgSmem<NC, S>;
  constexpr int T = Sh::T, TS = Sh::TS, KT = Sh::KT, PLANE = Sh::PLANE, SBO = Sh::SBO, LBO = Sh::LBO, HALF = Sh::HALF,
                RPB = Sm::RPB, LG = Sh::LG, VC = Sh::VC, SEG = Sh::SEG, KV = Sh::KV;
  extern __shared__ __align__(1024) unsigned char smem_umma[];
  unsigned char* smem = smem_umma;
  const int tid = threadIdx.x, n = a.n, lane = tid & 31, warp = tid >> 5;
  const bool control = warp >= TS / 32;  // copy warp, MMA warp
  auto digits = [&](int b) { return smem + Sh::PAD + (size_t)b * (Sh::DBUF + Sh::PAD); };
  unsigned char* raw0 = smem + Sm::kOffRaw;
  unsigned char* rhs0 = smem + Sm::kOffB;
  int* scale = reinterpret_cast<int*>(smem + Sm::kOffScale);
  int* colmax = reinterpret_cast<int*>(smem + Sm::kOffColmax);
  int* bal = reinterpret_cast<int*>(smem + Sm::kOffBal);
  int* lit = reinterpret_cast<int*>(smem + Sm::kOffLit);
  int* misc = reinterpret_cast<int*>(smem + Sm::kOffMisc);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem + Sm::kOffBar);  // [2] MMAs done, per digit buffer
  uint64_t* lbar = mbar + 2;                                          // [2] tile landed, per raw stage
  uint64_t* dbar = mbar + 4;                                          // [2] digits ready, per digit buffer
  uint64_t* rbar = mbar + 6;                                          // [2] stage read, per raw stage
  uint64_t* vbar = mbar + 8;                                          // [2] vote passed, per slicer group
  int* place = reinterpret_cast<int*>(smem + Sm::kOffSlot + 4);       // [2] the tile's place in its read-out
  volatile int* fail = place + 2;                                     // where the first wait gave up
  volatile int* req = place + 3;                                      // a column outgrew its scale
  volatile int* pos = place + 4;                                      // [2] next tile of each group

  a.tiles = (a.m + KT - 1) / KT;
  for (int i = tid; i < NC; i += T) {
    colmax[i] = 0;
    scale[i] = 0;
    bal[i] = 0;
    lit[i] = 0;
  }
  if (tid == 0) *fail = 0;
  if (tid == 0) *req = 0;
  if constexpr (Sh::PAD > 0) {
    for (int z = 0; z < 3; ++z)
      for (int i = tid; i < Sh::PAD / 16; i += T)
        *reinterpret_cast<uint4*>(smem + (size_t)z * (Sh::DBUF + Sh::PAD) + 16 * i) = make_uint4(0, 0, 0, 0);
  }
  // the generic writes so far (a previous work item's included) come before the copies and
  // the MMA operand reads
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  const int64_t t0 = a.tiles * bid / k;
  const int nt = (int)(a.tiles * (bid + 1) / k - t0);  // tiles of this CTA, i = 0 .. nt - 1
  // full tiles (i < nbulk) arrive by tensor copies when the columns allow them; the last rows
  // of the matrix, and unaligned columns, are read by the slicers from global memory
  const int nbulk = a.bulk ? (int)max((int64_t)0, min((int64_t)nt, a.m / KT - t0)) : 0;
  // tile i = 2 j + b uses stage and buffer b; the phase of its barriers has this parity
  auto par = [&](int i) { return ((bars.mpar >> (i & 1)) ^ (uint32_t)(i >> 1)) & 1u; };
  auto lpar = [&](int i) { return ((bars.lpar >> (i & 1)) ^ (uint32_t)(i >> 1)) & 1u; };

  // read-out role: TMEM lane quarter qd, columns hh HALF + [0, HALF) of C; lane L belongs to
  // lane group lg (plane, or weight parity), row segment seg and row li of C
  const int qd = warp & 3, hh = (warp >> 2) & 3;
  const int L = 32 * qd + lane, lg = L / VC, seg = L % VC / NC, li = L % NC;
  const int g = warp >> 3;  // slicer group
  ulonglong2* acc = reinterpret_cast<ulonglong2*>(a.w.fbuf) + (size_t)slot * NC * 128;  // [column][lane]

  if (warp == TS / 32) {
    // ---- copy warp: two tiles ahead, a tile per instruction (one box of the rank-3 map); once
    // the slicers have read a stage, the copy two ahead goes into it
    const uint32_t leader = elect_one();
    const bool has_b = a.src.nA < n;
    int issued = 0;  // tiles 0 .. issued - 1
    auto copy = [&]() {
      const int b = issued & 1;
      const int64_t row0 = (t0 + issued) * KT;
      if (leader) {
        mbar_arrive_expect_tx(&lbar[b], (uint32_t)(Sm::kRaw + (has_b ? Sm::kStageB : 0)));
        tma_load_3d(raw0 + (size_t)b * Sm::kRaw, map, 0, 0, (int)(row0 / RPB), &lbar[b]);
        if (has_b) bulk_g2s(rhs0 + (size_t)b * Sm::kStageB, a.src.b + row0, (uint32_t)Sm::kStageB, &lbar[b]);
      }
      __syncwarp();
      ++issued;
    };
    while (issued < 2 && issued < nbulk) copy();
    bool ok = true;
    for (int i = 0; i + 2 < nbulk && ok; ++i) {
      ok = __all_sync(0xffffffffu, xg_wait(&rbar[i & 1], par(i), fail, 2));
      if (ok) copy();
    }
    // no copy may still be writing when the CTA moves on
    for (int i = issued > 2 ? issued - 2 : 0; i < issued; ++i) mbar_wait_bounded(&lbar[i & 1], lpar(i));
  } else if (control) {
    // ---- MMA warp: once a tile's digits are ready, its MMAs.  Planes and k-steps add (byte
    // offset >> 4) to the 14-bit address field, which stays below 2^14 (shared addresses
    // < 256 KB); plane -1 is the zero plane before the buffer.
    const uint32_t leader = elect_one();
    const uint64_t d0 = umma_sdesc(smem_addr(digits(0)), LBO, SBO);
    for (int i = 0; i < nt; ++i) {
      const int b = i & 1;
      if (!__all_sync(0xffffffffu, xg_wait(&dbar[b], par(i), fail, 2))) break;
      tc_fence_after();
      const int at = place[b];
      xg_issue_mmas<NC>(leader, tbase + (uint32_t)(at / Sh::G * Sh::SCOLS), d0 + (uint64_t)b * ((Sh::DBUF + Sh::PAD) >> 4),
                        at % Sh::G == 0);
      umma_commit_if(leader, &mbar[b]);
      __syncwarp();
    }
  } else {
    // ---- slicer warps
    int nread = 0;       // read-outs in the 128-bit sums since they were last emptied

    // Tensor-memory sums -> 128-bit integers.  A thread folds the eight sums of its (lane,
    // column): digits q of the other factor for NC <= 32 (planes p and p + 4 for NC = 32),
    // the eight weights of its parity for NC = 64.
    // Eight sums d_q of spacing 7 or 14 bits are gathered by widening multiply-adds (one
    // instruction each) into 64-bit groups at 32-bit offsets, then carried into 128 bits.  Rows
    // of C below the diagonal block of the warp are not folded (NC = 64: a quarter of the work).
    auto readout = [&](int sets) {
      constexpr int JS = NC == 4 ? 1 : (NC == 64 ? 4 : 2);
      const uint32_t lane_base = tbase + ((uint32_t)(32 * qd) << 16) + (uint32_t)(hh * HALF);
      const bool keep = nread++ > 0;  // uniform: every slicer counts the read-outs
#pragma unroll 1
      for (int c0 = 0; c0 < HALF; c0 += JS) {
        if (NC == 64 && hh * HALF + c0 + JS <= 32 * (qd & 1)) continue;  // columns left of every row of the warp
        ulonglong2* p = acc + (size_t)(hh * HALF + c0) * 128 + L;
        ulonglong2 old[JS];
#pragma unroll
        for (int j = 0; j < JS; ++j) old[j] = keep ? __ldcg(p + j * 128) : make_ulonglong2(0, 0);
        i128 sum[JS];
#pragma unroll
        for (int part = 0; part < (NC == 32 ? 2 : 1); ++part) {
          int dq[JS][8];
#pragma unroll 1
          for (int set = 0; set < (Sh::NS == 1 ? 1 : sets); ++set) {
            uint32_t v[8][JS];
#pragma unroll
            for (int sg = 0; sg < SEG; ++sg) {  // a lane keeps the columns of its own segment
              uint32_t w[8][JS];
#pragma unroll
              for (int q = 0; q < 8; ++q)
                tmem_ld(lane_base + (uint32_t)(set * Sh::SCOLS + part * 256 + q * VC + sg * NC + c0), w[q]);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int j = 0; j < JS; ++j) v[q][j] = sg == 0 || sg == seg ? w[q][j] : v[q][j];
            }
#pragma unroll
            for (int j = 0; j < JS; ++j)
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int t = __float2int_rn(__uint_as_float(v[q][j]));
                dq[j][q] = set == 0 ? t : dq[j][q] + t;  // at most 16 2^24
              }
          }
#pragma unroll
          for (int j = 0; j < JS; ++j) {
            const int(&d)[8] = dq[j];
            if constexpr (NC == 64) {  // offsets 0, 14, .., 98
              const long long a0 = mad_wide(d[5], 1 << 28, mad_wide(d[6], 1 << 14, (long long)d[7]));
              const long long a1 = mad_wide(d[3], 1 << 24, mad_wide(d[4], 1 << 10, a0 >> 32));
              const long long a2 = mad_wide(d[1], 1 << 20, mad_wide(d[2], 1 << 6, a1 >> 32));
              const long long a3 = mad_wide(d[0], 1 << 2, a2 >> 32);
              sum[j] = (i128)(((u128)(u64)(((u64)(unsigned)a3 << 32) | (unsigned)a2) << 64) |
                              (((u64)(unsigned)a1 << 32) | (unsigned)a0));
            } else {  // offsets 0, 7, .., 49
              const long long l =
                  mad_wide(d[4], 1 << 21, mad_wide(d[5], 1 << 14, mad_wide(d[6], 1 << 7, (long long)d[7])));
              const long long h =
                  mad_wide(d[0], 1 << 21, mad_wide(d[1], 1 << 14, mad_wide(d[2], 1 << 7, (long long)d[3])));
              const i128 t = ((i128)h << 28) + l;
              sum[j] = part == 0 ? t : (sum[j] << 28) + t;
            }
          }
        }
#pragma unroll
        for (int j = 0; j < JS; ++j)
          store_i128(p + j * 128, (i128)(((u128)old[j].y << 64) | old[j].x) + sum[j]);
      }
    };
    // 128-bit sums -> the integer accumulators of C at the current column scales.  Lane groups
    // 1.. hand their sums to group 0 through `scratch` (a free digit buffer).
    auto emit = [&](unsigned char* scratch) {
      pdl_wait();  // the accumulators have been cleared
      ulonglong2* sc = reinterpret_cast<ulonglong2*>(scratch);
      if (lg + seg > 0) {
        constexpr int JB = HALF < 8 ? HALF : 8;
#pragma unroll 1
        for (int j0 = 0; j0 < HALF; j0 += JB) {
          ulonglong2 t[JB];
#pragma unroll
          for (int j = 0; j < JB; ++j) t[j] = __ldcg(acc + (size_t)(hh * HALF + j0 + j) * 128 + L);
#pragma unroll
          for (int j = 0; j < JB; ++j) sc[((size_t)(lg * SEG + seg - 1) * NC + li) * NC + hh * HALF + j0 + j] = t[j];
        }
      }
      joint_sync();
      if (lg + seg == 0 && li < n) {
        const int si = scale[li];
        ulonglong2 next = __ldcg(acc + (size_t)(hh * HALF) * 128 + L);
#pragma unroll 1
        for (int j = 0; j < HALF; ++j) {
          const int jj = hh * HALF + j;
          i128 v = (i128)(((u128)next.y << 64) | next.x);
          if (j + 1 < HALF) next = __ldcg(acc + (size_t)(jj + 1) * 128 + L);
          if (jj < li || jj >= n) continue;
          auto part = [&](int g) -> i128 {
            const ulonglong2 t = sc[((size_t)(g - 1) * NC + li) * NC + jj];  // g = lane group SEG + segment
            return (i128)(((u128)t.y << 64) | t.x);
          };
          if constexpr (NC == 64) {
            v += part(1) >> 7;  // odd weights: a multiple of 2^7 (weight 15 is empty)
          } else {
#pragma unroll 1
            for (int g = 1; g < LG * SEG; ++g) v = (g % SEG == 0 ? v * 128 : v) + part(g);
          }
          const int sj = scale[jj];
          if (si >= kEsMin && sj >= kEsMin && si <= kEsMax && sj <= kEsMax)  // else flagged at the end, or zero
            sacc_add(a.w.sacc + (size_t)tri_index(li, jj) * kLimbs, v, si + sj - 2 * kEsMin);
        }
      }
      joint_sync();
      nread = 0;
    };

    // This thread's two units of a tile: rows r0 .. r0 + 7 of column cu; eight consecutive threads
    // hold eight consecutive columns of a digit plane, so their stores fill whole core-matrix
    // rows.  Plane column cv and row rv are column cv % NC, row rv of segment cv / NC.
    constexpr int TG = Sh::TG;
    const int gt = tid & (TG - 1);
    int cu[2], r0[2];
    const unsigned char* line[2];  // the unit in its 128-byte line of the staged tile (or in the
    // right-hand side): chunk q of 16 bytes at this address ^ 16 q (the swizzle and the unit's
    // first chunk, a multiple of its chunks, only flip other bits or the same ones)
    bool live[2];
    unsigned arun[2] = {0, 0};  // largest |x| the unit's column has shown (range record)
    unsigned char* dst[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int w = (gt >> 3) + u * (TG / 8), cv = 8 * (w / (KV / 8)) + (gt & 7), rv = 8 * (w % (KV / 8));
      cu[u] = cv % NC;
      r0[u] = cv / NC * KV + rv;
      live[u] = cu[u] < n;
      const int line_no = (r0[u] / RPB) * NC + cu[u];
      const bool rhs_unit = cu[u] == a.src.nA;
      line[u] = rhs_unit ? rhs0 + (size_t)g * Sm::kStageB + r0[u] * sizeof(S)
                         : raw0 + (size_t)g * Sm::kRaw + (size_t)line_no * 128 +
                               ((((r0[u] % RPB) * (int)sizeof(S) / 16) ^ (line_no & 7)) << 4);
      dst[u] = digits(g) + (cv >> 3) * SBO + (cv & 7) * 16 + (rv >> 3) * LBO;
    }
    auto clear_dead = [&]() {  // columns past n: zero digits
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (!live[u])
#pragma unroll
          for (int p = 0; p < 8; ++p) *reinterpret_cast<uint4*>(dst[u] + p * PLANE) = make_uint4(0, 0, 0, 0);
    };
    clear_dead();

    Rows8<S> v[2];
    // tile i: loaded into v, voted on (no column of it outgrows its scale), cut into its buffer
    // (freed: its stage has been given back)
    bool have = false, freed = false, voted = false, cut = false, over[2] = {false, false};
    int es[2] = {0, 0};
    int i = g;                 // this group's next tile
    int first = 0;             // first tile of the sums in tensor memory
    int done0 = 0, done1 = 1;  // the groups' positions at the last meeting
    for (;;) {
      bool meet = i >= nt;  // uniform in the group, like every flag but over
      if (!meet) {
        if (!have) {
          const bool bulk = i < nbulk;
          if (bulk) xg_wait(&lbar[g], lpar(i), fail, 1);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!live[u]) continue;
            if (bulk) {
#pragma unroll
              for (int q = 0; q < 8 * (int)sizeof(S) / 16; ++q)
                v[u].chunk(q, *reinterpret_cast<const uint4*>(reinterpret_cast<uintptr_t>(line[u]) ^ (uintptr_t)(16 * q)));
            } else {
              const int64_t row = (t0 + i) * KT + r0[u], left = a.m - row;
              const S* col = a.src.col(cu[u]) + row;
#pragma unroll
              for (int j = 0; j < 8; ++j) v[u].set(j, j < left ? __ldg(col + j) : S(0));
            }
          }
          have = true;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!live[u]) continue;
            const unsigned am = v[u].amax();
            arun[u] = max(arun[u], am);
            es[u] = Rows8<S>::exponent(am);
          }
        }
        if (!voted) {
          const int above0 = live[0] ? es[0] - scale[cu[0]] : 0, above1 = live[1] ? es[1] - scale[cu[1]] : 0;
          const bool above = max(above0, above1) > 0;  // needs every element of both units
          over[0] = above0 > 0;
          over[1] = above1 > 0;
          // the other group's vote on the tile before comes first, or it has stopped
          bool passed = i == 0;
          while (!passed && !*req && !*fail) passed = mbar_test_wait(&vbar[g ^ 1], par(i - 1));
          voted = !group_or(g, above | (!passed & !*fail));
          // The copy warp may refill the stage only now: the vote took every element of every
          // thread, so all loads have returned.  An arrival right after the loads does not wait
          // for them (the copy of the tile two ahead overtook loads in flight, seen with the
          // right-hand side of a 4-column class in L2).
          if (gt == 0 && !freed) mbar_arrive(&rbar[g]);
          freed = true;
          if (voted && gt == 0) mbar_arrive(&vbar[g]);
        }
        if (voted && !cut) {
          if (i >= 2) xg_wait(&mbar[g], par(i - 2), fail, 2);  // the MMAs are done with this buffer
          // eight digits of every element
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (!live[u]) continue;
            const int base = Rows8<S>::base(scale[cu[u]]);
            int sh[8], any = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              sh[j] = v[u].shift(j, base);
              any |= sh[j];
            }
            unsigned sg[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              sg[e] = __byte_perm(v[u].hw[2 * e], v[u].hw[2 * e + 1], 0x7632) & 0x80008000u;
            u64 Nb[8];
            if (any & Rows8<S>::kFar) {  // an element more than 2^24 below the scale (or zero)
#pragma unroll
              for (int j = 0; j < 8; ++j) Nb[j] = cut56<true>(v[u].h(j), v[u].l(j), sh[j] & (Rows8<S>::kWrap - 1));
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) Nb[j] = cut56<false>(v[u].h(j), v[u].l(j), sh[j]);
            }
            put_plane_pairs<PLANE, 0>(dst[u], Nb, sg);
          }
          cut = true;
        }
        meet = !voted || i >= first + Sh::GT;
      }
      if (meet) {
        // ---- both groups meet: read the sums out, and empty the 128-bit ones when a scale
        // rises (their unit changes) or they are full, and at the end
        if (have && !voted && (over[0] || over[1])) *req = 1;
        if (gt == 0) pos[g] = i;
        joint_sync();
        const int p0 = pos[0], p1 = pos[1];  // the first tile of each group not handed over
        const bool raise = *req != 0, last = p0 >= nt && p1 >= nt;
        if (p0 > done0 || p1 > done1) {
          if (p0 > 0) xg_wait(&mbar[0], par(p0 - 2), fail, 2);
          if (p1 > 1) xg_wait(&mbar[1], par(p1 - 2), fail, 2);
          tc_fence_after();
          readout((min(p0, p1) - first + Sh::G - 1) / Sh::G);
        }
        const bool empty = nread > 0 && (raise || last || nread >= Sh::MAX_READS);
        if (empty) {
          emit(digits(0));  // every MMA is done: the buffers are free, and cut again below
          clear_dead();
        }
        joint_sync();  // every read of the flags, the scales and the sums is done
        if (last) break;
        if (raise) {
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (have && !voted && over[u]) atomicMax(&scale[cu[u]], max(es[u] + Sh::SLACK, kEsMin));
          if (tid == 0) *req = 0;
        }
        joint_sync();
        if (raise || empty) cut = false;
        done0 = p0;
        done1 = p1;
        first = min(p0, p1);
        continue;
      }
      if (gt == 0) place[g] = i - first;
      fence_proxy_async_smem();  // the digit planes are read by the tensor core
      tc_fence_before();         // the read-out's TMEM loads come before the next MMAs
      __syncwarp();
      if (lane == 0) mbar_arrive(&dbar[g]);
      have = freed = voted = cut = false;
      i += 2;
    }
    // Light data (see light_floor) is looked for in each group's last tile, which v still holds,
    // against the final scales: all units, the single entries of a column's first 32 rows.  (In the
    // loop, where it holds registers, the look took 2 to 4 %, in sampled tiles as well.)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (!live[u]) continue;
      if (arun[u] > 0) atomicMax(&colmax[cu[u]], Rows8<S>::exponent(arun[u]));
      if (i > g) count_light(v[u], scale[cu[u]] - kLightBits, r0[u] % KV < 32 ? bal + cu[u] : nullptr, lit + cu[u]);
    }
  }
  // every thread carries the same phase counts to the next work item
  bars.mpar ^= (uint32_t)(((nt + 1) >> 1) & 1) | (uint32_t)((nt >> 1) & 1) << 1;
  bars.lpar ^= (uint32_t)(((nbulk + 1) >> 1) & 1) | (uint32_t)((nbulk >> 1) & 1) << 1;
  tc_fence_before();
  __syncthreads();
  const int fw = *fail;
  pdl_wait();  // before the first use of the flags
  if (fw) {
    bars.ok = false;  // a late arrival may still complete a phase: the CTA takes no more work
    if (tid == 0) {   // the gated launches redo the call and report {QL_ERR_TIMEOUT, where}
      atomicCAS(&a.w.flags[4], 0, fw);
      atomicOr(&a.w.flags[a.method == QL_TSQR ? 1 : 0], 2);
    }
  }
  for (int cc = tid; cc < n; cc += T) {  // column exponents of the whole matrix, for the later passes
    if (colmax[cc] > 0) atomicMax(&a.w.flags[64 + cc], colmax[cc]);
    if (lit[cc] || bal[cc] >= 4)  // four: a ragged tile may hold few rows of a column
      atomicOr(&a.w.flags[6 + (cc >> 5)], 1 << (cc & 31));
  }
  xg_finish<NC, T, S>(a, smem, colmax, misc, k);
}

template <int NC, typename S>
QL_DEV uint32_t xg_cta_begin(unsigned char* smem) {
  using Sm = XgSmem<NC, S>;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + Sm::kOffSlot);
  if ((threadIdx.x >> 5) == 0) tmem_alloc(tslot, 512);
  if (threadIdx.x == 0) {
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + Sm::kOffBar);
    for (int i = 0; i < 4; ++i) mbar_init(bar + i, 1);
    for (int i = 4; i < 6; ++i) mbar_init(bar + i, XgShape<NC>::TG / 32);  // one arrival per warp of the group
    for (int i = 6; i < 10; ++i) mbar_init(bar + i, 1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return *tslot;
}

template <int NC, typename S>
__global__ void __launch_bounds__(XgShape<NC>::T, 1)
    xgram_kernel(const __grid_constant__ GramArgs<S> a, const __grid_constant__ CUtensorMap map) {
  extern __shared__ __align__(1024) unsigned char smem_umma[];
  // The kernel before this one, which this one may overlap, is an ordinary launch (so X was
  // complete before it started) that clears the head of the workspace alone: nothing in the head,
  // flags and integer accumulators, is touched before pdl_wait.  The CTA's own 128-bit sums (fbuf)
  // are used before it; they must never be cleared there.
  pdl_release();
  const uint32_t tbase = xg_cta_begin<NC, S>(smem_umma);
  PipeBars bars;
  xgram_body<NC, S>(a, blockIdx.x, gridDim.x, tbase, bars, &map, blockIdx.x);
  tc_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tmem_dealloc(tbase, 512);
}

template <int NC, typename S>
ql_status xgram_launch_one(const GramCall& c, const GramWs& w) {
  using Sh = XgShape<NC>;
  using Sm = XgSmem<NC, S>;
  auto kern = xgram_kernel<NC, S>;
  static bool ready_on[kMaxDevices] = {};
  bool& ready = ready_on[device_slot()];
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!ready) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sm::kBytes) != cudaSuccess)
        return QL_ERR_CUDA;
      ready = true;
    }
  }
  const int64_t tiles = (c.m + Sh::KT - 1) / Sh::KT;
  int64_t g = (int64_t)device_sm_count();  // one CTA per SM: the shared memory allows no second one
  if (g > tiles) g = tiles;
  if (g < 1) g = 1;
  GramArgs<S> a{};
  a.src.A = static_cast<const S*>(c.A);
  a.src.lda = c.lda;
  a.src.b = static_cast<const S*>(c.b);
  a.src.nA = c.nA;
  a.m = c.m;
  a.n = c.n;
  a.tiles = tiles;
  a.pass = 1;
  a.method = c.method;
  a.epilogue = c.epilogue;
  a.w = w;
  a.R = c.R;
  a.ldr = c.ldr;
  a.Z = c.Z;
  a.rank_tol = c.rank_tol;
  a.x = c.x;
  a.resnorm = c.resnorm;
  a.Rext = c.Rext;
  a.info = c.info;
  CUtensorMap map{};
  a.bulk = xg_tensor_map(&map, NC, c.A, c.nA < c.n ? c.b : nullptr, std::is_same<S, double>::value ? QL_F64 : QL_F32,
                         c.m, c.nA, c.lda)
               ? 1
               : 0;
  a.mround = NC >= 16 ? 2 : 1;  // how the next pass's kernel of this class reads M
  count_launch();
  return launch_dependent(kern, (int)g, Sh::T, Sm::kBytes, c.stream, a, map) == cudaSuccess ? QL_OK : QL_ERR_CUDA;
}

template <typename S>
ql_status xgram_pass1(const GramCall& c, const GramWs& w) {
  if (c.n <= 4) return xgram_launch_one<4, S>(c, w);
  if (c.n <= 8) return xgram_launch_one<8, S>(c, w);
  if (c.n <= 16) return xgram_launch_one<16, S>(c, w);
  if (c.n <= 32) return xgram_launch_one<32, S>(c, w);
  return xgram_launch_one<64, S>(c, w);
}

}  // namespace ql
