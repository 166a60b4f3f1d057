// pbat_bs_template.h -- CUDA source of the bit-sliced enumeration kernels.
//
// The engine prepends a block of #defines and the graph-specific
// connectivity functions (bs_inv / bs_var, written by the planner in
// pbat_bs_plan.cu) and compiles the result with NVRTC for sm_103a.
//
// State layout: bit j of a thread's 32-bit word is the state whose BS_ELL
// lane arcs follow the bits of j; the BS_TB thread arcs follow the bits of
// the warp lane id; the BS_L walk arcs follow the walk index g; the BS_D
// prefix arcs are fixed per work item (one item per warp, from an atomic
// ticket: the equal division of Sec. 4.3).  The walk visits g in reflected
// Gray order over its upper BS_L - BS_IN bits and, for each such step, all
// 2^BS_IN settings of its lowest bits in an unrolled block whose walk words
// are compile-time constants that fold through the connectivity program.
//
// Per word the connectivity of its 32 states is c = bs_var(inv, walk words):
// bit j set iff the sink is reachable from the source in state j (the PLSA
// answer of Sec. 3.2).  R (Eq. 1) accumulates exactly: the lane mass of the
// connected bits comes from four byte tables (u64, scale 2^62, each entry
// paired with the bit counts of its lane-popcount classes so that one 16-byte
// load serves R and N_k), times the walk mass of g, into a 128-bit integer T
// per thread (scale 2^125); the thread-arc and prefix masses are applied once
// per item, in integer arithmetic (the FP64 rate of this part is 1/64 of its
// FP32 rate, so no per-item work uses FP64).
#pragma once

namespace pbat {

static const char* kBsTemplate = R"PBAT(
typedef unsigned int u32;
typedef unsigned long long u64;

#define BS_IN (BS_L >= BS_IN_BITS ? BS_IN_BITS : BS_L)
// launch bounds of the single-network kernels: with BS_MINB blocks per SM
// requested, the compiler keeps registers within 65536 / (BS_MINB * BS_NTHR)
#if defined(BS_MINB) && BS_MINB > 0
#define KERNEL_BOUNDS __launch_bounds__(BS_NTHR, BS_MINB)
#else
#define KERNEL_BOUNDS __launch_bounds__(BS_NTHR)
#endif
#define BS_OUT (BS_L - BS_IN)

struct dd { double hi, lo; };   // host-side double-double (only carried, never computed here)

struct u128 { u64 lo, hi; };
__device__ __forceinline__ void u128_add(u128& a, u64 blo, u64 bhi) {
  asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(a.lo), "+l"(a.hi) : "l"(blo), "l"(bhi));
}
__device__ __forceinline__ u128 u128_sub(u128 a, u128 b) {
  u128 r;
  asm("sub.cc.u64 %0, %2, %4;\n\tsubc.u64 %1, %3, %5;" : "=l"(r.lo), "=l"(r.hi) : "l"(a.lo), "l"(a.hi), "l"(b.lo), "l"(b.hi));
  return r;
}
// (a * b) >> 64 for a 64-bit a and a 128-bit b (the lowest 64 bits dropped)
__device__ __forceinline__ u128 mul64x128_shr64(u64 a, u64 blo, u64 bhi) {
  const u64 h0 = __umul64hi(a, blo);
  const u64 l1 = a * bhi;
  const u64 h1 = __umul64hi(a, bhi);
  u128 r;
  asm("add.cc.u64 %0, %2, %3;\n\taddc.u64 %1, %4, 0;" : "=l"(r.lo), "=l"(r.hi) : "l"(l1), "l"(h0), "l"(h1));
  return r;
}
__device__ __forceinline__ u128 shfl_xor_u128(u128 v, int m) {
  u128 r;
  r.lo = __shfl_xor_sync(0xffffffffu, v.lo, m);
  r.hi = __shfl_xor_sync(0xffffffffu, v.hi, m);
  return r;
}
// exact sum over the warp (every lane gets it)
#if defined(BS_GRAD) && BS_GRAD && !BS_ACC_REG
// the fused kernel with a large connectivity program: five rounds of 128-bit
// shuffles (the hardware reductions below measured 2% slower there)
__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const u128 w = shfl_xor_u128(v, o);
    u128_add(v, w.lo, w.hi);
  }
  return v;
}
#else
// the value in five chunks of at most 26 bits, whose 32-lane sums fit 31
// bits, one hardware warp reduction each, recombined in 128-bit arithmetic
// (GB300, against five rounds of 128-bit shuffles: 40-arc R kernel 87.7 ->
// 73.0 ms, 34-arc directed 490 -> 472 us)
__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
  const u32 c0 = (u32)(v.lo & 0x3ffffffull), c1 = (u32)((v.lo >> 26) & 0x3ffffffull);
  const u32 c2 = (u32)(((v.lo >> 52) | (v.hi << 12)) & 0x3ffffffull);
  const u32 c3 = (u32)((v.hi >> 14) & 0x3ffffffull), c4 = (u32)(v.hi >> 40);
  const u64 s0 = __reduce_add_sync(0xffffffffu, c0), s1 = __reduce_add_sync(0xffffffffu, c1);
  const u64 s2 = __reduce_add_sync(0xffffffffu, c2), s3 = __reduce_add_sync(0xffffffffu, c3);
  const u64 s4 = __reduce_add_sync(0xffffffffu, c4);
  u128 r = u128{s0, 0ull};
  u128_add(r, s1 << 26, 0ull);
  u128_add(r, s2 << 52, s2 >> 12);
  u128_add(r, 0ull, s3 << 14);
  u128_add(r, 0ull, s4 << 40);
  return r;
}
#endif

__device__ __forceinline__ u128 u128_shr(u128 v, int s) {
  if (s <= 0) return v;
  if (s >= 128) return u128{0ull, 0ull};
  if (s >= 64) return u128{v.hi >> (s - 64), 0ull};
  return u128{(v.lo >> s) | (v.hi << (64 - s)), v.hi >> s};
}

// Products of arc reliabilities (the prefix masses) as integer floating
// point: value m * 2^(-63 - e), m in [2^63, 2^64) or m = 0, e >= 0.  A
// product keeps 63 significant bits.
struct mx { u64 m; int e; int pad; };
__device__ __forceinline__ mx mx_mul(mx a, mx b) {
  u64 h = __umul64hi(a.m, b.m);
  int e = a.e + b.e - 1;
  if (!(h >> 63)) { h <<= 1; ++e; }
  return mx{h, e, 0};
}
// x times a 128-bit value v at scale 2^124 is mx_prod(x, v) * 2^(-123 - x.e)
// (truncated; below 2^124)
__device__ __forceinline__ u128 mx_prod(mx x, u128 v) { return mul64x128_shr64(x.m, v.lo, v.hi); }

// Floating 128-bit accumulator: value v * 2^(-123 - E) with v < 2^126, so a
// sum of items keeps about 125 significant bits relative to its own size,
// whatever the mass of the enumerated range.
struct facc { u128 v; int E; int pad; };
__device__ __forceinline__ void facc_add(facc& a, u128 P, int e) {
  if (!(P.lo | P.hi)) return;
  if (!(a.v.lo | a.v.hi)) { a.v = P; a.E = e; return; }
  if (e >= a.E) {
    const u128 q = u128_shr(P, e - a.E);
    u128_add(a.v, q.lo, q.hi);
  } else {
    a.v = u128_shr(a.v, a.E - e);
    a.E = e;
    u128_add(a.v, P.lo, P.hi);
  }
  if (a.v.hi >> 62) { a.v = u128_shr(a.v, 1); a.E -= 1; }
}

// add v * 2^(s - 250) to a 256-bit fixed-point number held as 32-bit chunks
// in eight 64-bit limbs (the upper halves absorb the carries); v < 2^127 and
// s <= 129 keep it below 2^256
__device__ __forceinline__ void bs_limb_add(u64* limbs, u128 v, int s) {
  if (s < 0) {
    v = u128_shr(v, -s);
    s = 0;
  }
  if (!(v.lo | v.hi)) return;
  const int c0 = s >> 5, r = s & 31;
  const u64 q0 = v.lo << r;
  const u64 q1 = r ? ((v.hi << r) | (v.lo >> (64 - r))) : v.hi;
  const u64 q2 = r ? (v.hi >> (64 - r)) : 0ull;
  const u64 c[5] = {q0 & 0xffffffffull, q0 >> 32, q1 & 0xffffffffull, q1 >> 32, q2};
#pragma unroll
  for (int i = 0; i < 5; ++i)
    if (c[i] && c0 + i < 8) atomicAdd(&limbs[c0 + i], c[i]);
}

// N_k counts of one word, packed by lane-popcount class cl = 0..5 into
// fields of 8, 11, 12, 12, 11 and 8 bits: wide enough for one item's sum
// over 2^L words with L <= 10 (at most C(10,5) * C(5,cl) per field).
#define BS_NK_SHIFTS {0, 8, 19, 31, 43, 54}
#define BS_NK_WIDTHS {8, 11, 12, 12, 11, 8}

struct BsParams {
  u64 task_lo, n_tasks, budget_ns;
  int prune, nlev;       // prefix-mass table levels
  int ex_shift;          // log2 of the excluded-arc table's row length
  // merged runs: levels of the prefix arcs above a block, the mass scale of
  // the classes (see bs_merge) and log2 of their table's slots
  int nlev_hi, mass_exp, slots_log2;
  int hi_bits[10], hi_off[10];
  int lev_bits[10];      // prefix bits per level (low level first)
  int lev_off[10];       // first entry of each level in the prefix table
  u64 thw[32];           // thread-pattern masses, fixed point 2^63
  u64 binom[64];
};
struct facc;
struct BsWork {
  u64* counter; u32* status; u64* stats;
  dd* part_acc; u64* part_n; dd* out_acc; u64* out_n;
  u64* out_limbs;   // [n_acc][8]: 256-bit fixed point at scale 2^250, 32 bits per limb
  // merged runs: the classes in the order they were met (their slots), how
  // many there are, and the walking launch's ticket
  u32* list;
  u64* list_n;
  u64* counter2;
  u64* start;   // and when it began (bs_run_start)
  // per slot: the signature (0: unused), the summed mass of the class's items
  // in two chunks, their number by popcount (BS_HIST each), one of them, and
  // the sum S of that one
  u64 *key, *cmass;
  u32* hist;
  u64* rep;
  ulonglong2* csum;
  // per block of items and lane: items connected throughout and items left to
  // walk (a bit each), and the latter's slots ([block][bit][lane])
  uint2* cmask;
  u32* cls;
};

// One-launch runs (phase 0) take items by the atomic ticket over [0,
// n_tasks).  The walking launch of a merged run (phase 2) takes classes from
// the list: a warp's first by its index, counted over the blocks first, so
// that few classes are spread over the SMs and blocks without any return at
// once; only a list longer than the grid goes on by ticket (with a ticket for
// every class, the grid's warps queued on one counter: 27-arc R 38 -> 28 us).
__device__ __forceinline__ u64 bs_next_class(const BsWork& W, u64 n_list, u64 n_warps, int lane) {
  u64 i = ~0ull;
  if (n_list > n_warps) {
    if (lane == 0) i = n_warps + atomicAdd(W.counter2, 1ull);
    i = __shfl_sync(0xffffffffu, i, 0);
  }
  return i;
}
// Programmatic dependent launch: the launches of a merged run start while
// the one before drains, and wait here for its results.
__device__ __forceinline__ void bs_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void bs_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ u64 bs_timer() {
  u64 t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t;
}
__device__ __forceinline__ bool bs_late(u64 budget_ns, u64 t_start, u32* status) {
  const u64 now = bs_timer();
  if (now <= t_start || now - t_start <= budget_ns) return false;
  atomicOr(status, 1u);
  return true;
}
// The launches of a merged run all count its time limit from when the first
// warp of the first one asked, kept beside the status.  (Another SM's clock may
// have been read a little later than this one's.)
__device__ __forceinline__ u64 bs_run_start(u64* start) {
  u64 first = *(volatile u64*)start;
  if (!first) {
    const u64 now = bs_timer();
    first = atomicCAS(start, 0ull, now);
    if (!first) first = now;
  }
  return first;
}
__device__ __forceinline__ bool bs_run_late(u64 budget_ns, u64* start, u32* status) {
  return bs_late(budget_ns, bs_run_start(start), status);
}
// Whether the time is up, the same answer in every lane of a warp or every
// thread of a block: one lane reads the clock.  The loops that ask go on with
// collectives of the whole warp, and the lanes come here from code where they
// part, so each lane reading for itself could leave some of them waiting for
// the others.  Out of line, and called under a limit only: inlined, it made
// the compiler join the parted lanes of bs_merge_body's loop over the classes
// later (24 nodes, 40 arcs, L = 6: 44.5 -> 60.3 M warp instructions, 103 -> 129 us).
__device__ __noinline__ bool bs_time_up(u64 budget_ns, u64* start, u32* status, int lane) {
  __syncwarp();
  int up = 0;
  if (lane == 0) up = bs_run_late(budget_ns, start, status);
  return __shfl_sync(0xffffffffu, up, 0) != 0;
}
__device__ __noinline__ bool bs_block_time_up(u64 budget_ns, u64* start, u32* status) {
  int up = 0;
  if (threadIdx.x == 0) up = bs_run_late(budget_ns, start, status);
  return __syncthreads_or(up) != 0;
}
// Whether the run was given up, out of time or of class slots (the host then
// discards it), the same answer in every thread of a block or of a warp: one
// reads the word, which other blocks of the same launch may be setting.
__device__ __forceinline__ bool bs_block_given_up(const u32* status) {
  return __syncthreads_or(threadIdx.x == 0 && *(volatile const u32*)status != 0u) != 0;
}
__device__ __forceinline__ bool bs_warp_given_up(const u32* status, int lane) {
  const u32 s = lane == 0 ? *(volatile const u32*)status : 0u;
  return __shfl_sync(0xffffffffu, s, 0) != 0u;
}

// Mass of the prefix arcs of `prefix`: product over table levels.
__device__ __forceinline__ mx bs_level_mass(int nlev, const int* bits, const int* off,
                                            const mx* __restrict__ ptab, u64 prefix) {
  mx w = mx{1ull << 63, 0, 0};
  int sh = 0;
  for (int l = 0; l < nlev; ++l) {
    const u64 v = (prefix >> sh) & ((1ull << bits[l]) - 1ull);
    const mx t = ptab[off[l] + v];
    w = l ? mx_mul(w, t) : t;
    sh += bits[l];
  }
  return w;
}
__device__ __forceinline__ mx bs_prefix_mass(const BsParams& P, const mx* __restrict__ ptab, u64 prefix) {
  return bs_level_mass(P.nlev, P.lev_bits, P.lev_off, ptab, prefix);
}
// Per-lane constants of the 32x32 bit transpose below: byte selectors of the
// 16- and 8-bit rounds, rotate amounts and keep-masks of the 4-, 2- and
// 1-bit rounds.
struct BsTr { u32 sel16, sel8, rot4, rot2, rot1, keep4, keep2, keep1; };
__device__ __forceinline__ BsTr bs_tr_init(int lane) {
  BsTr t;
  t.sel16 = (lane & 16) ? 0x3276u : 0x5410u;
  t.sel8 = (lane & 8) ? 0x3715u : 0x6240u;
  t.rot4 = (lane & 4) ? 28u : 4u;
  t.rot2 = (lane & 2) ? 30u : 2u;
  t.rot1 = (lane & 1) ? 31u : 1u;
  t.keep4 = (lane & 4) ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
  t.keep2 = (lane & 2) ? 0xCCCCCCCCu : 0x33333333u;
  t.keep1 = (lane & 1) ? 0xAAAAAAAAu : 0x55555555u;
  return t;
}
// Round with distance sh: lanes with bit sh clear keep the low half of
// every 2sh-bit group and take the partner's low halves into their high
// halves; lanes with the bit set keep the high halves and take the
// partner's high halves into their low halves.  Byte-sized rounds are one
// byte permute; smaller ones a rotate and a bit select.
__device__ __forceinline__ u32 bs_transpose32(u32 x, const BsTr& t) {
  u32 y = __shfl_xor_sync(0xffffffffu, x, 16);
  x = __byte_perm(x, y, t.sel16);
  y = __shfl_xor_sync(0xffffffffu, x, 8);
  x = __byte_perm(x, y, t.sel8);
  y = __shfl_xor_sync(0xffffffffu, x, 4);
  x = (x & t.keep4) | (__funnelshift_l(y, y, t.rot4) & ~t.keep4);
  y = __shfl_xor_sync(0xffffffffu, x, 2);
  x = (x & t.keep2) | (__funnelshift_l(y, y, t.rot2) & ~t.keep2);
  y = __shfl_xor_sync(0xffffffffu, x, 1);
  x = (x & t.keep1) | (__funnelshift_l(y, y, t.rot1) & ~t.keep1);
  return x;
}

__device__ __forceinline__ u32 bs_pattern(int i) {
  return i == 0 ? 0xAAAAAAAAu : i == 1 ? 0xCCCCCCCCu : i == 2 ? 0xF0F0F0F0u : i == 3 ? 0xFF00FF00u : 0xFFFF0000u;
}
// (a * b) >> 128 (the product of the low halves dropped: at most two units low)
__device__ __forceinline__ u128 mulhi128(u128 a, u128 b) {
  u128 r = u128{a.hi * b.hi, __umul64hi(a.hi, b.hi)};
  u128_add(r, __umul64hi(a.hi, b.lo), 0ull);
  u128_add(r, __umul64hi(a.lo, b.hi), 0ull);
  return r;
}
// The mass of the 32 patterns set in v, from eight nibble tables t of 16
// subset sums (scale 2^127), times the mass f (scale 2^127): scale 2^126.
__device__ __forceinline__ u128 bs_subset_mass(u32 v, const ulonglong2* t, u128 f) {
  u128 s = u128{0ull, 0ull};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const ulonglong2 x = t[16 * i + ((v >> (4 * i)) & 15u)];
    u128_add(s, x.x, x.y);
  }
  return mulhi128(s, f);
}
// Every 2^split_log2-th bit, from bit `part` on: one warp's share of a
// block's words when 2^split_log2 warps work on it.
__device__ __forceinline__ u32 bs_part_mask(int split_log2, u32 part) {
  return (split_log2 == 0 ? 0xffffffffu : split_log2 == 1 ? 0x55555555u : split_log2 == 2 ? 0x11111111u
          : split_log2 == 3 ? 0x01010101u : split_log2 == 4 ? 0x00010001u : 1u) << part;
}
// The set bits of v by the popcount of their position, a byte each.
__device__ __forceinline__ u64 bs_popcount_bytes(u32 v) {
  return (u64)(__popc(v & 0x00000001u) | (__popc(v & 0x00010116u) << 8) | (__popc(v & 0x01161668u) << 16) |
               (__popc(v & 0x16686880u) << 24)) |
         ((u64)(__popc(v & 0x68808000u) | (__popc(v & 0x80000000u) << 8)) << 32);
}
// Counts of a block's items in `full` by popcount inside the block, lane k
// ending with popcount k's.  Every lane packs its own into bytes (at most
// C(10, 5) = 252 each over the warp) and three warp reductions add them.
__device__ __forceinline__ u32 bs_block_counts(u32 full, int lane) {
  const u64 v = bs_popcount_bytes(full);
  const int sh = 8 * __popc(lane);
  const u64 lo = v << sh, hi = sh ? v >> (64 - sh) : 0ull;
  const u32 r0 = __reduce_add_sync(0xffffffffu, (u32)lo), r1 = __reduce_add_sync(0xffffffffu, (u32)(lo >> 32));
  const u32 r2 = __reduce_add_sync(0xffffffffu, (u32)hi);
  const u32 r = lane < 4 ? r0 : lane < 8 ? r1 : r2;
  return (r >> (8 * (lane & 3))) & 255u;
}
// The class of signature `key` (never 0): its slot, by linear probing from
// its hash; claimed by compare-and-swap when new (`fresh`).  A table of
// 2^nsig slots or more is indexed by the signature itself.  ~0: no free slot
// within reach.
__device__ __forceinline__ u32 bs_class(u64* table, int slots_log2, int nsig, u64 key, bool& fresh) {
  const u32 mask = (1u << slots_log2) - 1u;
  u32 slot = (u32)key & mask;
  if (nsig > slots_log2) {
    u64 h = key * 0x9E3779B97F4A7C15ull;   // the finaliser of splitmix64
    h = (h ^ (h >> 30)) * 0xBF58476D1CE4E5B9ull;
    slot = (u32)((h ^ (h >> 27)) >> 20) & mask;
  }
  fresh = false;
  for (int probe = 0; probe < 256; ++probe) {
    u64 k = *(volatile u64*)&table[slot];
    if (!k) {
      k = atomicCAS(&table[slot], 0ull, key);
      if (!k) { fresh = true; return slot; }
    }
    if (k == key) return slot;
    slot = (slot + 1u) & mask;
  }
  return ~0u;
}

// A mass m (integer floating point hi times the 128-bit v, scale 2^124) at
// scale 2^(98 + mass_exp), where all the items' masses add up to at most
// 2^98, added to a class's two chunks -- the lower of BS_CLASS_SHIFT bits --
// each by itself; and the mass back from its chunks.
#define BS_CLASS_SHIFT 38
__device__ __forceinline__ void bs_add_mass(u64* chunks, mx hi, u128 v, int mass_exp) {
  const u128 F = u128_shr(mx_prod(hi, v), 25 + hi.e - mass_exp);
  const u64 lo = F.lo & ((1ull << BS_CLASS_SHIFT) - 1ull);
  const u64 up = (F.lo >> BS_CLASS_SHIFT) | (F.hi << (64 - BS_CLASS_SHIFT));
  if (lo) atomicAdd(&chunks[0], lo);
  if (up) atomicAdd(&chunks[1], up);
}
__device__ __forceinline__ mx bs_class_mass(const u64* chunks, int mass_exp) {
  u128 t = u128{chunks[0], 0ull};
  const u64 up = chunks[1];
  u128_add(t, up << BS_CLASS_SHIFT, up >> (64 - BS_CLASS_SHIFT));
  if (!(t.lo | t.hi)) return mx{0ull, 0, 0};
  const int lz = t.hi ? __clzll((long long)t.hi) : 64 + __clzll((long long)t.lo);
  const u64 m = lz >= 64 ? t.lo << (lz - 64) : (lz ? (t.hi << lz) | (t.lo >> (64 - lz)) : t.hi);
  return mx{m, lz - 29 + mass_exp, 0};   // 128 - lz bits at scale 2^(98 + mass_exp)
}
// Adds the popcounts of the items in `same` of a lane to a class's counters
// (h, by popcount), two 32-bit counters to an addition; pc: the popcount of
// their common arcs.
__device__ __forceinline__ void bs_add_counts(u32* h, u32 same, int pc) {
  u64* p = (u64*)h + (pc >> 1);
  const u64 n = bs_popcount_bytes(same) << (8 * (pc & 1));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const u64 two = ((n >> (16 * i)) & 255ull) | ((n >> (16 * i + 8)) & 255ull) << 32;
    if (two) atomicAdd(&p[i], two);
  }
}
// |a - b|; neg: a < b (classes' sums round apart by up to 2^-61, so a pair
// whose true difference is zero may come out below it)
__device__ __forceinline__ u128 bs_absdiff(u128 a, u128 b, bool& neg) {
  neg = a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
  return neg ? u128_sub(b, a) : u128_sub(a, b);
}
// one fold: adds w (V1 - V0) to G, returns V0 + p (V1 - V0)
__device__ __forceinline__ u128 bs_fold2(u128 V0, u128 V1, u64 p, u64 w, u128& G) {
  bool neg;
  const u128 d = bs_absdiff(V1, V0, neg);
  if (!neg) {
    const u128 g = mul64x128_shr64(w, d.lo, d.hi);   // scale 2^123
    u128_add(G, g.lo, g.hi);
  }
  u128 x = mul64x128_shr64(p, d.lo, d.hi);
  x = u128{x.lo << 1, (x.hi << 1) | (x.lo >> 63)};
  if (neg) return u128_sub(V0, x);
  u128_add(V0, x.lo, x.hi);
  return V0;
}
// A fold block's 32 items per lane, folded over the five low arcs (see
// bs_kernel_grad_p3): the items 8 q to 8 q + 7 over the lowest three, then
// the four results over the other two.  item(j): item j's conditional
// reliability (scale 2^124); p, w: the low arcs' p and the masses above each,
// as in BsFoldParams; G: the sums per arc.
template <class Item>
__device__ __forceinline__ u128 bs_fold_group(const u64* p, const u64* w, int q, u128 (&G)[5], Item item) {
  u128 V[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) V[i] = item(8 * q + i);
#pragma unroll
  for (int i = 0; i < 4; ++i) V[i] = bs_fold2(V[2 * i], V[2 * i + 1], p[0], w[4 * q + i], G[0]);
#pragma unroll
  for (int i = 0; i < 2; ++i) V[i] = bs_fold2(V[2 * i], V[2 * i + 1], p[1], w[16 + 2 * q + i], G[1]);
  return bs_fold2(V[0], V[1], p[2], w[24 + q], G[2]);
}
__device__ __forceinline__ u128 bs_fold_groups(const u64* p, const u64* w, u128 (&V)[4], u128 (&G)[5]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) V[i] = bs_fold2(V[2 * i], V[2 * i + 1], p[3], w[28 + i], G[3]);
  return bs_fold2(V[0], V[1], p[4], w[30], G[4]);
}
template <class Item>
__device__ __forceinline__ u128 bs_fold_low(const u64* p, const u64* w, u128 (&G)[5], Item item) {
  u128 V[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) V[q] = bs_fold_group(p, w, q, G, item);
  return bs_fold_groups(p, w, V, G);
}
// Sum over the lanes of a low arc's G by the mid patterns' masses (2^124).
__device__ __forceinline__ u128 bs_fold_sum(u128 G, u64 m_mid) {
  const u128 g = warp_sum_u128(mul64x128_shr64(m_mid, G.lo, G.hi));   // 2^122
  return u128{g.lo << 2, (g.hi << 2) | (g.lo >> 62)};
}
// The mid arcs over the lanes, and the block's sums per arc (scale 2^124):
// lane l ends with low arc l's (from FIRST on), lane `low` + l with mid arc
// l's, in X; every lane with the block's V.
template <int FIRST>
__device__ __forceinline__ u128 bs_fold_mid(u128 V, const u128 (&G)[5], int low, int mid, const u64* p, const u64* w,
                                            u64 m_mid, int lane, u128& X) {
  X = u128{0ull, 0ull};
#pragma unroll
  for (int i = FIRST; i < 5; ++i) {
    if (i >= low) break;
    const u128 g = bs_fold_sum(G[i], m_mid);
    if (lane == i) X = g;
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    if (i >= mid) break;
    const u128 o = shfl_xor_u128(V, 1 << i);
    const bool one = (lane >> i) & 1;
    u128 g = u128{0ull, 0ull};
    const int at = (i == 0 ? 0 : i == 1 ? 16 : i == 2 ? 24 : i == 3 ? 28 : 30) + (lane >> (i + 1));
    V = bs_fold2(one ? o : V, one ? V : o, p[i], w[at], g);
    if (lane & ((1 << (i + 1)) - 1)) g = u128{0ull, 0ull};   // each pair once
    g = warp_sum_u128(g);
    g = u128{g.lo << 1, (g.hi << 1) | (g.lo >> 63)};
    if (lane == low + i) X = g;
  }
  V.lo = __shfl_sync(0xffffffffu, V.lo, 0);
  V.hi = __shfl_sync(0xffffffffu, V.hi, 0);
  return V;
}

//@@GENERATED@@
// connectivity of one uniform state (every word 0 or ~0): the prune test
__device__ __forceinline__ u32 bs_uniform(const u32* a) {
  u32 e[BS_NCORE > 0 ? BS_NCORE : 1];
  bs_inv(a, e);
  u32 w[BS_L > 0 ? BS_L : 1];
#pragma unroll
  for (int b = 0; b < BS_L; ++b) w[b] = a[BS_WALK0 + b];
  return bs_var(e, w);
}

__device__ __forceinline__ void bs_init_arcs(u32* a, int lane) {
#pragma unroll
  for (int i = 0; i < BS_ELL; ++i)
    a[i] = i == 0 ? 0xAAAAAAAAu : i == 1 ? 0xCCCCCCCCu : i == 2 ? 0xF0F0F0F0u : i == 3 ? 0xFF00FF00u : 0xFFFF0000u;
#pragma unroll
  for (int i = 0; i < BS_TB; ++i) a[BS_ELL + i] = 0u - (u32)((lane >> i) & 1);
#pragma unroll
  for (int b = 0; b < BS_L; ++b) a[BS_WALK0 + b] = 0u;
}

// 0: walk the item, 1: every state disconnected, 2: every state connected.
// One bit-sliced evaluation answers both extremes: bit 0 has every arc below
// the prefix working, bit 1 every such arc failed (the prefix arcs are the
// same in every bit).
__device__ __forceinline__ int bs_prune(const u32* a) {
  u32 u[BS_M];
#pragma unroll
  for (int k = 0; k < BS_M; ++k) u[k] = k < BS_TOP ? 1u : a[k];
  const u32 ext = bs_uniform(u);
  if (!(ext & 1u)) return 1;
  return (ext & 2u) ? 2 : 0;
}

// An item's counts by popcount below the prefix, into the warp's own rel
// (BS_TOP + 1, cleared here): 32-bit additions in shared memory, which are
// one instruction, where 64-bit ones are a compare-and-swap loop that the
// threads of one popcount run in turn (an item has at most C(20, 10) =
// 184,756 states of one popcount).  Then the warp adds them to the block's
// (bs_item_counts) or a class's (bs_class_counts), a lane per popcount.
__device__ __forceinline__ void bs_flush_bins(u64* bins, u32* rel, int lane) {
  constexpr int sh[6] = BS_NK_SHIFTS, wd[6] = BS_NK_WIDTHS;
  if (lane <= BS_TOP) rel[lane] = 0u;
  __syncwarp();
  if (lane < (1 << BS_TB)) {
    u32* mine = rel + __popc(lane);
#pragma unroll 1
    for (int r = 0; r <= BS_L; ++r) {
      const u64 n = bins[r * BS_NTHR];
#pragma unroll
      for (int cl = 0; cl < 6; ++cl) {
        const u32 c = (u32)(n >> sh[cl]) & ((1u << wd[cl]) - 1u);
        if (c) atomicAdd(&mine[r + cl], c);
      }
    }
  }
  __syncwarp();
}
__device__ __forceinline__ void bs_item_counts(const u32* rel, u64* s_nbins, int pc_pre, int lane) {
  if (lane <= BS_TOP && rel[lane]) atomicAdd(&s_nbins[pc_pre + lane], (u64)rel[lane]);
}

// End of a block: entry i combines the warps' floating accumulators
// s_acc[w * stride + i] in integer arithmetic and adds the sum to the result
// with integer atomics (every sum is non-negative, and integer addition is
// exact, so the order of the blocks does not matter); then the block's N_k
// counts.  The host converts the result once.
__device__ __forceinline__ void bs_add_out(u64* limbs, const facc* s_acc, int stride, int n_acc, int nthr) {
  for (int i = threadIdx.x; i < n_acc; i += nthr) {
    facc t = s_acc[i];
    for (int w = 1; w < nthr / 32; ++w) facc_add(t, s_acc[w * stride + i].v, s_acc[w * stride + i].E);
    bs_limb_add(limbs + 8 * i, t.v, 127 - t.E);   // v * 2^(-123 - E) at scale 2^250
  }
}
__device__ __forceinline__ void bs_write_out(const BsWork& W, const facc* s_acc, int stride, int n_acc,
                                             const u64* s_nbins, int nthr) {
  bs_add_out(W.out_limbs, s_acc, stride, n_acc, nthr);
  for (int i = threadIdx.x; i <= BS_M; i += nthr)
    if (s_nbins[i]) atomicAdd(&W.out_n[i], s_nbins[i]);
}

// ---------------------------------------------------------------------------
// Merged runs.  Most items that the prune leaves share what their prefix
// leaves of the network with many others (bs_sig), so the run goes in three
// launches:
//   bs_merge  prunes the items, 32 x 32 of them at a time, sums those that
//             are connected throughout, and gives each one left to the class
//             of its signature: its mass, its popcount;
//   bs_walk   walks one item of every class for all of them;
//   bs_fold   (fused kernel) the prefix arcs' gradient from the items' sums.
// Against walking every item left (GB300, whole passes through the API): a
// 24-node, 40-arc network (2^40 states) fused 49.3 -> 0.30 ms, R 20.2 -> 0.17
// ms; a 20-node, 34-arc directed network 0.38 -> 0.072 and 0.65 -> 0.086 ms;
// 11 nodes, 31 arcs, fused 0.39 -> 0.13 ms.  The large runs are bound by
// instruction issue (bs_merge and bs_fold work per 32 items, bs_walk per
// class), the small ones by the latency of their two or three launches.
// ---------------------------------------------------------------------------
#if BS_MERGE
#define BS_BLK (BS_LOW + BS_MID)   // prefix arcs inside a merge block
#define BS_HI (BS_D - BS_BLK)      // prefix arcs above it
#define BS_MERGE_NTHR 128
#define BS_HIST ((BS_D + 2) & ~1)  // counters by popcount of a class, an even number
__device__ __forceinline__ void bs_merge_body(const BsParams& P, const mx* __restrict__ ptab,
                                              const ulonglong2* __restrict__ mtab, int split_log2, const BsWork& W) {
  __shared__ ulonglong2 s_nib[128];   // subset sums of the low prefix pattern masses
  __shared__ facc s_acc[BS_MERGE_NTHR / 32];
  __shared__ u64 s_ci[BS_D + 1];      // items connected throughout, by popcount
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 128; i += BS_MERGE_NTHR) s_nib[i] = mtab[i];
  for (int i = tid; i <= BS_D; i += BS_MERGE_NTHR) s_ci[i] = 0ull;
  bs_let_next_start();
  __syncthreads();
  const u128 m_mid = u128{mtab[128 + lane].x, mtab[128 + lane].y};
  facc accR = facc{u128{0ull, 0ull}, 0, 0};
  // a block's items left to walk are shared by 2^split_log2 warps (each takes
  // every so manyeth bit of the words), so that few blocks still fill the GPU
  const u64 nwarps = (u64)gridDim.x * (BS_MERGE_NTHR / 32);
  const u64 nblk = P.n_tasks >> BS_BLK, blk0 = P.task_lo >> BS_BLK;
  const u32 valid = lane < (1 << BS_MID) ? (BS_LOW >= 5 ? 0xffffffffu : (1u << (1 << BS_LOW)) - 1u) : 0u;
  for (u64 t = (u64)blockIdx.x * (BS_MERGE_NTHR / 32) + warp; t < nblk << split_log2; t += nwarps) {
    const u64 b = t >> split_log2;
    const u32 part = (u32)t & ((1u << split_log2) - 1u);
    if (P.budget_ns && bs_time_up(P.budget_ns, W.start, W.status, lane)) break;
    const u64 hi = blk0 + b;
    u32 a[BS_M], z[BS_NSIG > 0 ? BS_NSIG : 1], dn, up;
#pragma unroll
    for (int j = 0; j < BS_D; ++j)
      a[BS_TOP + j] = j < BS_LOW ? bs_pattern(j) : j < BS_BLK ? 0u - (u32)((lane >> (j - BS_LOW)) & 1)
                                                              : 0u - (u32)((hi >> (j - BS_BLK)) & 1ull);
    bs_sig(a, z, dn, up);
    const u32 full = dn & valid;
    u32 left = up & valid & ~full;
    const int pc_hi = __popcll((long long)hi);
    if (part == 0) {
      if (BS_GRAD) W.cmask[b * 32 + lane] = make_uint2(full, left);
      if (__any_sync(0xffffffffu, full)) {
        const u32 n = bs_block_counts(full, lane);
        if (lane <= BS_BLK && n) atomicAdd(&s_ci[pc_hi + lane], (u64)n);
        const u128 S = warp_sum_u128(u128_shr(bs_subset_mass(full, s_nib, m_mid), 2));
        const mx w = bs_level_mass(P.nlev_hi, P.hi_bits, P.hi_off, ptab, hi);
        facc_add(accR, mx_prod(w, S), w.e);
      }
    }
    if (!__any_sync(0xffffffffu, left)) continue;
    // every 2^split_log2-th bit
    left &= bs_part_mask(split_log2, part);
    const mx whi = bs_level_mass(P.nlev_hi, P.hi_bits, P.hi_off, ptab, hi);
    while (left) {
      // one of the lane's items, and all of them with its signature
      const int j = __ffs(left) - 1;
      u32 k0 = 0u, k1 = 0u, same = left;
#pragma unroll
      for (int i = 0; i < BS_NSIG; ++i) {
        const u32 top = z[i] << (31 - j);   // item j's bit on top
        if (i < 32) k0 = __funnelshift_l(top, k0, 1); else k1 = __funnelshift_l(top, k1, 1);
        same &= ~(z[i] ^ (u32)((int)top >> 31));
      }
      left &= ~same;
      const u64 key = ((u64)k1 << 32) | k0 | 1ull << 63;
      bool fresh;
      const u32 slot = bs_class(W.key, P.slots_log2, BS_NSIG, key, fresh);
      if (slot == ~0u) { atomicOr(W.status, 2u); continue; }   // the host runs the items one by one instead
      if (fresh) {
        W.rep[slot] = (hi << BS_BLK) | (u64)(lane << BS_LOW) | (u64)j;
        W.list[atomicAdd(W.list_n, 1ull)] = slot;
      }
      bs_add_mass(W.cmass + 2 * (size_t)slot, whi, u128_shr(bs_subset_mass(same, s_nib, m_mid), 2), P.mass_exp);
      bs_add_counts(W.hist + (size_t)slot * BS_HIST, same, pc_hi + __popc(lane));
      if (BS_GRAD)
        for (u32 s = same; s; s &= s - 1u) W.cls[(b << BS_BLK) + (u64)(((__ffs(s) - 1) << BS_MID) + lane)] = slot;
    }
  }
  if (lane == 0) s_acc[warp] = accR;
  __syncthreads();
  if (tid == 0) {
    facc r = s_acc[0];
    for (int w = 1; w < BS_MERGE_NTHR / 32; ++w) facc_add(r, s_acc[w].v, s_acc[w].E);
    bs_limb_add(W.out_limbs, r.v, 127 - r.E);
  }
  // an item connected throughout stands for C(arcs below, j) states with j
  // more working arcs
  for (int i = tid; i <= BS_M; i += BS_MERGE_NTHR) {
    u64 n = 0;
    for (int j = 0; j <= BS_TOP && j <= i; ++j)
      if (i - j <= BS_D) n += s_ci[i - j] * P.binom[j];
    if (n) atomicAdd(&W.out_n[i], n);
  }
}
// N_k of a class: its representative's states by popcount below the prefix
// (rel, BS_TOP + 1 of them) for every popcount that its prefixes have.
__device__ __forceinline__ void bs_class_counts(const BsWork& W, u64 slot, int lane, const u32* rel, u64* s_nbins) {
  const u64 r = lane <= BS_TOP ? rel[lane] : 0u;
  for (int p0 = 0; p0 <= BS_D; p0 += 32) {
    const u32 h = p0 + lane <= BS_D ? W.hist[(size_t)slot * BS_HIST + p0 + lane] : 0u;
    u32 some = __ballot_sync(0xffffffffu, h != 0u);
    while (some) {
      const int q = __ffs(some) - 1;
      some &= some - 1u;
      const u64 n = (u64)__shfl_sync(0xffffffffu, h, q) * r;
      if (n) atomicAdd(&s_nbins[p0 + q + lane], n);
    }
  }
  __syncwarp();
}
#endif

// ---------------------------------------------------------------------------
// R + N_k
// ---------------------------------------------------------------------------
#if !BS_GRAD
// PHASE 0: a one-launch run; 2: the walking launch of a merged run.  One entry
// point per phase, so that a one-launch kernel carries none of the other's
// state in its registers.
template <int PHASE>
__device__ __forceinline__ void bs_kernel_body(const BsParams& P, const u64* __restrict__ lane_tab,
                                               const u64* __restrict__ wmid_tab,
                                               const mx* __restrict__ ptab, const BsWork& W) {
  extern __shared__ __align__(16) unsigned char smem[];
  ulonglong2* s_lt = (ulonglong2*)smem;                     // [4][256] {lane mass 2^62, packed counts}
  u64* s_wmid = (u64*)(s_lt + 4 * 256);                     // [2^L], scale 2^63
  u64* s_bins = s_wmid + (1 << BS_L);                       // [L + 1][NTHR]
  facc* s_acc = (facc*)(s_bins + (BS_L + 1) * BS_NTHR);     // [warps]: each warp's R
  u64* s_nbins = (u64*)(s_acc + BS_NTHR / 32);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 4 * 256; i += BS_NTHR) s_lt[i] = ((const ulonglong2*)lane_tab)[i];
  for (int i = tid; i < (1 << BS_L); i += BS_NTHR) s_wmid[i] = wmid_tab[i];
  for (int i = tid; i <= BS_M; i += BS_NTHR) s_nbins[i] = 0ull;
  u64 n_list = 0, next = 0;
  if constexpr (PHASE == 2) {
    bs_wait_previous();
    n_list = *W.list_n;
    next = (u64)warp * gridDim.x + blockIdx.x;
    if (blockIdx.x >= n_list) return;   // no class
  }
  if (PHASE != 2) __syncthreads();
  else if (bs_block_given_up(W.status)) return;
  u64* bins = s_bins + tid;
  const bool thr_on = lane < (1 << BS_TB);
  const u64 thw = thr_on ? P.thw[lane] : 0ull;
  const u64 t_start = bs_timer();
  u64 n_walk = 0, n_full = 0, n_dead = 0;
  facc accR = facc{u128{0ull, 0ull}, 0, 0};   // this warp's R (the same in every lane)
  u32 a[BS_M];
  bs_init_arcs(a, lane);
  constexpr int phase = PHASE;
  u32* rel = (u32*)(s_nbins + BS_M + 1) + warp * (BS_TOP + 1);   // an item's counts below the prefix

  for (;;) {
    u64 task = 0;
    if constexpr (phase == 2) {
      task = next < n_list ? (u64)W.list[next] : ~0ull;
      next = bs_next_class(W, n_list, (u64)gridDim.x * (BS_NTHR / 32), lane);
    }
    if (lane == 0) {
      if constexpr (phase == 0) task = atomicAdd(W.counter, 1ull);
      if (P.budget_ns && (phase == 2 ? bs_run_late(P.budget_ns, W.start, W.status)
                                     : bs_late(P.budget_ns, t_start, W.status))) task = ~0ull;
    }
    task = __shfl_sync(0xffffffffu, task, 0);
    u64 prefix;
    if constexpr (phase == 2) {   // a class, by its slot
      if (task == ~0ull) break;
#if BS_MERGE
      prefix = W.rep[task];
#endif
    } else {
      if (task >= P.n_tasks) break;
      prefix = P.task_lo + task;
    }
#pragma unroll
    for (int j = 0; j < BS_D; ++j) a[BS_TOP + j] = 0u - (u32)((prefix >> j) & 1ull);
    const int pc_pre = __popcll((long long)prefix);
    if (P.prune && phase == 0) {
      const int pr = bs_prune(a);
      if (pr == 1) { ++n_dead; continue; }
      if (pr == 2) {
        ++n_full;
        for (int j = lane; j <= BS_TOP; j += 32) atomicAdd(&s_nbins[pc_pre + j], P.binom[j]);
        const mx w = bs_prefix_mass(P, ptab, prefix);
        facc_add(accR, mx_prod(w, u128{0ull, 1ull << 60}), w.e);
        continue;
      }
    }
    ++n_walk;
    u32 e[BS_NCORE > 0 ? BS_NCORE : 1];
    bs_inv(a, e);
#pragma unroll
    for (int r = 0; r <= BS_L; ++r) bins[r * BS_NTHR] = 0ull;
    u128 T = u128{0ull, 0ull};
    u32 gout = 0;
    int pco = 0;
#pragma unroll 1
    for (u32 s = 0; s < (1u << BS_OUT); ++s) {
      if (s) {
        const int b = __ffs(s) - 1;
        gout ^= 1u << b;
        pco += ((gout >> b) & 1u) ? 1 : -1;
      }
      u32 w[BS_L > 0 ? BS_L : 1];
#pragma unroll
      for (int b = 0; b < BS_OUT; ++b) w[BS_IN + b] = 0u - ((gout >> b) & 1u);
#pragma unroll
      for (int r = 0; r < (1 << BS_IN); ++r) {
#pragma unroll
        for (int b = 0; b < BS_IN; ++b) w[b] = ((r >> b) & 1) ? ~0u : 0u;
        const u32 c = bs_var(e, w) & BS_LANE_MASK;
        // one warp vote, as in the fused kernel: when some word of the warp
        // is partly connected every word reads its lane-table entries (a
        // cut word the zero entries); otherwise each word is cut or fully
        // connected
        if (__any_sync(0xffffffffu, c != 0u && c != BS_LANE_MASK)) {
          const u32 g = (gout << BS_IN) | (u32)r;
          const int pc = pco + __popc(r);
          const ulonglong2 t0 = s_lt[0 * 256 + (c & 0xffu)], t1 = s_lt[1 * 256 + ((c >> 8) & 0xffu)];
          const ulonglong2 t2 = s_lt[2 * 256 + ((c >> 16) & 0xffu)], t3 = s_lt[3 * 256 + (c >> 24)];
          const u64 sR = t0.x + t1.x + t2.x + t3.x;
          const u64 wm = s_wmid[g];
          u128_add(T, sR * wm, __umul64hi(sR, wm));
          bins[pc * BS_NTHR] += t0.y + t1.y + t2.y + t3.y;
        } else if (c) {
          // every lane state connected: the lane mass is exactly 1
          const u64 wm = s_wmid[(gout << BS_IN) | (u32)r];
          u128_add(T, wm << 62, wm >> 2);
          bins[(pco + __popc(r)) * BS_NTHR] += BS_FULL_COUNTS;
        }
      }
    }
    // item total: exact warp sum of T x thread mass (scale 2^124), times the
    // prefix mass (a class: its items' summed mass), once per item
    const u128 S = warp_sum_u128(mul64x128_shr64(thw, T.lo, T.hi));
    mx w;
    bs_flush_bins(bins, rel, lane);
    if constexpr (phase == 2) {
#if BS_MERGE
      bs_class_counts(W, task, lane, rel, s_nbins);
      w = bs_class_mass(W.cmass + 2 * task, P.mass_exp);
#endif
    } else {
      bs_item_counts(rel, s_nbins, pc_pre, lane);
      w = bs_prefix_mass(P, ptab, prefix);
    }
    facc_add(accR, mx_prod(w, S), w.e);
  }
  if (lane == 0) {
    if (n_walk) atomicAdd(&W.stats[0], n_walk);
    if (n_full) atomicAdd(&W.stats[1], n_full);
    if (n_dead) atomicAdd(&W.stats[2], n_dead);
    s_acc[warp] = accR;
  }
  __syncthreads();
  bs_write_out(W, s_acc, 1, 1, s_nbins, BS_NTHR);
}

#define KERNEL_R_ARGS const __grid_constant__ BsParams P, const u64* __restrict__ lane_tab, \
                  const u64* __restrict__ wmid_tab, const mx* __restrict__ ptab, const BsWork W
#if !BS_MERGE
extern "C" __global__ void KERNEL_BOUNDS bs_kernel(KERNEL_R_ARGS) { bs_kernel_body<0>(P, lane_tab, wmid_tab, ptab, W); }
#else
extern "C" __global__ void __launch_bounds__(BS_MERGE_NTHR) bs_kernel_p1(const __grid_constant__ BsParams P,
    const mx* __restrict__ ptab, const ulonglong2* __restrict__ mtab, int split_log2, const BsWork W) {
  bs_merge_body(P, ptab, mtab, split_log2, W);
}
extern "C" __global__ void KERNEL_BOUNDS bs_kernel_p2(KERNEL_R_ARGS) { bs_kernel_body<2>(P, lane_tab, wmid_tab, ptab, W); }
#endif
#endif

#if BS_GRAD
// ---------------------------------------------------------------------------
// Fused R + N_k + dR/dp.  Every gradient term is a difference of two exact
// integer sums over the two halves of state pairs (X, X + e_i) that carry
// identical weights, so it is exact and non-negative:
//   thread arcs: per-thread totals T of warp lanes t and t ^ 2^i;
//   lane arcs: the 32x32 bit matrix (threads x lanes) of a word is
//     transposed across the warp, so lane j holds the states of lane pattern
//     j; its total T2 (thread-pattern masses from byte tables) pairs lanes j
//     and j ^ 2^i in the same way;
//   walk arcs: A_b, the part of T collected while walk arc b works, against
//     T - A_b; both are summed over items and divided by p_b and 1 - p_b once,
//     at the end;
//   prefix arcs: item totals times the prefix mass without that arc, summed
//     apart for the arc working and failed.
// Per item every quantity is first summed exactly over the warp in 128-bit
// integers with fixed-point per-lane weights; then the lane that owns an arc
// (lanes k and k - 32 own internal arc k) scales it by the item's prefix
// mass (integer floating point) and adds it to that arc's two floating
// 128-bit accumulators in shared memory.  Walk masses are 128-bit (scale
// 2^127).
struct BsGradParams {
  u64 thw_ex[5][32];    // thread-pattern masses without thread arc i (2^63)
  u64 lw_ex[5][32];     // lane-pattern masses without lane arc i (2^63)
  dd inv_p[64], inv_q[64];
};

static_assert(BS_TOP <= 32, "lane k owns internal arc k");

// The prefix factor of internal arc k for this item.  Internal arcs, and
// prefix arcs with p in [2^-20, 1 - 2^-20], take the whole prefix mass: a
// prefix arc's two sums then carry its own factor p or 1 - p, which the
// host divides out once (as for walk arcs) -- the sums' errors are relative
// to their terms, so the division does not amplify them.  Prefix arcs with
// p outside that range (bits set in BS_PEX_MASK) take the item's prefix
// mass without their own factor, from the excluded-arc table.
__device__ __forceinline__ mx bs_arc_factor(const BsParams& P, const mx* __restrict__ ptab,
                                            const mx* __restrict__ ptab_ex, u64 prefix, int k, mx wpre) {
  if (k < BS_TOP || !((BS_PEX_MASK >> k) & 1ull)) return wpre;
  const int j = k - BS_TOP;
  int l = 0, sh = 0;
  while (sh + P.lev_bits[l] <= j) { sh += P.lev_bits[l]; ++l; }
  mx f = wpre;
  int s2 = 0;
  for (int q = 0; q < P.nlev; ++q) {
    const u64 bits = (prefix >> s2) & ((1ull << P.lev_bits[q]) - 1ull);
    const mx t = q == l ? ptab_ex[((size_t)j << P.ex_shift) + bits] : ptab[P.lev_off[q] + bits];
    f = q ? mx_mul(f, t) : t;
    s2 += P.lev_bits[q];
  }
  return f;
}

// The mass factors of an item (or class) for R, of internal arc `lane` and of
// arc `lane + 32`.
#if BS_MERGE
#define BS_CLASS_FACTORS() wpre = f0 = f1 = bs_class_mass(W.cmass + 2 * task, P.mass_exp)
#else
#define BS_CLASS_FACTORS() wpre = f0 = f1 = mx{0ull, 0, 0}
#endif
#define BS_FACTORS()                                                                                  \
  if constexpr (phase == 2) {                                                                         \
    BS_CLASS_FACTORS();                                                                               \
  } else {                                                                                            \
    wpre = bs_prefix_mass(P, ptab, prefix);                                                           \
    f0 = bs_arc_factor(P, ptab, ptab_ex, prefix, lane, wpre);                                         \
    f1 = lane + 32 < BS_M ? bs_arc_factor(P, ptab, ptab_ex, prefix, lane + 32, wpre) : wpre;          \
  }

template <int PHASE>
__device__ __forceinline__ void bs_kernel_grad_body(
    const BsParams& P, const BsGradParams& Q, const u64* __restrict__ lane_tab,
    const u64* __restrict__ thr_tab, const u64* __restrict__ wmid128, const mx* __restrict__ ptab,
    const mx* __restrict__ ptab_ex, const BsWork& W) {
  extern __shared__ __align__(16) unsigned char smem[];
  ulonglong2* s_lt = (ulonglong2*)smem;                     // [4][256] {lane mass 2^62, packed counts}
  ulonglong2* s_wm = s_lt + 4 * 256;                        // [2^L] walk masses {lo, hi} (2^127)
  u64* s_tt = (u64*)(s_wm + (1 << BS_L));                   // [4][256] thread-pattern masses (2^62)
  u64* s_bins = s_tt + 4 * 256;                             // [L + 1][NTHR]
  u128* s_A = (u128*)(s_bins + (BS_L + 1) * BS_NTHR);       // [BS_OUT][NTHR]
  u64* s_nbins = (u64*)(s_A + (BS_OUT > 0 ? BS_OUT : 1) * BS_NTHR);
  // per warp: R, then A_k and B_k of every arc k (of a class: of the arcs
  // below the prefix)
  constexpr int n_acc = PHASE == 2 ? 1 + 2 * BS_TOP : 1 + 2 * BS_M, m_acc = PHASE == 2 ? BS_TOP : BS_M;
  facc* s_acc = (facc*)(((size_t)(s_nbins + BS_M + 1) + (BS_NTHR / 32) * (BS_TOP + 1) * 4 + 7) & ~(size_t)7);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 4 * 256; i += BS_NTHR) s_lt[i] = ((const ulonglong2*)lane_tab)[i];
  for (int i = tid; i < 4 * 256; i += BS_NTHR) s_tt[i] = thr_tab[i];
  for (int i = tid; i < (1 << BS_L); i += BS_NTHR) s_wm[i] = ((const ulonglong2*)wmid128)[i];
  for (int i = tid; i <= BS_M; i += BS_NTHR) s_nbins[i] = 0ull;
  u64 n_list = 0, next = 0;
  if constexpr (PHASE == 2) {
    bs_wait_previous();
    bs_let_next_start();
    n_list = *W.list_n;
    next = (u64)warp * gridDim.x + blockIdx.x;
    if (blockIdx.x >= n_list) return;   // no class
  }
  for (int i = tid; i < (BS_NTHR / 32) * n_acc; i += BS_NTHR) s_acc[i] = facc{u128{0ull, 0ull}, 0, 0};
  if (PHASE != 2) __syncthreads();
  else if (bs_block_given_up(W.status)) return;
  facc* acc = s_acc + warp * n_acc;
  u64* bins = s_bins + tid;
  u128* A = s_A + tid;
  const BsTr tr = bs_tr_init(lane);
  const bool thr_on = lane < (1 << BS_TB);
  const u64 thw = thr_on ? P.thw[lane] : 0ull;
  const u64 t_start = bs_timer();
  u64 n_walk = 0, n_full = 0, n_dead = 0;
#if BS_ACC_REG
  // short items: this lane's accumulators -- R and the two sums of internal
  // arcs `lane` and `lane + 32` -- in registers.  Long items keep them all in
  // the shared slots: registers are worth more to the walk.
  facc accR = facc{u128{0ull, 0ull}, 0, 0}, accA = accR, accB = accR;
#if BS_M > 32
  facc accA2 = accR, accB2 = accR;
#endif
#endif
  u32 a[BS_M];
  bs_init_arcs(a, lane);
  constexpr int phase = PHASE;
  u32* rel = (u32*)(s_nbins + BS_M + 1) + warp * (BS_TOP + 1);   // an item's counts below the prefix

  for (;;) {
    u64 task = 0;
    if constexpr (phase == 2) {
      task = next < n_list ? (u64)W.list[next] : ~0ull;
      next = bs_next_class(W, n_list, (u64)gridDim.x * (BS_NTHR / 32), lane);
    }
    if (lane == 0) {
      if constexpr (phase == 0) task = atomicAdd(W.counter, 1ull);
      if (P.budget_ns && (phase == 2 ? bs_run_late(P.budget_ns, W.start, W.status)
                                     : bs_late(P.budget_ns, t_start, W.status))) task = ~0ull;
    }
    task = __shfl_sync(0xffffffffu, task, 0);
    u64 prefix;
    if constexpr (phase == 2) {   // a class, by its slot
      if (task == ~0ull) break;
#if BS_MERGE
      prefix = W.rep[task];
#endif
    } else {
      if (task >= P.n_tasks) break;
      prefix = P.task_lo + task;
    }
#pragma unroll
    for (int j = 0; j < BS_D; ++j) a[BS_TOP + j] = 0u - (u32)((prefix >> j) & 1ull);
    const int pc_pre = __popcll((long long)prefix);
    int pr = 0;
    if (P.prune && phase == 0) {
      pr = bs_prune(a);
      if (pr == 1) { ++n_dead; continue; }
    }
#if BS_ACC_REG
    // the prefix factors of an item that is not cut off, before its walk so
    // that their table loads overlap it (a cut-off item needs none: with
    // prune-aware prefix arcs most items are cut off or fully connected)
    mx wpre, f0, f1;
    BS_FACTORS();
#endif
    u128 S;      // sum over the warp of T x thread mass, scale 2^124
    // warp sums of the internal arc this lane owns (internal arcs are below
    // 32): the exact pair difference, or for a walk arc A and T - A
    u128 myX = u128{0ull, 0ull}, myY = u128{0ull, 0ull};
    if (pr == 2) {
      ++n_full;
      for (int j = lane; j <= BS_TOP; j += 32) atomicAdd(&s_nbins[pc_pre + j], P.binom[j]);
      S = u128{0ull, 1ull << 60};   // the whole item: mass 1 at scale 2^124
    } else {
      ++n_walk;
      u32 e[BS_NCORE > 0 ? BS_NCORE : 1];
      bs_inv(a, e);
#pragma unroll
      for (int r = 0; r <= BS_L; ++r) bins[r * BS_NTHR] = 0ull;
#pragma unroll
      for (int b = 0; b < BS_OUT; ++b) A[b * BS_NTHR] = u128{0ull, 0ull};
      u128 T = u128{0ull, 0ull}, T2 = u128{0ull, 0ull};
      u128 Ain[BS_IN > 0 ? BS_IN : 1];
#pragma unroll
      for (int b = 0; b < BS_IN; ++b) Ain[b] = u128{0ull, 0ull};
      u32 gout = 0;
      int pco = 0;
#pragma unroll 1
      for (u32 s = 0; s < (1u << BS_OUT); ++s) {
        if (s) {
          const int b = __ffs(s) - 1;
          gout ^= 1u << b;
          const bool on = (gout >> b) & 1u;
          pco += on ? 1 : -1;
          // outer walk arc b: A collects the growth of T while the arc works
          u128 ab = A[b * BS_NTHR];
          if (on) ab = u128_sub(ab, T); else u128_add(ab, T.lo, T.hi);
          A[b * BS_NTHR] = ab;
        }
        u32 w[BS_L > 0 ? BS_L : 1];
#pragma unroll
        for (int b = 0; b < BS_OUT; ++b) w[BS_IN + b] = 0u - ((gout >> b) & 1u);
        // the inner words' packed counts by inner popcount, in registers
        u64 nb[BS_IN + 1];
#pragma unroll
        for (int j = 0; j <= BS_IN; ++j) nb[j] = 0ull;
#pragma unroll
        for (int r = 0; r < (1 << BS_IN); ++r) {
#pragma unroll
          for (int b = 0; b < BS_IN; ++b) w[b] = ((r >> b) & 1) ? ~0u : 0u;
          const u32 g = (gout << BS_IN) | (u32)r;
          const u32 c = bs_var(e, w) & BS_LANE_MASK;
          const ulonglong2 wv = s_wm[g];
          if (__any_sync(0xffffffffu, c != 0u && c != BS_LANE_MASK)) {
            // some word of the warp is partly connected: no branch on the
            // word's class (a cut word reads the zero entries, a connected
            // one the mass of all its lanes), and the lane transpose
            const ulonglong2 t0 = s_lt[0 * 256 + (c & 0xffu)], t1 = s_lt[1 * 256 + ((c >> 8) & 0xffu)];
            const ulonglong2 t2 = s_lt[2 * 256 + ((c >> 16) & 0xffu)], t3 = s_lt[3 * 256 + (c >> 24)];
            const u128 x = mul64x128_shr64(t0.x + t1.x + t2.x + t3.x, wv.x, wv.y);
            u128_add(T, x.lo, x.hi);
#pragma unroll
            for (int b = 0; b < BS_IN; ++b)
              if ((r >> b) & 1) u128_add(Ain[b], x.lo, x.hi);
            nb[__popc(r)] += t0.y + t1.y + t2.y + t3.y;
            const u32 ct = bs_transpose32(c, tr);
            const u64 s2 = s_tt[ct & 0xffu] + s_tt[256 + ((ct >> 8) & 0xffu)] +
                           s_tt[512 + ((ct >> 16) & 0xffu)] + s_tt[768 + (ct >> 24)];
            const u128 x2 = mul64x128_shr64(s2, wv.x, wv.y);
            u128_add(T2, x2.lo, x2.hi);
          } else if (c) {
            // every word of the warp is cut or fully connected (no lane-arc
            // pair differs): a connected word's lane mass is exactly 1, the
            // walk mass at scale 2^125
            const u128 x = u128{(wv.x >> 2) | (wv.y << 62), wv.y >> 2};
            u128_add(T, x.lo, x.hi);
#pragma unroll
            for (int b = 0; b < BS_IN; ++b)
              if ((r >> b) & 1) u128_add(Ain[b], x.lo, x.hi);
            nb[__popc(r)] += BS_FULL_COUNTS;
          }
        }
#pragma unroll
        for (int j = 0; j <= BS_IN; ++j) bins[(pco + j) * BS_NTHR] += nb[j];
      }
#pragma unroll
      for (int b = 0; b < BS_OUT; ++b)
        if ((gout >> b) & 1u) { u128 ab = A[b * BS_NTHR]; u128_add(ab, T.lo, T.hi); A[b * BS_NTHR] = ab; }
      bs_flush_bins(bins, rel, lane);
      if constexpr (phase == 2) {
#if BS_MERGE
        bs_class_counts(W, task, lane, rel, s_nbins);
#endif
      } else {
        bs_item_counts(rel, s_nbins, pc_pre, lane);
      }
      // ---- exact warp sums; slot k of `red` holds internal arc k's value
      S = warp_sum_u128(mul64x128_shr64(thw, T.lo, T.hi));
#pragma unroll
      for (int i = 0; i < BS_ELL; ++i) {
        const u128 o = shfl_xor_u128(T2, 1 << i);
        const u128 d2 = u128_sub(T2, o);
        const u128 v = ((lane >> i) & 1) ? mul64x128_shr64(Q.lw_ex[i][lane], d2.lo, d2.hi) : u128{0ull, 0ull};
        const u128 sv = warp_sum_u128(v);
        if (lane == i) myX = sv;
      }
#pragma unroll
      for (int i = 0; i < BS_TB; ++i) {
        const u128 o = shfl_xor_u128(T, 1 << i);
        const u128 d1 = u128_sub(T, o);
        const u128 v = (((lane >> i) & 1) && thr_on) ? mul64x128_shr64(Q.thw_ex[i][lane], d1.lo, d1.hi)
                                                     : u128{0ull, 0ull};
        const u128 sv = warp_sum_u128(v);
        if (lane == BS_ELL + i) myX = sv;
      }
#pragma unroll
      for (int b = 0; b < BS_L; ++b) {
        const u128 Ab = b < BS_IN ? Ain[b < BS_IN ? b : 0] : A[(b >= BS_IN ? b - BS_IN : 0) * BS_NTHR];
        const u128 sa = warp_sum_u128(mul64x128_shr64(thw, Ab.lo, Ab.hi));
        // the failed half: S - sa, the lanes' truncated products of T less
        // those of A (each lane's difference is that of T - A, or one unit
        // more, at scale 2^124; never negative)
        const u128 sz = u128_sub(S, sa);
        if (lane == BS_WALK0 + b) { myX = sa; myY = sz; }
      }
    }
    // ---- per-arc scaling on the owning lanes (internal arcs lane, lane + 32)
#if !BS_ACC_REG
    mx wpre, f0, f1;
    BS_FACTORS();
    facc accR, accA, accB;
    if (lane == 0) accR = acc[0];
    if (lane < m_acc) {
      accA = acc[1 + 2 * lane];
      accB = acc[2 + 2 * lane];
    }
#endif
    if (lane == 0) facc_add(accR, mx_prod(wpre, S), wpre.e);
    {
      // arc `lane`: a prefix arc goes into A when it works in this item and
      // into B when it fails (the item's mass without its factor); an
      // internal arc of a fully connected item has no pair that differs
      // (a class's prefix arcs are left to bs_fold, from its sum S)
      u128 X = u128{0ull, 0ull}, Y = u128{0ull, 0ull};
      if (lane >= BS_TOP) {
        if (phase == 0 && lane < BS_M) {
          if ((prefix >> (lane - BS_TOP)) & 1ull) X = S; else Y = S;
        }
      } else if (pr != 2) {
        X = myX;
        Y = myY;
      }
#if BS_MERGE
      if (phase == 2 && lane == 0) W.csum[task] = make_ulonglong2(S.lo, S.hi);
#endif
      facc_add(accA, mx_prod(f0, X), f0.e);
      facc_add(accB, mx_prod(f0, Y), f0.e);
    }
#if !BS_ACC_REG
    if (lane == 0) acc[0] = accR;
    if (lane < m_acc) {
      acc[1 + 2 * lane] = accA;
      acc[2 + 2 * lane] = accB;
    }
#endif
    if (phase == 0 && lane + 32 < BS_M) {
      // arc lane + 32 is a prefix arc (lanes own arcs below 32 and the top
      // prefix arcs): the item's total, by whether the arc works here
      const int j = lane + 32 - BS_TOP;
#if BS_ACC_REG && BS_M > 32
      if ((prefix >> j) & 1ull) facc_add(accA2, mx_prod(f1, S), f1.e);
      else facc_add(accB2, mx_prod(f1, S), f1.e);
#else
      facc* ak = acc + 1 + 2 * (lane + 32);
      facc va = ak[0], vb = ak[1];
      if ((prefix >> j) & 1ull) facc_add(va, mx_prod(f1, S), f1.e);
      else facc_add(vb, mx_prod(f1, S), f1.e);
      ak[0] = va;
      ak[1] = vb;
#endif
    }
    __syncwarp();
  }
  if (lane == 0) {
    if (n_walk) atomicAdd(&W.stats[0], n_walk);
    if (n_full) atomicAdd(&W.stats[1], n_full);
    if (n_dead) atomicAdd(&W.stats[2], n_dead);
  }
#if BS_ACC_REG
  if (lane == 0) acc[0] = accR;
  if (lane < m_acc) {
    acc[1 + 2 * lane] = accA;
    acc[2 + 2 * lane] = accB;
  }
#if BS_M > 32
  if (PHASE == 0 && lane + 32 < BS_M) {
    acc[1 + 2 * (lane + 32)] = accA2;
    acc[2 + 2 * (lane + 32)] = accB2;
  }
#endif
#endif
  // ---- per block: R, then A_k and B_k of every arc; the host forms the
  // gradient (A - B for prefix arcs, A / p - B / (1 - p) for walk arcs, A
  // for lane and thread arcs)
  __syncthreads();
  bs_write_out(W, s_acc, n_acc, n_acc, s_nbins, BS_NTHR);
}

#define KERNEL_G_ARGS const __grid_constant__ BsParams P, const __grid_constant__ BsGradParams Q, \
                  const u64* __restrict__ lane_tab, const u64* __restrict__ thr_tab, \
                  const u64* __restrict__ wmid128, const mx* __restrict__ ptab, \
                  const mx* __restrict__ ptab_ex, const BsWork W
#define KERNEL_G_PASS P, Q, lane_tab, thr_tab, wmid128, ptab, ptab_ex, W
#if !BS_MERGE
extern "C" __global__ void KERNEL_BOUNDS bs_kernel_grad(KERNEL_G_ARGS) { bs_kernel_grad_body<0>(KERNEL_G_PASS); }
#else
extern "C" __global__ void __launch_bounds__(BS_MERGE_NTHR) bs_kernel_grad_p1(const __grid_constant__ BsParams P,
    const mx* __restrict__ ptab, const ulonglong2* __restrict__ mtab, int split_log2, const BsWork W) {
  bs_merge_body(P, ptab, mtab, split_log2, W);
}
extern "C" __global__ void KERNEL_BOUNDS bs_kernel_grad_p2(KERNEL_G_ARGS) { bs_kernel_grad_body<2>(KERNEL_G_PASS); }
#endif

#if BS_MERGE
// ---------------------------------------------------------------------------
// The prefix arcs' gradient of a merged run.  Every item has its conditional
// reliability V: 0 when cut, 1 when connected throughout, else its class's S.
// A warp folds a block of items arc by arc, V' = V0 + p (V1 - V0): lane u
// holds the items of mid pattern u and folds the low arcs over its 32 items,
// the mid arcs fold over the lanes.  On the way each arc of the block
// collects the pair differences V1 - V0 weighted by the other arcs' masses;
// the arcs above it take the block's V, by whether they work (the host
// divides those sums by p and 1 - p).  A fold costs one product for two
// items, so the whole launch is a few instructions per item, where adding
// every item to every prefix arc took about 250.
// ---------------------------------------------------------------------------
struct BsFoldParams {
  u64 p[10];            // low, then mid arcs: p at 2^63
  u64 wlow[31];         // masses (2^63) of the low arcs above arc b: 16, 8, 4, 2, 1 patterns for b = 0..4
  u64 wmid[31];         // of the mid arcs above mid arc b
  u64 mid[32];          // mid pattern masses (2^63)
};
// Few blocks (TEAM): the four warps of a thread block share one, a group of
// eight items per lane each, and the first folds their results -- a block is
// otherwise 15 us of one warp's latency.
template <bool TEAM>
__device__ __forceinline__ void bs_fold_body(const BsParams& P, const BsFoldParams& Q, const mx* __restrict__ ptab,
                                             const BsWork& W) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // A_k and B_k of every prefix arc, per warp
  __shared__ facc s_acc[BS_MERGE_NTHR / 32][BS_D ? 2 * BS_D : 1];
  __shared__ u128 s_V[TEAM ? 4 : 1][32], s_X[TEAM ? 4 : 1][4];   // a team's folded groups and sums
  facc* acc = s_acc[warp];
  for (int i = lane; i < 2 * BS_D; i += 32) acc[i] = facc{u128{0ull, 0ull}, 0, 0};
  bs_wait_previous();
  // (the masks and slots of a run that was given up are not all written)
  if (bs_block_given_up(W.status)) return;
  const u64 nblk = P.n_tasks >> BS_BLK, blk0 = P.task_lo >> BS_BLK;
  const u64 step = TEAM ? (u64)gridDim.x : (u64)gridDim.x * (BS_MERGE_NTHR / 32);
  const u64 m_mid = Q.mid[lane];
  // lane l < BS_BLK: arc l of the block; lanes: arcs `lane` and `lane + 32` above it
  facc accP = facc{u128{0ull, 0ull}, 0, 0}, accA = accP, accB = accP, accA2 = accP, accB2 = accP;
  for (u64 b = TEAM ? blockIdx.x : (u64)blockIdx.x * (BS_MERGE_NTHR / 32) + warp; b < nblk; b += step) {
    if (P.budget_ns && (TEAM ? bs_block_time_up(P.budget_ns, W.start, W.status)
                             : bs_time_up(P.budget_ns, W.start, W.status, lane))) break;
    const u64 hi = blk0 + b;
    const uint2 m = W.cmask[b * 32 + lane];
    if (!__any_sync(0xffffffffu, m.x | m.y)) continue;   // (the same in every warp of a team)
    const u32* cls = W.cls + (b << BS_BLK) + lane;
    u128 G[5], X, V;
#pragma unroll
    for (int i = 0; i < 5; ++i) G[i] = u128{0ull, 0ull};
    auto item = [&](int j) {
      u128 v = u128{0ull, (m.x >> j) & 1u ? 1ull << 60 : 0ull};
      if ((m.y >> j) & 1u) {
        const ulonglong2 s = W.csum[cls[j << BS_MID]];
        v = u128{s.x, s.y};
      }
      return v;
    };
    if constexpr (TEAM) {
      s_V[warp][lane] = bs_fold_group(Q.p, Q.wlow, warp, G, item);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const u128 g = bs_fold_sum(G[i], m_mid);
        if (lane == i) s_X[warp][i] = g;
      }
      __syncthreads();
      if (warp == 0) {
        u128 T[4] = {s_V[0][lane], s_V[1][lane], s_V[2][lane], s_V[3][lane]};
        V = bs_fold_mid<3>(bs_fold_groups(Q.p, Q.wlow, T, G), G, BS_LOW, BS_MID, Q.p + 5, Q.wmid, m_mid, lane, X);
        if (lane < 3 && lane < BS_LOW)
#pragma unroll
          for (int q = 0; q < 4; ++q) u128_add(X, s_X[q][lane].lo, s_X[q][lane].hi);
      }
      __syncthreads();
      if (warp != 0) continue;
    } else {
      V = bs_fold_mid<0>(bs_fold_low(Q.p, Q.wlow, G, item), G, BS_LOW, BS_MID, Q.p + 5, Q.wmid, m_mid, lane, X);
    }
    const mx w = bs_level_mass(P.nlev_hi, P.hi_bits, P.hi_off, ptab, hi);
    if (lane < BS_BLK) facc_add(accP, mx_prod(w, X), w.e);
    const u128 Sv = mx_prod(w, V);
    if (lane < BS_HI) { if ((hi >> lane) & 1ull) facc_add(accA, Sv, w.e); else facc_add(accB, Sv, w.e); }
    if (lane + 32 < BS_HI) { if ((hi >> (lane + 32)) & 1ull) facc_add(accA2, Sv, w.e); else facc_add(accB2, Sv, w.e); }
  }
  if (lane < BS_BLK) acc[2 * lane] = accP;
  if (lane < BS_HI) {
    acc[2 * (BS_BLK + lane)] = accA;
    acc[2 * (BS_BLK + lane) + 1] = accB;
  }
  if (lane + 32 < BS_HI) {
    acc[2 * (BS_BLK + lane + 32)] = accA2;
    acc[2 * (BS_BLK + lane + 32) + 1] = accB2;
  }
  __syncthreads();
  bs_add_out(W.out_limbs + 8 * (1 + 2 * BS_TOP), s_acc[0], 2 * BS_D, 2 * BS_D, BS_MERGE_NTHR);
}
extern "C" __global__ void __launch_bounds__(BS_MERGE_NTHR, 5) bs_kernel_grad_p3(
    const __grid_constant__ BsParams P, const __grid_constant__ BsFoldParams Q, const mx* __restrict__ ptab,
    const BsWork W) {
  if (gridDim.x * (BS_MERGE_NTHR / 32) > P.n_tasks >> BS_BLK) bs_fold_body<true>(P, Q, ptab, W);
  else bs_fold_body<false>(P, Q, ptab, W);
}
#endif
#endif
)PBAT";


// Batched: every network's connectivity program is a struct of static
// functions (inv, var, and sig where items are merged) with its sizes as
// constants.  The walking kernel takes one item of every class -- or, where
// items are not merged, (network, prefix) items from one ticket, networks
// with the most items first -- and switches to that network's connectivity
// function (bsb_conn), which only stages the item's 2^L connectivity words in
// shared memory.  The accumulate (bsb_finish) is written once in the kernel body,
// so the module's compile time barely grows with the number of networks: it
// weights each word by every p-vector, 16 at a time in registers (byte
// tables interleaved by p-vector, read through L1), and adds each item's
// mass per p-vector exactly into a 256-bit fixed-point number (eight 32-bit
// chunks in 64-bit limbs) with integer atomics.  N_k counts collect per warp
// in shared memory.
static const char* kBsBatchTemplate = R"PBAT(
#define BSB_LIMBS 8
#define BSB_KC 16
struct BGraph {
  u64 task_begin, n_tasks;
  int gidx, m, nlev, prune;
  int lev_bits[8], lev_off[8];
  int lt_off, nt_off, wm_off, pt_off, pt_size, thw_off, nk_off, tb;
  int L, top;
  u32 lane_mask;
  int pad0;
  // gradient module only: offsets of the 128-bit walk masses, the thread
  // byte tables, the excluded-arc masses of lane, thread and prefix arcs,
  // and of this network's results; lane arcs, prefix arcs, thread mask
  int wm2_off, tt_off, lwex_off, thwex_off, ptex_off, out_off, ell, d;
  u32 thr_mask;
  int pad1;
  u64 full_counts;
  u64 pex_mask;   // gradient module: prefix arcs using the excluded-arc tables
  u64 binom[64];
  // merged modules: the arcs of a block and above it, the signature, and
  // where this network's blocks, slots and items begin (see BMerge)
  int low, mid, nhi, nsig, slots_log2, pad2;
  u64 blk_begin, slot_base, item_base;
};
// Work arrays of a merged batch.  Slots hold signatures and the class that
// each stands for; a class its network, one of its items, its number of items
// by popcount, and per p-vector its mass (two chunks) and its sum S.  Blocks:
// per lane the items connected throughout and left to walk (a bit each);
// items: the slot, and for the first of a lane with that slot the lane's items
// with it.
struct BMerge {
  u64* key; u32* id_of;
  u32* net; u64* rep; u32* hist; u64* cmass; ulonglong2* csum;
  uint2* cmask; uint2* ent;
  u64* n_classes; u64* ticket; u64* start;   // start: when the run began (bs_run_start)
  u64 n_blocks;
  // few blocks: 2^split_log2 warps share one in the first (its words and its
  // p-vectors), `parts` in the second launch (its p-vectors)
  int split_log2, parts;
  u32 cap; int hist_stride;
  const ulonglong2* nib; const ulonglong2* mid; const u64* fold;
};
#ifndef BSB_MERGE
#define BSB_MERGE 0
#endif

// add P * 2^(-123 - e) (P < 2^124, e >= 0) to the 256-bit limbs (scale 2^250)
__device__ __forceinline__ void bsb_limb_add(u64* limbs, u128 P, int e) { bs_limb_add(limbs, P, 127 - e); }

// prefix mass of one p-vector: product over the levels of its table t
__device__ __forceinline__ mx bsb_prefix_mass(const mx* __restrict__ t, int nlev, const int (&lev_bits)[8],
                                              const int (&lev_off)[8], u64 prefix) {
  mx w = mx{1ull << 63, 0, 0};
  int sh = 0;
#pragma unroll
  for (int l = 0; l < 8; ++l) {
    if (l >= nlev) break;
    const u64 v = (prefix >> sh) & ((1ull << lev_bits[l]) - 1ull);
    const ulonglong2 q = __ldg((const ulonglong2*)(t + lev_off[l] + v));
    const mx f = mx{q.x, (int)(u32)q.y, 0};
    w = l ? mx_mul(w, f) : f;
    sh += lev_bits[l];
  }
  return w;
}

template <class G>
__device__ __forceinline__ u32 bsb_uniform(const u32* a) {
  u32 e[G::NCORE > 0 ? G::NCORE : 1];
  G::inv(a, e);
  u32 w[G::L > 0 ? G::L : 1];
#pragma unroll
  for (int b = 0; b < G::L; ++b) w[b] = a[G::WALK0 + b];
  return G::var(e, w);
}

// A merged module walks few items and holds two functions per network: these
// are calls, compiled apart (64 networks: NVRTC 11.7 s inlined, 5.4 s so).
#if BSB_MERGE
#define BSB_NETWORK __noinline__
#else
#define BSB_NETWORK __forceinline__
#endif
// The per-network part of one item: its state words, the monotone prune,
// and the connectivity word of every walk state into cw (stride BSB_NTHR).
// Returns 0 when every state of the item is cut, 1 when every state is
// connected, 2 when cw holds the item's words.
template <class G>
__device__ BSB_NETWORK int bsb_conn(u64 prefix, int lane, int prune, u32* cw) {
  u32 a[G::M];
#pragma unroll
  for (int i = 0; i < G::ELL; ++i)
    a[i] = i == 0 ? 0xAAAAAAAAu : i == 1 ? 0xCCCCCCCCu : i == 2 ? 0xF0F0F0F0u : i == 3 ? 0xFF00FF00u : 0xFFFF0000u;
#pragma unroll
  for (int i = 0; i < G::TB; ++i) a[G::ELL + i] = 0u - (u32)((lane >> i) & 1);
#pragma unroll
  for (int b = 0; b < G::L; ++b) a[G::WALK0 + b] = 0u;
#pragma unroll
  for (int j = 0; j < G::D; ++j) a[G::TOP + j] = 0u - (u32)((prefix >> j) & 1ull);
  if (prune) {
    // one evaluation for both extremes: bit 0 has every arc below the prefix
    // up, the other bits have them all down (the prefix arcs are the same in
    // every bit)
    u32 u[G::M];
#pragma unroll
    for (int k = 0; k < G::M; ++k) u[k] = k < G::TOP ? 1u : a[k];
    const u32 ext = bsb_uniform<G>(u);
    if (!(ext & 1u)) return 0;
    if (ext & 2u) return 1;
  }
  u32 e[G::NCORE > 0 ? G::NCORE : 1];
  G::inv(a, e);
#pragma unroll 1
  for (u32 g = 0; g < (1u << G::L); ++g) {
    u32 w[G::L > 0 ? G::L : 1];
#pragma unroll
    for (int b = 0; b < G::L; ++b) w[b] = 0u - ((g >> b) & 1u);
    cw[g * BSB_NTHR] = G::var(e, w) & G::LANE_MASK;
  }
  return 2;
}
// Everything of an item past connectivity, shared by every network (inlined
// once, in the kernel body): counts N_k, then sums the exact fixed-point
// mass of every p-vector, BSB_KC of them at a time (Eq. 1 restricted to the
// item) -- per thread in registers, then over the warp by a reduce-scatter
// that leaves p-vector kk's item total on lanes 2 idx(kk) and 2 idx(kk) + 1,
// so that the prefix scaling and the limb additions run on 16 lanes at once.
// The network's constants are read once into registers.
// add the warp's counts of network B (k = 0..m) to the global N_k, then clear
__device__ __forceinline__ void bsb_flush_counts(const BGraph* __restrict__ B, u64* nkw, u64* nk, int lane) {
  const int m = B->m, off = B->nk_off;
  for (int i = lane; i <= m; i += 32) {
    const u64 v = nkw[i];
    if (v) atomicAdd(&nk[off + i], v);
    nkw[i] = 0ull;
  }
  __syncwarp();
}

// N_k of a class: its item's counts below the prefix (rel) for every popcount
// that its prefixes have, into the warp's counts nkw.
__device__ __forceinline__ void bsb_class_counts(const BMerge& A, u64 cls, int d, int top, int lane, u32* rel, u64* nkw) {
  __syncwarp();
  const u64 r = lane <= top ? rel[lane] : 0u;
  const u32* h = A.hist + cls * A.hist_stride;
  for (int q = 0; q <= d; ++q) {
    const u32 n = h[q];
    if (n && r) nkw[q + lane] += n * r;
    __syncwarp();
  }
  if (lane <= top) rel[lane] = 0u;
  __syncwarp();
}
// this thread's counts c11 by walk popcount + lane class: an item's to nkw, a
// class's below the prefix, then for all its items
#if BSB_MERGE
#define BSB_COUNTS()                                                          \
  if (thr_on) {                                                               \
    _Pragma("unroll") for (int i = 0; i < 11; ++i)                            \
      if (c11[i]) atomicAdd(&rel[__popc(lane) + i], (u32)c11[i]);             \
  }                                                                           \
  bsb_class_counts(A, cls, Bp->d, top, lane, rel, nkw)
#else
#define BSB_COUNTS()                                                          \
  if (thr_on) {                                                               \
    _Pragma("unroll") for (int i = 0; i < 11; ++i)                            \
      if (c11[i]) atomicAdd(&nkw[pc_pre + __popc(lane) + i], c11[i]);         \
  }
#endif

// N_k counts go to the warp's own array nkw (indexed by k within the
// network), which the kernel flushes to global memory when the warp moves
// to another network and at the end.
__device__ __forceinline__ void bsb_finish(const BGraph* __restrict__ Bp, int st, u64 prefix, int lane, int K,
                                           int Kp, const u64* __restrict__ lt, const u64* __restrict__ nt,
                                           const u64* __restrict__ wm, const mx* __restrict__ pt,
                                           const u64* __restrict__ thw, u64* limbs, u64* nkw, u64* bins,
                                           const u32* cw, const BMerge& A, u64 cls, u32* rel) {
  constexpr int nsh[6] = BS_NK_SHIFTS, nwd[6] = BS_NK_WIDTHS;
  const int gidx = Bp->gidx, L = Bp->L, tb = Bp->tb, nlev = Bp->nlev, top = Bp->top;
  const int lt_off = Bp->lt_off, nt_off = Bp->nt_off, wm_off = Bp->wm_off, pt_off = Bp->pt_off;
  const int pt_size = Bp->pt_size, thw_off = Bp->thw_off;
  const u32 lane_mask = Bp->lane_mask;
  const u64 full_counts = Bp->full_counts;
  int lev_bits[8], lev_off[8];
#pragma unroll
  for (int l = 0; l < 8; ++l) {
    lev_bits[l] = Bp->lev_bits[l];
    lev_off[l] = Bp->lev_off[l];
  }
  const int pc_pre = __popcll((long long)prefix);
  u64* glimbs = limbs + (size_t)gidx * K * BSB_LIMBS;
  const mx* gpt = pt + pt_off;
  if (st == 1) {
    // every state connected: binomial counts, and per p-vector the prefix mass
    for (int j = lane; j <= top; j += 32) nkw[pc_pre + j] += __ldg(&Bp->binom[j]);
    for (int k = lane; k < K; k += 32) {
      const mx w = bsb_prefix_mass(gpt + (size_t)k * pt_size, nlev, lev_bits, lev_off, prefix);
      bsb_limb_add(glimbs + (size_t)k * BSB_LIMBS, mx_prod(w, u128{0ull, 1ull << 60}), w.e);
    }
    return;
  }
  const int nw = 1 << L;
  for (int r = 0; r <= L; ++r) bins[r * BSB_NTHR] = 0ull;
  const u64* ntg = nt + nt_off;
  for (int g = 0; g < nw; ++g) {
    const u32 c = cw[g * BSB_NTHR];
    if (!c) continue;
    bins[__popc(g) * BSB_NTHR] += c == lane_mask ? full_counts
        : __ldg(ntg + (c & 0xffu)) + __ldg(ntg + 256 + ((c >> 8) & 0xffu)) +
          __ldg(ntg + 512 + ((c >> 16) & 0xffu)) + __ldg(ntg + 768 + (c >> 24));
  }
  const bool thr_on = lane < (1 << tb);
  {
    // this thread's counts by r + cl (walk popcount + lane class), then
    // shared atomics at k = prefix + thread + r + cl
    u64 c11[11];
#pragma unroll
    for (int i = 0; i < 11; ++i) c11[i] = 0ull;
#pragma unroll
    for (int r = 0; r <= 5; ++r) {
      if (r > L) break;
      const u64 n = bins[r * BSB_NTHR];
#pragma unroll
      for (int cl = 0; cl < 6; ++cl) c11[r + cl] += (n >> nsh[cl]) & ((1ull << nwd[cl]) - 1ull);
    }
    BSB_COUNTS();
  }
  const u64* ltg = lt + lt_off;
  const u64* wmg = wm + wm_off;
  const u64* thg = thw + thw_off + (size_t)lane * Kp;
  // p-vector whose total this lane holds after the reduce-scatter
  const int idx = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
  for (int k0 = 0; k0 < K; k0 += BSB_KC) {
    const int kc = min(BSB_KC, K - k0);
    u128 T[BSB_KC];
#pragma unroll
    for (int kk = 0; kk < BSB_KC; ++kk) T[kk] = u128{0ull, 0ull};
    for (int g = 0; g < nw; ++g) {
      const u32 c = cw[g * BSB_NTHR];
      if (!c) continue;
      // table rows hold whole chunks of 16 p-vectors (zero past K), so all
      // loads of a word are unconditional and in flight together
      const ulonglong2* wv = (const ulonglong2*)(wmg + (size_t)g * Kp + k0);
      if (c == lane_mask) {
        // every lane state connected: lane mass exactly 1, the walk mass at
        // scale 2^125
#pragma unroll
        for (int h = 0; h < BSB_KC / 2; ++h) {
          const ulonglong2 ww = __ldg(wv + h);
          u128_add(T[2 * h], ww.x << 62, ww.x >> 2);
          u128_add(T[2 * h + 1], ww.y << 62, ww.y >> 2);
        }
        continue;
      }
      const ulonglong2* l0 = (const ulonglong2*)(ltg + (size_t)(0 * 256 + (c & 0xffu)) * Kp + k0);
      const ulonglong2* l1 = (const ulonglong2*)(ltg + (size_t)(1 * 256 + ((c >> 8) & 0xffu)) * Kp + k0);
      const ulonglong2* l2 = (const ulonglong2*)(ltg + (size_t)(2 * 256 + ((c >> 16) & 0xffu)) * Kp + k0);
      const ulonglong2* l3 = (const ulonglong2*)(ltg + (size_t)(3 * 256 + (c >> 24)) * Kp + k0);
#pragma unroll
      for (int h = 0; h < BSB_KC / 2; ++h) {
        const ulonglong2 a0 = __ldg(l0 + h), a1 = __ldg(l1 + h), a2 = __ldg(l2 + h), a3 = __ldg(l3 + h);
        const ulonglong2 ww = __ldg(wv + h);
        const u64 sx = a0.x + a1.x + a2.x + a3.x, sy = a0.y + a1.y + a2.y + a3.y;
        u128_add(T[2 * h], sx * ww.x, __umul64hi(sx, ww.x));
        u128_add(T[2 * h + 1], sy * ww.y, __umul64hi(sy, ww.y));
      }
    }
    // thread-pattern masses (scale 2^124 after this), then the reduce-scatter
#pragma unroll
    for (int kk = 0; kk < BSB_KC; ++kk) {
      const u64 tw = (thr_on && kk < kc) ? __ldg(thg + k0 + kk) : 0ull;
      T[kk] = mul64x128_shr64(tw, T[kk].lo, T[kk].hi);
    }
#pragma unroll
    for (int st2 = 0; st2 < 4; ++st2) {
      const int o = 16 >> st2, n = 8 >> st2;
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < n; ++i) {
        const u128 send = up ? T[i] : T[i + n];
        const u128 keep = up ? T[i + n] : T[i];
        const u128 got = shfl_xor_u128(send, o);
        T[i] = keep;
        u128_add(T[i], got.lo, got.hi);
      }
    }
    {
      const u128 got = shfl_xor_u128(T[0], 1);
      u128_add(T[0], got.lo, got.hi);
    }
    if (!(lane & 1) && idx < kc) {
      const mx w = BSB_MERGE ? bs_class_mass(A.cmass + 2 * (cls * K + k0 + idx), 0)
          : bsb_prefix_mass(gpt + (size_t)(k0 + idx) * pt_size, nlev, lev_bits, lev_off, prefix);
      bsb_limb_add(glimbs + (size_t)(k0 + idx) * BSB_LIMBS, mx_prod(w, T[0]), w.e);
    }
  }
}
// ---------------------------------------------------------------------------
// Batched fused R + N_k + dR/dp (the gradient module): the item's
// connectivity words (cw, one per walk state) and their 32x32 lane
// transposes (ctw) are formed once; then for each p-vector in turn the
// per-arc sums of the single-network fused kernel are built from them --
// exact integer pair differences for lane and thread arcs, the parts A and
// T - A of the walk arcs (128-bit walk masses), item totals times the
// prefix mass without the arc for prefix arcs -- and added to that
// (network, p-vector)'s 256-bit results: R, then A_k and B_k of every
// internal arc k.  Prefix arcs take the item's whole prefix mass (the host
// divides their sums by p and 1 - p) unless some p-vector puts their p
// outside [2^-20, 1 - 2^-20] (bit set in pex_mask).
// ---------------------------------------------------------------------------
__device__ __forceinline__ mx bsb_ex_factor(const mx* __restrict__ tk, const mx* __restrict__ exk,
                                            int nlev, const int (&lev_bits)[8], const int (&lev_off)[8],
                                            u64 prefix, int j) {
  // prefix mass without prefix arc j: its level's entry from the excluded
  // table (rows of 128), the other levels from the plain table
  mx f = mx{1ull << 63, 0, 0};
  int sh = 0;
#pragma unroll
  for (int l = 0; l < 8; ++l) {
    if (l >= nlev) break;
    const u64 v = (prefix >> sh) & ((1ull << lev_bits[l]) - 1ull);
    const bool mine = j >= sh && j < sh + lev_bits[l];
    const ulonglong2 q = __ldg((const ulonglong2*)(mine ? exk + ((size_t)j << 7) + v : tk + lev_off[l] + v));
    const mx t = mx{q.x, (int)(u32)q.y, 0};
    f = l ? mx_mul(f, t) : t;
    sh += lev_bits[l];
  }
  return f;
}

__device__ __forceinline__ void bsb_finish_grad(
    const BGraph* __restrict__ Bp, int st, u64 prefix, int lane, int K, int Kp,
    const u64* __restrict__ lt, const u64* __restrict__ nt, const u64* __restrict__ wm2,
    const mx* __restrict__ pt, const u64* __restrict__ thw, const u64* __restrict__ tt,
    const u64* __restrict__ lwex, const u64* __restrict__ thwex, const mx* __restrict__ ptex,
    u64* limbs, u64* nkw, u64* bins, const u32* cw, u32* ctw, const BsTr& tr, const BMerge& A, u64 cls, u32* rel) {
  constexpr int nsh[6] = BS_NK_SHIFTS, nwd[6] = BS_NK_WIDTHS;
  const int L = Bp->L, tb = Bp->tb, ell = Bp->ell, top = Bp->top, m = Bp->m, nlev = Bp->nlev;
  const int pt_size = Bp->pt_size, d = Bp->d;
  const u32 lane_mask = Bp->lane_mask, thr_mask = Bp->thr_mask;
  int lev_bits[8], lev_off[8];
#pragma unroll
  for (int l = 0; l < 8; ++l) {
    lev_bits[l] = Bp->lev_bits[l];
    lev_off[l] = Bp->lev_off[l];
  }
  const int pc_pre = __popcll((long long)prefix);
  const bool thr_on = lane < (1 << tb);
  const int nw = 1 << L;
  // ---- N_k, as in the R module
  if (st == 1) {
    for (int j = lane; j <= top; j += 32) nkw[pc_pre + j] += __ldg(&Bp->binom[j]);
  } else {
    for (int r = 0; r <= L; ++r) bins[r * BSB_NTHR] = 0ull;
    const u64* ntg = nt + Bp->nt_off;
    for (int g = 0; g < nw; ++g) {
      const u32 c = cw[g * BSB_NTHR];
      if (!c) continue;
      bins[__popc(g) * BSB_NTHR] += c == lane_mask ? Bp->full_counts
          : __ldg(ntg + (c & 0xffu)) + __ldg(ntg + 256 + ((c >> 8) & 0xffu)) +
            __ldg(ntg + 512 + ((c >> 16) & 0xffu)) + __ldg(ntg + 768 + (c >> 24));
    }
    u64 c11[11];
#pragma unroll
    for (int i = 0; i < 11; ++i) c11[i] = 0ull;
#pragma unroll
    for (int r = 0; r <= 5; ++r) {
      if (r > L) break;
      const u64 n = bins[r * BSB_NTHR];
#pragma unroll
      for (int cl = 0; cl < 6; ++cl) c11[r + cl] += (n >> nsh[cl]) & ((1ull << nwd[cl]) - 1ull);
    }
    BSB_COUNTS();
    // ---- the lane transposes, once per word: lane j then holds the
    // threads' bits of lane pattern j (lanes past the thread patterns hold
    // no thread's states); zero when no lane's word is partly connected
    for (int g = 0; g < nw; ++g) {
      const u32 c = thr_on ? cw[g * BSB_NTHR] : 0u;
      const bool mixed = __any_sync(0xffffffffu, c != 0u && c != lane_mask);
      const u32 ct = mixed ? bs_transpose32(c, tr) : 0u;
      ctw[g * BSB_NTHR] = lane < (1 << ell) ? ct : 0u;
    }
  }
  const int stride = 1 + 2 * m;
  u64* gl = limbs + Bp->out_off;
  const u64* ltg = lt + Bp->lt_off;
  const u64* ttg = tt + Bp->tt_off;
  const ulonglong2* wmg = (const ulonglong2*)(wm2 + Bp->wm2_off);
  for (int k = 0; k < K; ++k) {
    u128 S = u128{0ull, 1ull << 60};   // a fully connected item: mass 1 at scale 2^124
    u128 myX = u128{0ull, 0ull}, myY = u128{0ull, 0ull};
    if (st == 2) {
      u128 T = u128{0ull, 0ull}, T2 = u128{0ull, 0ull};
      u128 Aw[5];
#pragma unroll
      for (int b = 0; b < 5; ++b) Aw[b] = u128{0ull, 0ull};
      for (int g = 0; g < nw; ++g) {
        const u32 c = cw[g * BSB_NTHR], ct = ctw[g * BSB_NTHR];
        if (!(c | ct)) continue;
        const ulonglong2 wv = __ldg(wmg + (size_t)g * Kp + k);
        const u128 full = u128{(wv.x >> 2) | (wv.y << 62), wv.y >> 2};   // scale 2^125
        if (c) {
          u128 x = full;
          if (c != lane_mask) {
            const u64 sR = __ldg(ltg + (size_t)(c & 0xffu) * Kp + k) +
                           __ldg(ltg + (size_t)(256 + ((c >> 8) & 0xffu)) * Kp + k) +
                           __ldg(ltg + (size_t)(512 + ((c >> 16) & 0xffu)) * Kp + k) +
                           __ldg(ltg + (size_t)(768 + (c >> 24)) * Kp + k);
            x = mul64x128_shr64(sR, wv.x, wv.y);
          }
          u128_add(T, x.lo, x.hi);
#pragma unroll
          for (int b = 0; b < 5; ++b)
            if (b < L && ((g >> b) & 1)) u128_add(Aw[b], x.lo, x.hi);
        }
        if (ct) {
          u128 y = full;
          if (ct != thr_mask) {
            const u64 s2 = __ldg(ttg + (size_t)(ct & 0xffu) * Kp + k) +
                           __ldg(ttg + (size_t)(256 + ((ct >> 8) & 0xffu)) * Kp + k) +
                           __ldg(ttg + (size_t)(512 + ((ct >> 16) & 0xffu)) * Kp + k) +
                           __ldg(ttg + (size_t)(768 + (ct >> 24)) * Kp + k);
            y = mul64x128_shr64(s2, wv.x, wv.y);
          }
          u128_add(T2, y.lo, y.hi);
        }
      }
      // exact warp sums (scale 2^124); lane k ends with internal arc k's
      const u64 thwk = thr_on ? __ldg(thw + Bp->thw_off + (size_t)lane * Kp + k) : 0ull;
      S = warp_sum_u128(mul64x128_shr64(thwk, T.lo, T.hi));
      for (int i = 0; i < ell; ++i) {
        const u128 o = shfl_xor_u128(T2, 1 << i);
        const u128 d2 = u128_sub(T2, o);
        const u64 w = ((lane >> i) & 1) && lane < (1 << ell)
                          ? __ldg(lwex + Bp->lwex_off + ((size_t)(i * 32 + lane)) * Kp + k) : 0ull;
        const u128 sv = warp_sum_u128(mul64x128_shr64(w, d2.lo, d2.hi));
        if (lane == i) myX = sv;
      }
      for (int i = 0; i < tb; ++i) {
        const u128 o = shfl_xor_u128(T, 1 << i);
        const u128 d1 = u128_sub(T, o);
        const u64 w = ((lane >> i) & 1) && thr_on
                          ? __ldg(thwex + Bp->thwex_off + ((size_t)(i * 32 + lane)) * Kp + k) : 0ull;
        const u128 sv = warp_sum_u128(mul64x128_shr64(w, d1.lo, d1.hi));
        if (lane == ell + i) myX = sv;
      }
#pragma unroll
      for (int b = 0; b < 5; ++b) {
        if (b >= L) break;
        const u128 sa = warp_sum_u128(mul64x128_shr64(thwk, Aw[b].lo, Aw[b].hi));
        const u128 sz = u128_sub(S, sa);   // the failed half, as in the fused kernel
        if (lane == ell + tb + b) { myX = sa; myY = sz; }
      }
    }
    // ---- prefix factors of p-vector k and the additions to its results
    const mx* tk = pt + Bp->pt_off + (size_t)k * pt_size;
    const mx wpre = BSB_MERGE ? bs_class_mass(A.cmass + 2 * (cls * K + k), 0)
                              : bsb_prefix_mass(tk, nlev, lev_bits, lev_off, prefix);
    u64* out = gl + (size_t)k * stride * BSB_LIMBS;
    if (lane == 0) bsb_limb_add(out, mx_prod(wpre, S), wpre.e);
#if BSB_MERGE
    // a class's prefix arcs are left to bs_batch_grad_p3, from its sum S
    if (lane == 0) A.csum[cls * K + k] = make_ulonglong2(S.lo, S.hi);
    if (lane < top) {
      bsb_limb_add(out + (1 + 2 * lane) * BSB_LIMBS, mx_prod(wpre, myX), wpre.e);
      bsb_limb_add(out + (2 + 2 * lane) * BSB_LIMBS, mx_prod(wpre, myY), wpre.e);
    }
#else
    const mx* exk = ptex + Bp->ptex_off + ((size_t)k * d << 7);
    if (lane < m) {
      u128 X = u128{0ull, 0ull}, Y = u128{0ull, 0ull};
      mx f = wpre;
      if (lane >= top) {
        // a prefix arc: the item's total, into A when the arc works in this
        // item and into B when it fails -- with the whole prefix mass (the
        // host divides by p and 1 - p), or for an arc whose p is outside
        // [2^-20, 1 - 2^-20] under some p-vector, without its own factor
        if ((Bp->pex_mask >> lane) & 1ull)
          f = bsb_ex_factor(tk, exk, nlev, lev_bits, lev_off, prefix, lane - top);
        if ((prefix >> (lane - top)) & 1ull) X = S; else Y = S;
      } else if (st == 2) {
        X = myX;
        Y = myY;
      }
      bsb_limb_add(out + (1 + 2 * lane) * BSB_LIMBS, mx_prod(f, X), f.e);
      bsb_limb_add(out + (2 + 2 * lane) * BSB_LIMBS, mx_prod(f, Y), f.e);
    }
    if (lane + 32 < m) {
      const int j = lane + 32 - top;
      const mx f = ((Bp->pex_mask >> (lane + 32)) & 1ull)
                       ? bsb_ex_factor(tk, exk, nlev, lev_bits, lev_off, prefix, j) : wpre;
      const bool on = (prefix >> j) & 1ull;
      bsb_limb_add(out + ((on ? 1 : 2) + 2 * (lane + 32)) * BSB_LIMBS, mx_prod(f, S), f.e);
    }
#endif
  }
}
#if BSB_MERGE
// ---------------------------------------------------------------------------
// Merged batches: as the single networks' merged runs (bs_merge_body), for
// every network and p-vector at once.
//   bs_batch*_p1  prunes every network's items, 32 x 32 at a time, sums those
//                 connected throughout, and interns the signatures of the others
//   bs_batch*_p2  adds each item's masses and popcount to its class
//   bs_batch*     walks one item of every class (bsb_conn, bsb_finish)
//   bs_batch*_p3  (gradient) folds the prefix arcs, per block and p-vector
// GB300, against a walk for every item left: 64 networks (2.9e10 states) x 16
// p-vectors, R 5.42 -> 0.43 ms, with the gradient 24.1 -> 1.89 ms.  The walking launch is bound by instruction issue and the table
// rows it reads through L1, the others by the latency of the table and the
// class memory, hence the several warps per block of items.
// ---------------------------------------------------------------------------
#define BSB_MNTHR 128
// The per-network part of a block: which of its items are connected
// throughout and which are left to walk, and the latter's signatures, one
// word per bit and lane, in zs.
template <class G>
__device__ __noinline__ void bsb_classify(u64 hi, int lane, u32* zs, u32& full, u32& left) {
  constexpr int BLK = G::LOW + G::MID;
  u32 a[G::M], z[G::NSIG > 0 ? G::NSIG : 1], dn, up;
#pragma unroll
  for (int j = 0; j < G::D; ++j)
    a[G::TOP + j] = j < G::LOW ? bs_pattern(j) : j < BLK ? 0u - (u32)((lane >> (j - G::LOW)) & 1)
                                                          : 0u - (u32)((hi >> (j - BLK)) & 1ull);
  G::sig(a, z, dn, up);
  const u32 valid = lane < (1 << G::MID) ? (G::LOW >= 5 ? 0xffffffffu : (1u << (1 << G::LOW)) - 1u) : 0u;
  full = dn & valid;
  left = up & valid & ~full;
#pragma unroll
  for (int i = 0; i < G::NSIG; ++i) zs[i * 32 + lane] = z[i];
}
__device__ __forceinline__ int bsb_block_net(const BGraph* __restrict__ graphs, int G, u64 t) {
  int lo = 0, hi = G - 1;
  while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (graphs[mid].blk_begin <= t) lo = mid; else hi = mid - 1; }
  return lo;
}
// mass of the arcs above a block (the levels of a merged batch's table)
__device__ __forceinline__ mx bsb_hi_mass(const BGraph* __restrict__ B, const mx* __restrict__ pt, int k, u64 hi) {
  return bs_level_mass(B->nlev, B->lev_bits, B->lev_off, pt + B->pt_off + (size_t)k * B->pt_size, hi);
}
// What bsb_merge does with a block once its network's part is done.
__device__ __forceinline__ void bsb_merge_block(const BGraph* __restrict__ B, int net, u64 t, u64 hi, int part, int lane, int K,
                                                const u32* zs, u32 full, u32 left, const mx* __restrict__ pt,
                                                const BMerge& A, u64* limbs, u64* nk, u32* status) {
  const int low = B->low, mid = B->mid, blk = low + mid, top = B->top, nsig = B->nsig;
  const int pc_hi = __popcll((long long)hi);
  if (part == 0) A.cmask[t * 32 + lane] = make_uint2(full, left);
  if (__any_sync(0xffffffffu, full)) {
    if (part == 0) {
      // lane q: states with pc_hi + q working arcs, over the items' popcounts
      const u32 n = bs_block_counts(full, lane);
      u64 s = 0;
      for (int i = 0; i <= blk; ++i) {
        const u64 c = __shfl_sync(0xffffffffu, n, i);
        if (lane >= i && lane - i <= top) s += c * __ldg(&B->binom[lane - i]);
      }
      if (s) atomicAdd(&nk[B->nk_off + pc_hi + lane], s);
    }
    for (int k = part; k < K; k += 1 << A.split_log2) {
      const size_t gk = (size_t)net * K + k;
      const ulonglong2 mm = __ldg(&A.mid[gk * 32 + lane]);
      const u128 S = warp_sum_u128(u128_shr(bs_subset_mass(full, A.nib + gk * 128, u128{mm.x, mm.y}), 2));
      if (lane == 0) {
        const mx w = bsb_hi_mass(B, pt, k, hi);
        bsb_limb_add(limbs + B->out_off + (size_t)k * (BSB_GRAD ? 1 + 2 * B->m : 1) * BSB_LIMBS, mx_prod(w, S), w.e);
      }
    }
  }
  left &= bs_part_mask(A.split_log2, part);
  while (left) {
    const int j = __ffs(left) - 1;
    u32 k0 = 0u, k1 = 0u, same = left;
    for (int i = 0; i < nsig; ++i) {
      const u32 z = zs[i * 32 + lane], b = z << (31 - j);   // item j's bit on top
      if (i < 32) k0 = __funnelshift_l(b, k0, 1); else k1 = __funnelshift_l(b, k1, 1);
      same &= ~(z ^ (u32)((int)b >> 31));
    }
    left &= ~same;
    bool fresh;
    const u32 at = bs_class(A.key + B->slot_base, B->slots_log2, nsig, ((u64)k1 << 32) | k0 | 1ull << 63, fresh);
    if (at == ~0u) { atomicOr(status, 2u); continue; }   // the host walks the items one by one instead
    const u32 slot = (u32)B->slot_base + at;
    if (fresh) {
      const u64 id = atomicAdd(A.n_classes, 1ull);
      if (id < A.cap) {
        A.id_of[slot] = (u32)id;
        A.net[id] = (u32)net;
        A.rep[id] = (hi << blk) | (u64)(lane << low) | (u64)j;
        for (int i = 0; i < A.hist_stride; ++i) A.hist[id * A.hist_stride + i] = 0u;
        for (int i = 0; i < 2 * K; ++i) A.cmass[2 * id * K + i] = 0ull;
      } else {
        atomicOr(status, 2u);
      }
    }
    uint2* e = A.ent + B->item_base + (hi << blk) + lane;
    for (u32 s = same; s; s &= s - 1u) {
      const int i = __ffs(s) - 1;
      e[i << mid] = make_uint2(slot, i == j ? same : 0u);
    }
  }
}
extern "C" __global__ void __launch_bounds__(BSB_MNTHR) BSB_SCATTER(
    const BGraph* __restrict__ graphs, int G, int K, const mx* __restrict__ pt, const BMerge A, u32* status,
    u64 budget_ns) {
  __shared__ mx s_hi[BSB_MNTHR / 32][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (bs_warp_given_up(status, lane)) return;
  for (u64 v = (u64)blockIdx.x * (BSB_MNTHR / 32) + warp; v < A.n_blocks * A.parts; v += (u64)gridDim.x * (BSB_MNTHR / 32)) {
    if (budget_ns && bs_time_up(budget_ns, A.start, status, lane)) break;
    const u64 t = v / A.parts;
    const int part = (int)(v - t * A.parts);
    u32 left = A.cmask[t * 32 + lane].y;
    if (!__any_sync(0xffffffffu, left)) continue;
    const int net = bsb_block_net(graphs, G, t);
    const BGraph* __restrict__ B = graphs + net;
    const u64 hi = t - B->blk_begin;
    const int mid = B->mid, blk = B->low + mid, pc = __popcll((long long)hi) + __popc(lane);
    __syncwarp();
    for (int k = part + lane * A.parts; k < K; k += 32 * A.parts) s_hi[warp][k] = bsb_hi_mass(B, pt, k, hi);
    __syncwarp();
    uint2* e = A.ent + B->item_base + (hi << blk) + lane;
    while (left) {
      const int j = __ffs(left) - 1;
      const uint2 x = e[j << mid];
      left &= ~x.y;   // the first item of its class in the lane has them all
      const u32 id = A.id_of[x.x];
      if (part == 0) bs_add_counts(A.hist + (size_t)id * A.hist_stride, x.y, pc);
      for (int k = part; k < K; k += A.parts) {
        const size_t gk = (size_t)net * K + k;
        const ulonglong2 mm = __ldg(&A.mid[gk * 32 + lane]);
        bs_add_mass(A.cmass + 2 * ((size_t)id * K + k), s_hi[warp][k],
                    u128_shr(bs_subset_mass(x.y, A.nib + gk * 128, u128{mm.x, mm.y}), 2), 0);
      }
    }
  }
}
#if BSB_GRAD
extern "C" __global__ void __launch_bounds__(BSB_MNTHR) bs_batch_grad_p3(
    const BGraph* __restrict__ graphs, int G, int K, const mx* __restrict__ pt, const BMerge A, u64* limbs,
    u32* status, u64 budget_ns) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (bs_warp_given_up(status, lane)) return;
  for (u64 t = (u64)blockIdx.x * (BSB_MNTHR / 32) + warp; t < A.n_blocks * K; t += (u64)gridDim.x * (BSB_MNTHR / 32)) {
    if (budget_ns && bs_time_up(budget_ns, A.start, status, lane)) break;
    const u64 b = t / K;
    const int k = (int)(t - b * K);
    const uint2 m = A.cmask[b * 32 + lane];
    if (!__any_sync(0xffffffffu, m.x | m.y)) continue;
    const int net = bsb_block_net(graphs, G, b);
    const BGraph* __restrict__ B = graphs + net;
    const u64 hi = b - B->blk_begin;
    const int low = B->low, mid = B->mid, blk = low + mid, nhi = B->nhi, top = B->top;
    const u64* __restrict__ f = A.fold + ((size_t)net * K + k) * 104;   // laid out as BsFoldParams
    const uint2* e = A.ent + B->item_base + (hi << blk) + lane;
    u128 Gs[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) Gs[i] = u128{0ull, 0ull};
    u128 V = bs_fold_low(f, f + 10, Gs, [&](int j) {
      u128 v = u128{0ull, (m.x >> j) & 1u ? 1ull << 60 : 0ull};
      if ((m.y >> j) & 1u) {
        const ulonglong2 s = A.csum[(size_t)A.id_of[e[j << mid].x] * K + k];
        v = u128{s.x, s.y};
      }
      return v;
    });
    u128 X;
    V = bs_fold_mid<0>(V, Gs, low, mid, f + 5, f + 41, f[72 + lane], lane, X);
    const mx w = bsb_hi_mass(B, pt, k, hi);
    u64* out = limbs + B->out_off + (size_t)k * (1 + 2 * B->m) * BSB_LIMBS;
    if (lane < blk) bsb_limb_add(out + (1 + 2 * (top + lane)) * BSB_LIMBS, mx_prod(w, X), w.e);
    const u128 Sv = mx_prod(w, V);
    for (int q = lane; q < nhi; q += 32)
      bsb_limb_add(out + (((hi >> q) & 1ull ? 1 : 2) + 2 * (top + blk + q)) * BSB_LIMBS, Sv, w.e);
  }
}
#endif
#endif
//@@BATCH_KERNEL@@
)PBAT";
}  // namespace pbat
