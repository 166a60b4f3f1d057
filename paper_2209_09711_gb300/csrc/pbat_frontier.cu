// pbat_frontier.cu -- the per-state PBAT kernel and the final reduction.
//
// Work decomposition (equal division, arXiv 2209.09711 Sec. 4.3, Eq. 6-7):
// the top `prefix_bits` arcs of the state word form a prefix; each prefix
// value is one work item, taken by one warp from an atomic ticket.  Inside
// an item, lane j fixes the `lane_bits` lowest arcs to the pattern j and
// walks the `walk_bits` middle arcs in reflected Gray-code order, so every
// step changes exactly one arc (the BAT of Sec. 3.1 visits the same set of
// vectors in binary order; only the set matters for Eq. 1).
//
// Per state, connectivity is the PLSA of Sec. 3.2 done as frontier
// expansion on node bitmasks: adj[u] (one word per node, per thread, in
// shared memory) holds u's working out-neighbours; the frontier pops its
// lowest node with ffs, adds adj[u] minus the visited set, and stops when the
// sink appears or the frontier empties.  Monotonicity skips the search when
// the flipped arc cannot change the answer (an arc added to a connected
// state, or removed from a disconnected one).
//
// Accumulation is exact: the walk-arc mass of every walk pattern g is a
// 128-bit fixed-point table entry W[g] ~ 2^127 * prod_{walk arcs} w(g), and a
// thread adds W[g] for each connected state into a 128-bit integer T.  The
// prefix and lane factors are applied once per item in double-double.  N_k
// is a per-thread histogram by the popcount of g.  The gradient of Eq. 1
// (PBAT differentiated term by term) needs, for every walk arc b, the mass
// A_b of connected states with that arc working; Gray order makes this one
// update per step: when arc b turns on, remember T; when it turns off, add
// the growth of T since then.  Being integer, these differences are exact.
//
// Exact monotone prune per item: with every free (lane + walk) arc working
// the sink is unreachable -> the whole item contributes nothing; with every
// free arc failed it is reachable -> the item adds its closed-form mass
// Pr(prefix), C(f, j) states with |prefix| + j working arcs, and gradient
// terms for the prefix arcs only (free arcs have zero derivative there).
#include <cuda_runtime.h>

#include "pbat_internal.h"

namespace pbat {

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

template <typename M>
__device__ __forceinline__ int lowest_node(M x);
template <>
__device__ __forceinline__ int lowest_node<uint32_t>(uint32_t x) {
  return __ffs(x) - 1;
}
template <>
__device__ __forceinline__ int lowest_node<unsigned long long>(unsigned long long x) {
  return __ffsll((long long)x) - 1;
}

// Frontier expansion (PLSA, Sec. 3.2) on this thread's adjacency rows.
template <typename M>
__device__ __forceinline__ bool sink_reached(const M* adj, int stride, M sbit, M tbit) {
  M vis = sbit, fr = sbit;
  while (fr) {
    const int u = lowest_node<M>(fr);
    fr &= fr - 1;
    const M nb = adj[u * stride] & ~vis;
    if (nb & tbit) return true;
    vis |= nb;
    fr |= nb;
  }
  return false;
}

// Reachability of one arbitrary state, computed identically by every lane
// (used twice per work item by the prune).  Repeated passes over the arc
// list until nothing changes.
__device__ __noinline__ bool state_connected(const FrontierParams& P, unsigned long long x) {
  unsigned long long reach = 1ull << P.source;
  const unsigned long long tb = 1ull << P.sink;
  for (int pass = 0; pass < P.n; ++pass) {
    const unsigned long long before = reach;
    for (int k = 0; k < P.m; ++k) {
      if (!((x >> k) & 1ull)) continue;
      const unsigned long long bu = 1ull << P.au[k], bv = 1ull << P.av[k];
      if (reach & bu) reach |= bv;
      if (!P.directed && (reach & bv)) reach |= bu;
    }
    if (reach & tb) return true;
    if (reach == before) return false;
  }
  return (reach & tb) != 0;
}

// Exact sum over the warp (every lane gets it) of values below 2^127: five
// chunks of at most 26 bits, whose 32-lane sums fit 31 bits, one hardware
// warp reduction each (the top chunk holds 23 bits).
__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
  const uint32_t c0 = (uint32_t)(v.lo & 0x3ffffffull), c1 = (uint32_t)((v.lo >> 26) & 0x3ffffffull);
  const uint32_t c2 = (uint32_t)(((v.lo >> 52) | (v.hi << 12)) & 0x3ffffffull);
  const uint32_t c3 = (uint32_t)((v.hi >> 14) & 0x3ffffffull), c4 = (uint32_t)(v.hi >> 40);
  const unsigned long long s0 = __reduce_add_sync(0xffffffffu, c0), s1 = __reduce_add_sync(0xffffffffu, c1);
  const unsigned long long s2 = __reduce_add_sync(0xffffffffu, c2), s3 = __reduce_add_sync(0xffffffffu, c3);
  const unsigned long long s4 = __reduce_add_sync(0xffffffffu, c4);
  u128 r = u128{s0, 0ull};
  u128_add_to(r, u128{s1 << 26, 0ull});
  u128_add_to(r, u128{s2 << 52, s2 >> 12});
  u128_add_to(r, u128{0ull, s3 << 14});
  u128_add_to(r, u128{0ull, s4 << 40});
  return r;
}
// (a * b) >> 128, at most two units low (the product of the low halves dropped)
__device__ __forceinline__ u128 mulhi128(u128 a, u128 b) {
  u128 r = u128{a.hi * b.hi, __umul64hi(a.hi, b.hi)};
  u128_add_to(r, u128{__umul64hi(a.hi, b.lo), 0ull});
  u128_add_to(r, u128{__umul64hi(a.lo, b.hi), 0ull});
  return r;
}
// Sum over the warp of T (scale 2^127) times a lane's mass: the sum is
// returned times 2^*e.  Each product keeps 126 significant bits and is shifted
// to the largest one's exponent, so the sum is good to 2^-115 of itself
// however small the masses are.
__device__ __forceinline__ u128 warp_sum_scaled(u128 T, const LaneMass& w, int* e) {
  const int lz = T.hi ? __clzll((long long)T.hi) : 64 + __clzll((long long)T.lo);
  const bool some = (T.lo | T.hi) && (w.m.lo | w.m.hi);
  u128 n = T;   // T << lz
  if (lz >= 64) n = u128{0ull, n.lo};
  const int r = lz & 63;
  if (r) n = u128{n.lo << r, (n.hi << r) | (n.lo >> (64 - r))};
  const u128 p = mulhi128(n, w.m);   // below 2^127: the product is p 2^(-126 - E)
  const int E = some ? lz + w.e : 1 << 20;
  const int lo = (int)__reduce_min_sync(0xffffffffu, (unsigned)(E + (1 << 16))) - (1 << 16);
  const int sh = some ? E - lo + 5 : 128;
  u128 q = u128_zero();
  if (sh < 64) q = u128{(p.lo >> sh) | (p.hi << (64 - sh)), p.hi >> sh};
  else if (sh < 128) q = u128{p.hi >> (sh - 64), 0ull};
  *e = lo >= (1 << 19) ? 0 : 5 - 126 - lo;
  return warp_sum_u128(q);
}

__device__ __forceinline__ dd shfl_dd(dd v, int src) {
  return dd{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}
// Mass of the prefix arcs of `prefix` (every lane), and with EX for lane j's
// prefix arc (j < 32, and j + 32) the mass without it: products over the
// lanes, one factor each, by shuffles -- FP64 runs at 1/64 of the FP32 rate
// here, and a product over the arcs in turn, in every lane, was half of an
// item's FP64 work.
template <bool EX>
__device__ __forceinline__ dd prefix_mass(const FrontierParams& P, unsigned long long prefix, int lane, dd* ex) {
  const int base = P.lane_bits + P.walk_bits, d = P.prefix_bits;
  dd whole = dd{1.0, 0.0}, ex0 = whole, ex1 = whole;
  for (int j0 = 0; j0 < d; j0 += 32) {
    const int j = j0 + lane;
    dd f = dd{1.0, 0.0};
    if (j < d) f = ((prefix >> j) & 1ull) ? dd{P.p[base + j], 0.0} : P.q[base + j];
    // up: the product of this lane's factor and those below it (with EX);
    // all: of every lane's factor
    dd all = f;
    if (EX) {
      dd up = f, dn = f;
      for (int o = 1; o < 32 && o < d - j0; o <<= 1) {
        const dd a = dd{__shfl_up_sync(0xffffffffu, up.hi, o), __shfl_up_sync(0xffffffffu, up.lo, o)};
        const dd b = dd{__shfl_down_sync(0xffffffffu, dn.hi, o), __shfl_down_sync(0xffffffffu, dn.lo, o)};
        if (lane >= o) up = dd_mul(up, a);
        if (lane + o < 32) dn = dd_mul(dn, b);
      }
      all = shfl_dd(dn, 0);
      dd below = dd{__shfl_up_sync(0xffffffffu, up.hi, 1), __shfl_up_sync(0xffffffffu, up.lo, 1)};
      dd above = dd{__shfl_down_sync(0xffffffffu, dn.hi, 1), __shfl_down_sync(0xffffffffu, dn.lo, 1)};
      if (lane == 0) below = dd{1.0, 0.0};
      if (lane == 31) above = dd{1.0, 0.0};
      const dd x = dd_mul(below, above);
      if (j0 == 0) ex0 = x; else ex1 = dd_mul(x, whole);
    } else {
      for (int o = 16; o > 0; o >>= 1) {
        if (o >= d - j0 && o > 1) continue;   // only ones up there
        all = dd_mul(all, dd{__shfl_xor_sync(0xffffffffu, all.hi, o), __shfl_xor_sync(0xffffffffu, all.lo, o)});
      }
      all = shfl_dd(all, 0);
    }
    if (j0 > 0 && EX) ex0 = dd_mul(ex0, all);
    whole = dd_mul(whole, all);
  }
  if (EX) {
    ex[0] = ex0;
    ex[1] = ex1;
  }
  return whole;
}

__device__ __forceinline__ void acc_signed(dd& slot, dd v, bool plus) {
  slot = plus ? dd_add(slot, v) : dd_sub(slot, v);
}

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

template <typename M, bool GRAD>
__global__ void __launch_bounds__(256) frontier_kernel(const __grid_constant__ FrontierParams P,
                                                       const u128* __restrict__ wmid_g,
                                                       DevWork W) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = P.walk_bits, ell = P.lane_bits, n = P.n, m = P.m;
  const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = nthr >> 5;
  const int nW = 1 << L;

  size_t off = 0;
  u128* s_wmid = reinterpret_cast<u128*>(smem + off);
  off = align16(off + (size_t)nW * sizeof(u128));
  M* s_adj = reinterpret_cast<M*>(smem + off);
  off = align16(off + (size_t)n * nthr * sizeof(M));
  uint32_t* s_ncnt = reinterpret_cast<uint32_t*>(smem + off);
  off = align16(off + (size_t)(L + 1) * nthr * sizeof(uint32_t));
  u128* s_seg = reinterpret_cast<u128*>(smem + off);
  if (GRAD) off = align16(off + (size_t)2 * L * nthr * sizeof(u128));
  dd* s_wacc = reinterpret_cast<dd*>(smem + off);
  off = align16(off + (size_t)nwarps * (1 + m) * sizeof(dd));
  unsigned long long* s_nbins = reinterpret_cast<unsigned long long*>(smem + off);
  if (GRAD) off = align16(off + (size_t)(m + 1) * sizeof(unsigned long long));
  // lane masses without each lane arc (from the parameters where they have no room here)
  LaneMass* s_lwx = reinterpret_cast<LaneMass*>(smem + off);

  if (GRAD && P.lane_tab)
    for (int i = tid; i < ell * 32; i += nthr) s_lwx[i] = P.lane_w_ex[i >> 5][i & 31];
  for (int i = tid; i < nW; i += nthr) s_wmid[i] = wmid_g[i];
  for (int i = tid; i < nwarps * (1 + m); i += nthr) s_wacc[i] = dd{0.0, 0.0};
  for (int i = tid; i <= m; i += nthr) s_nbins[i] = 0ull;
  __syncthreads();

  M* adj = s_adj + tid;
  uint32_t* ncnt = s_ncnt + tid;
  u128* seg_start = s_seg + tid;
  u128* seg_acc = s_seg + (size_t)L * nthr + tid;
  dd* wacc = s_wacc + (size_t)warp * (1 + m);
  const M sbit = (M)1 << P.source, tbit = (M)1 << P.sink;
  const bool lane_on = lane < (1 << ell);
  const LaneMass lw = P.lane_w[lane];   // zero past the lane patterns
  const int top = ell + L;  // first prefix arc
  const unsigned long long t_start = globaltimer_ns();
  unsigned long long n_walk = 0, n_full = 0, n_dead = 0;

  for (;;) {
    unsigned long long task = 0;
    if (lane == 0) {
      task = atomicAdd(W.counter, 1ull);
      if (P.budget_ns && globaltimer_ns() - t_start > P.budget_ns) {
        atomicOr(W.status, 1u);
        task = ~0ull;
      }
    }
    task = __shfl_sync(0xffffffffu, task, 0);
    if (task >= P.n_tasks) break;
    const unsigned long long prefix = P.task_lo + task;
    const unsigned long long xpre = top < 64 ? (prefix << top) : 0ull;
    const int pc_pre = __popcll((long long)prefix);

    if (P.prune) {
      if (!state_connected(P, xpre | P.free_mask)) {
        ++n_dead;
        continue;
      }
      if (state_connected(P, xpre)) {
        ++n_full;
        for (int j = lane; j <= top; j += 32) atomicAdd(&s_nbins[pc_pre + j], P.binom[j]);
        dd ex[2];
        const dd wpre = prefix_mass<GRAD>(P, prefix, lane, ex);
        if (lane == 0) wacc[0] = dd_add(wacc[0], wpre);
        if (GRAD) {
          for (int j = lane; j < P.prefix_bits; j += 32)
            acc_signed(wacc[1 + top + j], j < 32 ? ex[0] : ex[1], (prefix >> j) & 1ull);
        }
        continue;
      }
    }
    ++n_walk;

    // ---- Gray walk of the middle arcs, one state per step
    unsigned long long x = xpre | (unsigned long long)(lane_on ? lane : 0);
    for (int u = 0; u < n; ++u) adj[u * nthr] = (M)0;
    for (int k = 0; k < m; ++k) {
      if ((x >> k) & 1ull) {
        adj[P.au[k] * nthr] |= (M)1 << P.av[k];
        if (!P.directed) adj[P.av[k] * nthr] |= (M)1 << P.au[k];
      }
    }
    bool conn = sink_reached<M>(adj, nthr, sbit, tbit);
    u128 T = u128_zero();
    for (int c = 0; c <= L; ++c) ncnt[c * nthr] = 0u;
    if (GRAD) {
      for (int b = 0; b < L; ++b) {
        seg_start[b * nthr] = u128_zero();
        seg_acc[b * nthr] = u128_zero();
      }
    }
    if (conn) {
      u128_add_to(T, s_wmid[0]);
      ncnt[0] += 1u;
    }
    uint32_t g = 0;
    int pc = 0;
    for (uint32_t s = 1; s < (uint32_t)nW; ++s) {
      const int b = __ffs(s) - 1;
      const int k = ell + b;
      const unsigned long long bit = 1ull << k;
      x ^= bit;
      g ^= 1u << b;
      const bool added = (x & bit) != 0ull;
      const int u = P.au[k], v = P.av[k];
      const bool present = (x & P.grp[k]) != 0ull;
      M* ru = adj + u * nthr;
      *ru = present ? (*ru | ((M)1 << v)) : (*ru & ~((M)1 << v));
      if (!P.directed) {
        M* rv = adj + v * nthr;
        *rv = present ? (*rv | ((M)1 << u)) : (*rv & ~((M)1 << u));
      }
      pc += added ? 1 : -1;
      if (added != conn) conn = sink_reached<M>(adj, nthr, sbit, tbit);
      if (GRAD) {
        if (added)
          seg_start[b * nthr] = T;
        else
          u128_add_to(seg_acc[b * nthr], u128_sub(T, seg_start[b * nthr]));
      }
      if (conn) {
        u128_add_to(T, s_wmid[g]);
        ncnt[pc * nthr] += 1u;
      }
    }
    // the walk ends on g = 2^(L-1): only the top walk arc is still working
    if (GRAD && L > 0) u128_add_to(seg_acc[(L - 1) * nthr], u128_sub(T, seg_start[(L - 1) * nthr]));

    // ---- item epilogue: histogram, then masses in double-double
    if (lane_on) {
      const int base = pc_pre + __popc(lane);
      for (int c = 0; c <= L; ++c) {
        const uint32_t cnt = ncnt[c * nthr];
        if (cnt) atomicAdd(&s_nbins[base + c], (unsigned long long)cnt);
      }
    }
    // Sums over the lanes are integers to a common exponent (warp_sum_scaled);
    // every arc's ends on the lane that owns it, which scales all of them at
    // once in double-double.  (In double-double throughout, 14 warp sums of
    // five rounds were 1,300 FP64 instructions per item, and FP64 issues at
    // 1/64 of the FP32 rate: 23 arcs, 16,384 items, 1.30 ms; 0.29 so.)
    int eS;
    const u128 S = warp_sum_scaled(T, lw, &eS);
    dd ex[2];
    const dd wpre = prefix_mass<GRAD>(P, prefix, lane, ex);
    const dd wsum = dd_ldexp(u128_to_dd(S), eS);
    if (lane == 0) wacc[0] = dd_add(wacc[0], dd_mul(wpre, wsum));
    if (GRAD) {
      // of internal arc `lane`: a walk arc's masses with it working (X) and
      // failed (Y), a lane arc's pair differences (X)
      u128 X = u128_zero(), Y = u128_zero();
      int eX = 0, eY = 0;
      for (int b = 0; b < L; ++b) {
        const u128 A = seg_acc[b * nthr];
        int ea, ez;
        const u128 sa = warp_sum_scaled(A, lw, &ea), sz = warp_sum_scaled(u128_sub(T, A), lw, &ez);
        if (lane == ell + b) {
          X = sa;
          Y = sz;
          eX = ea;
          eY = ez;
        }
      }
      for (int i = 0; i < ell; ++i) {
        // the pair's lane with the arc working holds the larger T (exactly)
        const u128 o = u128{__shfl_xor_sync(0xffffffffu, T.lo, 1 << i), __shfl_xor_sync(0xffffffffu, T.hi, 1 << i)};
        const u128 df = (lane >> i) & 1 ? u128_sub(T, o) : u128_zero();
        int eg;
        const u128 sg = warp_sum_scaled(df, P.lane_tab ? s_lwx[i * 32 + lane] : P.lane_w_ex[i][lane], &eg);
        if (lane == i) {
          X = sg;
          eX = eg;
        }
      }
      if (lane < top) {
        dd y = dd_ldexp(u128_to_dd(X), eX);
        if (lane >= ell)
          y = dd_sub(dd_mul(y, P.inv_p[lane]), dd_mul(dd_ldexp(u128_to_dd(Y), eY), P.inv_q[lane]));
        wacc[1 + lane] = dd_add(wacc[1 + lane], dd_mul(wpre, y));
      }
      for (int j = lane; j < P.prefix_bits; j += 32)
        acc_signed(wacc[1 + top + j], dd_mul(j < 32 ? ex[0] : ex[1], wsum), (prefix >> j) & 1ull);
      __syncwarp();
    }
  }

  if (lane == 0) {
    atomicAdd(&W.stats[0], n_walk);
    atomicAdd(&W.stats[1], n_full);
    atomicAdd(&W.stats[2], n_dead);
  }
  __syncthreads();
  for (int i = tid; i <= m; i += nthr) {
    dd s = dd{0.0, 0.0};
    for (int w = 0; w < nwarps; ++w) s = dd_add(s, s_wacc[(size_t)w * (1 + m) + i]);
    W.part_acc[(size_t)blockIdx.x * (1 + m) + i] = s;
    W.part_n[(size_t)blockIdx.x * (m + 1) + i] = s_nbins[i];
  }
}

// Fixed-order sum of the per-block partials (PBAT STEP 3).  One CTA per
// output value; thread t sums blocks t, t + 256, ... in order, then a fixed
// shared-memory tree combines the 256 partial sums, so the result does not
// depend on scheduling.
constexpr int kReduceThreads = 256;

// Output i sums entry i of every block's partials (n_acc double-double
// sums and n_cnt counts per block) in a fixed order.
__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(DevWork W, int nblocks, int n_acc, int n_cnt) {
  __shared__ dd s_acc[kReduceThreads];
  __shared__ unsigned long long s_n[kReduceThreads];
  const int i = blockIdx.x, t = threadIdx.x;
  dd s = dd{0.0, 0.0};
  unsigned long long c = 0ull;
  for (int b = t; b < nblocks; b += kReduceThreads) {
    if (i < n_acc) s = dd_add(s, W.part_acc[(size_t)b * n_acc + i]);
    if (i < n_cnt) c += W.part_n[(size_t)b * n_cnt + i];
  }
  s_acc[t] = s;
  s_n[t] = c;
  __syncthreads();
  for (int h = kReduceThreads / 2; h > 0; h >>= 1) {
    if (t < h) {
      s_acc[t] = dd_add(s_acc[t], s_acc[t + h]);
      s_n[t] += s_n[t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    if (i < n_acc) W.out_acc[i] = s_acc[0];
    if (i < n_cnt) W.out_n[i] = s_n[0];
  }
}

size_t frontier_smem_bytes(int n, int m, int L, int nthr, bool grad, bool wide, bool lane_tab) {
  size_t off = 0;
  off = align16(off + ((size_t)1 << L) * sizeof(u128));
  off = align16(off + (size_t)n * nthr * (wide ? 8 : 4));
  off = align16(off + (size_t)(L + 1) * nthr * sizeof(uint32_t));
  if (grad) off = align16(off + (size_t)2 * L * nthr * sizeof(u128));
  off = align16(off + (size_t)(nthr / 32) * (1 + m) * sizeof(dd));
  off = align16(off + (size_t)(m + 1) * sizeof(unsigned long long));
  if (grad && lane_tab) off += (size_t)kMaxLaneBits * 32 * sizeof(LaneMass);
  return off;
}

const void* frontier_kernel_ptr(bool grad, bool wide) {
  if (wide)
    return grad ? (const void*)frontier_kernel<unsigned long long, true>
                : (const void*)frontier_kernel<unsigned long long, false>;
  return grad ? (const void*)frontier_kernel<uint32_t, true>
              : (const void*)frontier_kernel<uint32_t, false>;
}

cudaError_t launch_frontier(bool grad, bool wide, int grid, int nthr, size_t smem,
                            cudaStream_t st, const FrontierParams& P, const u128* wmid,
                            const DevWork& W) {
  if (wide) {
    if (grad)
      frontier_kernel<unsigned long long, true><<<grid, nthr, smem, st>>>(P, wmid, W);
    else
      frontier_kernel<unsigned long long, false><<<grid, nthr, smem, st>>>(P, wmid, W);
  } else {
    if (grad)
      frontier_kernel<uint32_t, true><<<grid, nthr, smem, st>>>(P, wmid, W);
    else
      frontier_kernel<uint32_t, false><<<grid, nthr, smem, st>>>(P, wmid, W);
  }
  return cudaGetLastError();
}

cudaError_t launch_reduce(cudaStream_t st, const DevWork& W, int nblocks, int n_acc, int n_cnt) {
  reduce_kernel<<<n_acc > n_cnt ? n_acc : n_cnt, kReduceThreads, 0, st>>>(W, nblocks, n_acc, n_cnt);
  return cudaGetLastError();
}

}  // namespace pbat
