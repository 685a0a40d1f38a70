// pmwa_kernels.cu -- sm_103a kernels of one PMWA Monte Carlo step.
//
//   k_boundary   Step 2 (Eq. 4) + Step 3 on the bonds between domains;
//                one warp per boundary bond, x bonds then y bonds, in
//                place on the current configuration.
//   k_temporal   Step 1 (Eq. 3), one warp per site.
//   k_rho        Supplement S-I worm density at equal-time slices, k_green
//                its equal-time sums, k_npoint products on listed sites.
//   k_pack, k_packed_check, k_unpack   checkpoints.
//   k_check      invariants of the current configuration, one warp per site.
// Steps 3-6 of every other bond and site run in k_tile (pmwa_tile.cu).
//
// Configuration layout in HBM: site i owns the slot key[i*cap .. i*cap+cap)
// of 64-bit event keys sorted in time, and cnt[i] = count | base << 31.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "pmwa_device.cuh"

namespace pmwa {

static inline int blocks_for(long long n, int bs) { return int((n + bs - 1) / bs); }

constexpr int kMaxWormsPerInterval = 128;
constexpr uint32_t kCntMask = 0x7fffffffu;

__device__ __forceinline__ int cnt_n(uint32_t c) { return int(c & kCntMask); }
__device__ __forceinline__ int cnt_base(uint32_t c) { return int(c >> 31); }
__device__ __forceinline__ uint32_t cnt_make(int n, int base) { return uint32_t(n) | (uint32_t(base) << 31); }

// An instance's record advanced to sweep iteration `it` of a batched call, in
// shared memory (all threads; the caller synchronises): at_iteration, copied a
// word a thread.
__device__ __forceinline__ void stage_record(Dev* sd, const Dev* g, const BatchBase& bb, int it) {
  static_assert(sizeof(Dev) % 8 == 0, "copied by words");
  const uint64_t* from = reinterpret_cast<const uint64_t*>(g);
  uint64_t* to = reinterpret_cast<uint64_t*>(sd);
  for (int k = threadIdx.x; k < int(sizeof(Dev) / 8); k += blockDim.x) to[k] = from[k];
  __syncthreads();
  if (threadIdx.x == 0) set_iteration(*sd, *g, bb, it);
}

// Supplement S-I worm density at K equal-time slices tau_k = k beta / K:
// eta g_sigma(x) of the interval between vertex legs holding tau_k.  2^sh
// threads a site (slice_lanes: the power of two from K up to a warp), one a
// slice: each finds its slice by bisection in the site's list (which its
// neighbours' loads keep in L1) and writes next to them.  The binary64 pipe bounds it,
// so the polynomials of this estimator are fused multiply-adds (the decisions
// of Steps 1 and 2 keep their separately rounded ones).  256x256 sites, K = 16:
// 177 us with a thread a site, now 162 us (cold).
__device__ __forceinline__ double g_sigma_fused(int sigma, double x) {
  const double y = -2.0 * x;
  const int h = __double2hiint(y) & 0x7fffffff;  // |y| compared on the integer pipe: 2^-6, 2^-4, 2^-2, 1
  double e;
  if (h < 0x3ff00000) {
    const int d = h < 0x3f900000 ? 7 : h < 0x3fb00000 ? 9 : h < 0x3fd00000 ? 13 : 19;
    double p = c_inv_fact[d];
    for (int n = d - 1; n >= 1; --n) p = fma(p, y, c_inv_fact[n]);
    e = p * y;
  } else {
    e = exp_det(y) - 1.0;
  }
  return sigma ? (2.0 + e) / -e : -e / (2.0 + e);
}

__global__ void k_rho(const __grid_constant__ Dev d, int K, int sh, double* out) {
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if ((t >> sh) >= d.N) return;
  const int s = int(t >> sh), step = 1 << sh;
  const uint64_t* Kk = d.keyA + size_t(s) * d.cap;
  const int n = cnt_n(d.cntA[s]);
  int lastleg = n - 1;
  while (lastleg >= 0 && kworm(Kk[lastleg])) --lastleg;
  const uint64_t q62 = kTwo62 / uint64_t(K), r62 = kTwo62 % uint64_t(K);
  for (int k = int(t) & (step - 1); k < K; k += step) {
    const uint64_t pt = uint64_t(k) * q62 + (uint64_t(k) * r62) / uint64_t(K);
    double r;
    if (lastleg < 0) {
      const double x = __dmul_rn(double(kTwo59), d.XW);
      r = __dmul_rn(d.eta, g_sigma_fused(0, x));
    } else {
      int lo = 0, hi = n;  // the first event above pt
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (kpk(Kk[mid]) <= pt) lo = mid + 1; else hi = mid;
      }
      int h = lo, j = lo - 1;  // last leg with pk <= pt and the next leg after it, cyclic
      while (h < n && kworm(Kk[h])) ++h;
      if (h == n) { h = 0; while (kworm(Kk[h])) ++h; }
      while (j >= 0 && kworm(Kk[j])) --j;
      if (j < 0) j = lastleg;
      const double x = __dmul_rn(__ull2double_rn(wpts(kpk(Kk[j]), kpk(Kk[h]))), d.XW);
      r = __dmul_rn(d.eta, g_sigma_fused(kab(Kk[j]) ^ kbl(Kk[h]), x));
    }
    out[size_t(s) * K + k] = r;
  }
}

static void run_rho(const Dev& d, int K, double* out, cudaStream_t st) {
  const int sh = slice_lanes(K);
  k_rho<<<blocks_for((long long)d.N << sh, 128), 128, 0, st>>>(d, K, sh, out);
}

static inline int site_warps(int N) { return blocks_for((long long)N * 32, 128); }

// ---------------------------------------------------------------------------
// Step 2 (spatial-boundary update, Eq. 4) and Step 3 on one boundary bond,
// in place on the current configuration.
__device__ __forceinline__ double vweight(const Dev& d, int S) {
  const int s0 = S & 1, s1 = (S >> 1) & 1, s2 = (S >> 2) & 1, s3 = (S >> 3) & 1;
  if (s0 + s1 != s2 + s3) return 0.0;
  if (s0 == s2) return d.dvw[s0 | (s1 << 1)];
  return d.tkink;
}

struct Legs {
  int single;
  uint64_t plo, phi, Idn, Iup;
  int far_dn, far_up;
  int wdn, wup;  // worms between the vertex and the next vertex leg below / above (0: none in the legs)
};

// the two legs of the vertex at pv on a site: to the next vertex leg below
// and above, worms ignored; one interval round the circle if v is alone.
// With temporal domains a leg also ends at the nearest temporal boundary,
// whose far state is the worldline's state there.
__device__ __forceinline__ bool site_legs_into(const Dev& d, const uint64_t* K, int n, uint64_t pv, Legs* L) {
  const int iv = slot_find(K, n, pv);
  if (iv < 0) return false;
  int jn = iv, jp = iv, wu = 0, wd = 0;
  for (int k = 0; k < n; ++k) { jn = (jn + 1 == n) ? 0 : jn + 1; if (jn == iv || !kworm(K[jn])) break; ++wu; }
  for (int k = 0; k < n; ++k) { jp = (jp == 0) ? n - 1 : jp - 1; if (jp == iv || !kworm(K[jp])) break; ++wd; }
  L->single = (jn == iv);
  L->wup = wu;
  L->wdn = wd;
  if (d.ntau > 1) {
    const uint64_t bu = tb_pk(d, tb_above(d, pv)), bd = tb_pk(d, tb_below(d, pv));
    if (L->single || up_dist(pv, bu) < up_dist(pv, kpk(K[jn]))) { L->phi = bu; L->far_up = slot_state(K, n, 0, bu); }
    else { L->phi = kpk(K[jn]); L->far_up = kbl(K[jn]); }
    if (L->single || up_dist(bd, pv) < up_dist(kpk(K[jp]), pv)) { L->plo = bd; L->far_dn = slot_state(K, n, 0, bd); }
    else { L->plo = kpk(K[jp]); L->far_dn = kab(K[jp]); }
    L->single = 0;
    L->Iup = wpts(pv, L->phi);
    L->Idn = wpts(L->plo, pv);
    return true;
  }
  if (L->single) { L->plo = L->phi = pv; L->Idn = L->Iup = kTwo59; L->far_dn = L->far_up = 0; return true; }
  L->phi = kpk(K[jn]); L->far_up = kbl(K[jn]); L->Iup = wpts(pv, L->phi);
  L->plo = kpk(K[jp]); L->far_dn = kab(K[jp]); L->Idn = wpts(L->plo, pv);
  return true;
}

// (wup = -1: there is no event at pv)
__device__ __noinline__ Legs site_legs(const Dev& d, const uint64_t* K, int n, uint64_t pv) {
  Legs L;
  L.wup = 0;
  if (!site_legs_into(d, K, n, pv, &L)) L.wup = -1;
  return L;
}

// Warp-cooperative list edits on a staged site list (all 32 lanes call them
// with the same arguments and see the same result).
//
// insert `key` at index `at`, shifting K[at..n) up by one, 32 keys at a time
// from the top (each chunk is read before any lane writes it)
__device__ __forceinline__ void aslot_insert(uint64_t* K, int n, int at, uint64_t key) {
  const int lane = threadIdx.x & 31;
  for (int top = n; top > at; top -= 32) {
    const int k = top - 1 - lane;
    const bool act = k >= at;
    uint64_t v = 0;
    if (act) v = K[k];
    __syncwarp();
    if (act) K[k + 1] = v;
    __syncwarp();
  }
  if (lane == 0) K[at] = key;
  __syncwarp();
}

// keep the keys for which drop(key) is false, in order; returns their count
template <class Drop>
__device__ __forceinline__ int warp_compact(uint64_t* K, int n, Drop drop) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int w = 0;
  for (int b = 0; b < n; b += 32) {
    const int k = b + lane;
    uint64_t key = 0;
    bool keep = false;
    if (k < n) { key = K[k]; keep = !drop(key); }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    __syncwarp();
    if (keep) K[w + __popc(m & lt)] = key;
    w += __popc(m);
    __syncwarp();
  }
  return w;
}

// first index >= from (a multiple of 32) whose key has tag `tag` and is at
// least `least` (n if none)
__device__ __forceinline__ int warp_find_tag(const uint64_t* K, int n, int from, int tag, uint64_t least) {
  const int lane = threadIdx.x & 31;
  for (int b = from; b < n; b += 32) {
    const int k = b + lane;
    const uint64_t key = k < n ? K[k] : 0;
    const unsigned m = __ballot_sync(0xffffffffu, k < n && ktag(key) == tag && key >= least);
    if (m) return b + __ffs(int(m)) - 1;
  }
  return n;
}

// keys below `key` in the sorted list; all of the first `from` (a multiple of
// 32) are known to be.  32 keys a step, without a bisection's chain of loads.
__device__ __forceinline__ int warp_lower(const uint64_t* K, int n, int from, uint64_t key) {
  const int lane = threadIdx.x & 31;
  for (int b = from; b < n; b += 32) {
    const unsigned m = __ballot_sync(0xffffffffu, b + lane < n && K[b + lane] < key);
    if (m != 0xffffffffu) return b + __popc(m);
  }
  return n;
}

// index of the event at time point pv, looked for from `hint` on first (-1: none)
__device__ __forceinline__ int warp_find_pk(const uint64_t* K, int n, int hint, uint64_t pv) {
  const int lane = threadIdx.x & 31;
  for (int turn = 0; turn < 2; ++turn) {
    for (int b = turn ? 0 : hint & ~31; b < n; b += 32) {
      const unsigned m = __ballot_sync(0xffffffffu, b + lane < n && kpk(K[b + lane]) == pv);
      if (m) return b + __ffs(int(m)) - 1;
    }
  }
  return -1;
}

// the legs of the vertex at index iv, as site_legs without temporal domains:
// the lanes look at the 32 events on either side at once
__device__ __forceinline__ void near_legs(const uint64_t* K, int n, int iv, uint64_t pv, Legs* L) {
  const int lane = threadIdx.x & 31;
  int jn = iv, jp = iv, wu = 0, wd = 0;
  for (int b = 0; b < n; b += 32) {
    int x = iv + 1 + b + lane;
    if (x >= n) x -= n;
    const unsigned m = __ballot_sync(0xffffffffu, b + lane < n && !kworm(K[x]));
    if (m) {
      wu = b + __ffs(int(m)) - 1;
      jn = iv + 1 + wu;
      if (jn >= n) jn -= n;
      break;
    }
  }
  for (int b = 0; b < n; b += 32) {
    int x = iv - 1 - b - lane;
    if (x < 0) x += n;
    const unsigned m = __ballot_sync(0xffffffffu, b + lane < n && !kworm(K[x]));
    if (m) {
      wd = b + __ffs(int(m)) - 1;
      jp = iv - 1 - wd;
      if (jp < 0) jp += n;
      break;
    }
  }
  L->single = (jn == iv);
  L->wup = wu;
  L->wdn = wd;
  if (L->single) { L->plo = L->phi = pv; L->Idn = L->Iup = kTwo59; L->far_dn = L->far_up = 0; return; }
  const uint64_t kn = K[jn], kp = K[jp];
  L->phi = kpk(kn); L->far_up = kbl(kn); L->Iup = wpts(pv, L->phi);
  L->plo = kpk(kp); L->far_dn = kab(kp); L->Idn = wpts(L->plo, pv);
}

// erase the worms strictly inside (lo, hi) going up (lo == hi: all of them;
// erase false: the caller knows there are none) and draw new ones with end
// states p (above lo) and q (below hi); K holds n events (capacity cap).
// (the stream -- with the window of blocks that the lanes hold, so that it is not
// drawn again -- and the list's count go in and out by value: a stream or count
// whose address is taken lives in local memory)
struct Regen {
  uint64_t pos;
  int n, rc;
};
__device__ __noinline__ Regen regen_slow(const Dev& d, ZigTab z, WarpStream st, uint64_t* K, int n, uint64_t lo,
                                         uint64_t hi, int p, int q) {
  uint64_t offs[kMaxWormsPerInterval];
  int bad = 0;
  const int nw = sample_worms<kMaxWormsPerInterval>(z, st, wpts(lo, hi), p ^ q, d.SWs, d.SWI, offs, &bad);
  if (bad) return Regen{st.pos, n, bad};
  const uint64_t m0 = wm_above(lo);
  for (int k = 0; k < nw; ++k) {
    if (n >= d.cap) return Regen{st.pos, n, PMWA_ECAPACITY};
    const uint64_t key = wkey((m0 + offs[k]) & (kTwo59 - 1), 0, p ^ 1 ^ (k & 1));
    aslot_insert(K, n, warp_lower(K, n, 0, key & ~3ull), key);
    ++n;
  }
  return Regen{st.pos, n, PMWA_OK};
}

// Two outcomes hold for most intervals and need no draw loop: a first gap
// longer than the interval is no worm for equal end states, and one uniform
// worm for different ones (x <= 1: the sampler's next two words, the first
// always kept).
__device__ __forceinline__ int regen_interval(const Dev& d, const ZigTab& z, WarpDraws& st, uint64_t* K, int& n,
                                              uint64_t lo, uint64_t hi, int p, int q, bool erase) {
  if (erase) {
    const uint64_t span = (hi > lo) ? hi - lo : hi + kTwo62 - lo;
    n = warp_compact(K, n, [&](uint64_t key) {  // the worms of the interval
      if (!kworm(key)) return false;
      const uint64_t off = (kpk(key) + kTwo62 - lo) & (kTwo62 - 1);
      return off > 0 && off < span;
    });
  }
  const uint64_t M = wpts(lo, hi);
  if (M > 0 && st.gap(z) > M) {
    if (p == q) { ++st.s.pos; return PMWA_OK; }
    if (M <= d.SWI) {
      st.s.pos += 2;
      const uint64_t key = wkey((wm_above(lo) + __umul64hi(st.word(z), M)) & (kTwo59 - 1), 0, p ^ 1);
      if (n >= d.cap) return PMWA_ECAPACITY;
      aslot_insert(K, n, warp_lower(K, n, 0, key & ~3ull), key);
      ++n;
      return PMWA_OK;
    }
  }
  const Regen r = regen_slow(d, z, st.s, K, n, lo, hi, p, q);
  st.s.pos = r.pos;
  n = r.n;
  return r.rc;
}

__device__ __forceinline__ double fsig(int sigma, double em1) { return sigma ? -em1 : __dadd_rn(2.0, em1); }

// Eq. 4 in binary32 (lane < 16: state S = lane; all 32 lanes call it): the
// same heat bath with the leg factors from expm1f and the vertex weights
// rounded to binary32.  Its cumulative fractions c_S / tot lie within 2^-16
// of the binary64 ones (expm1f within a few units in the last place, at
// most four factors and one vertex weight, a sum of at most six terms, each
// a relative 2^-22 or better), so when the uniform r = (w >> 11) 2^-53 lies
// more than 2^-12 from 0, 1 and every boundary, the binary64 computation
// picks the same state.  (A state whose binary32 weight vanishes while its
// binary64 one does not has a fraction below 2^-100 and so sits within the
// margin of a neighbouring boundary or of 0.)  Returns that state, or -1.
__device__ __forceinline__ int heat_bath_f32(const Dev& d, const Legs& La, const Legs& Lb, uint64_t w, int lane) {
  float e4 = 0.f;
  if (lane < 4) {
    uint64_t I;
    if (lane == 0) I = La.single ? kTwo59 : La.Idn;
    else if (lane == 1) I = Lb.single ? kTwo59 : Lb.Idn;
    else if (lane == 2) I = La.single ? kTwo59 : La.Iup;
    else I = Lb.single ? kTwo59 : Lb.Iup;
    e4 = expm1f(-2.0f * __ull2float_rn(I) * d.XWf);
  }
  const float ea_dn = __shfl_sync(0xffffffffu, e4, 0), eb_dn = __shfl_sync(0xffffffffu, e4, 1);
  const float ea_up = __shfl_sync(0xffffffffu, e4, 2), eb_up = __shfl_sync(0xffffffffu, e4, 3);
  float wS = 0.f;
  if (lane < 16) {
    const int S = lane, s0 = S & 1, s1 = (S >> 1) & 1, s2 = (S >> 2) & 1, s3 = (S >> 3) & 1;
    if (s0 + s1 == s2 + s3) {
      float v = (s0 == s2) ? d.dvwf[s0 | (s1 << 1)] : d.tkinkf;
      auto f = [](int sg, float e) { return sg ? -e : 2.0f + e; };
      if (!La.single) v *= f(La.far_dn ^ s0, ea_dn);
      if (!Lb.single) v *= f(Lb.far_dn ^ s1, eb_dn);
      v *= La.single ? f(s2 ^ s0, ea_up) : f(s2 ^ La.far_up, ea_up);
      v *= Lb.single ? f(s3 ^ s1, eb_up) : f(s3 ^ Lb.far_up, eb_up);
      wS = v;
    }
  }
  float c = wS;  // inclusive running sums over the states
  for (int o = 1; o < 16; o <<= 1) {
    const float t = __shfl_up_sync(0xffffffffu, c, o);
    if (lane >= o) c += t;
  }
  const float tot = __shfl_sync(0xffffffffu, c, 15);
  if (!(tot > 0x1p-100f)) return -1;
  const float r = __ull2float_rn(w >> 11) * 0x1p-53f;
  const float fr = c / tot;
  const bool pos = lane < 16 && wS > 0.f;
  const bool near = (pos && fabsf(r - fr) <= 0x1p-12f) || r <= 0x1p-12f;
  if (__any_sync(0xffffffffu, near)) return -1;
  const unsigned hit = __ballot_sync(0xffffffffu, pos && r < fr);
  return hit ? __ffs(int(hit)) - 1 : -1;
}
__device__ __forceinline__ double em1_of(uint64_t I, double XW) {
  return expm1_det(__dmul_rn(-2.0, __dmul_rn(__ull2double_rn(I), XW)));
}

__device__ __forceinline__ int boundary_count(const Dev& d, int dir) {
  return dir == 0 ? (d.ndx > 1 ? d.ndx * d.Ly : 0) : (d.ndy > 1 ? d.ndy * d.Lx : 0);
}

// lower site of boundary bond number t of direction dir
__device__ __forceinline__ int boundary_site(const Dev& d, int dir, int t) {
  if (dir == 0) return ((t % d.ndx) * d.dom_x + d.dom_x - 1) + d.Lx * (t / d.ndx);
  return (t % d.Lx) + d.Lx * ((t / d.Lx) * d.dom_y + d.dom_y - 1);
}

// On-the-fly vertex generation: is grid point pos within half of a worm of
// either staged list (cyclic)?
__device__ __forceinline__ bool in_win_lists(const uint64_t* KA, int nA, const uint64_t* KB, int nB, uint64_t pos,
                                             uint64_t half) {
  for (int side = 0; side < 2; ++side) {
    const uint64_t* K = side ? KB : KA;
    const int n = side ? nB : nA;
    for (int i = 0; i < n; ++i) {
      if (!kworm(K[i])) continue;
      const uint64_t m = kpk(K[i]) >> 3;
      const uint64_t a = (pos - m) & (kTwo59 - 1), b = (m - pos) & (kTwo59 - 1);
      if (min(a, b) <= half) return true;
    }
  }
  return false;
}

// Step 2 + Step 3 on the boundary bond (a, dir) whose two site lists are
// staged in KA (nA events) and KB (nB events); returns a status.  With
// d.win_half > 0 the Step-3 part is confined to the windows around the worms
// of the two sites (on-the-fly vertex generation).
__device__ __forceinline__ int boundary_bond_update(const Dev& d, int a, int dir, uint64_t* KA, int& nA, int& baseA,
                                    uint64_t* KB, int& nB, int& baseB, const ZigTab& Z) {
  const int tag = bond_tag(d, a, dir);
  const int bid = 2 * a + dir;
  WarpDraws st;
  st.init(d.key0, d.key1, uint32_t(bid), c2_word(dir ? kBy : kBx, 0, d.replica), d.sweep, d.SWs);
  int rc = PMWA_OK;
  // Step 2: the bond's vertices in time order (worms move, vertices do not).
  // ia, ib: where the last one stands in the lists now, or before it (0 after
  // a redraw round the origin, whose worms may come to stand anywhere)
  uint64_t least = 0;
  int ia = 0, ib = 0;
  for (;;) {
    const int ka = warp_find_tag(KA, nA, ia & ~31, tag, least);
    if (ka >= nA) break;
    const uint64_t pv = kpk(KA[ka]);
    least = (pv + 1) << 2;
    const int kb = warp_find_pk(KB, nB, ib, pv);
    if (kb < 0) return PMWA_EINVARIANT;
    Legs La, Lb;
    if (d.ntau > 1) {
      La = site_legs(d, KA, nA, pv);
      Lb = site_legs(d, KB, nB, pv);
      if (La.wup < 0 || Lb.wup < 0) return PMWA_EINVARIANT;
    } else {
      near_legs(KA, nA, ka, pv, &La);
      near_legs(KB, nB, kb, pv, &Lb);
    }
    // heat-bath over the root states (Eq. 4): decided in binary32 when the
    // uniform lies clear of every boundary, else in binary64 with one lane
    // per leg factor and one lane per state and the weights summed in the
    // fixed order S = 0..15
    const int lane = threadIdx.x & 31;
    const uint64_t wu = st.word(Z);
    int Sn = heat_bath_f32(d, La, Lb, wu, lane);
    if (Sn < 0) {
    double e4 = 0.0;
    if (lane < 4) {
      uint64_t I;
      if (lane == 0) I = La.single ? kTwo59 : La.Idn;
      else if (lane == 1) I = Lb.single ? kTwo59 : Lb.Idn;
      else if (lane == 2) I = La.single ? kTwo59 : La.Iup;
      else I = Lb.single ? kTwo59 : Lb.Iup;
      e4 = em1_of(I, d.XW);
    }
    const double ea_dn = __shfl_sync(0xffffffffu, e4, 0), eb_dn = __shfl_sync(0xffffffffu, e4, 1);
    const double ea_up = __shfl_sync(0xffffffffu, e4, 2), eb_up = __shfl_sync(0xffffffffu, e4, 3);
    double wS = 0.0;
    if (lane < 16) {
      const int S = lane;
      double w = vweight(d, S);
      if (w > 0.0) {
        const int s0 = S & 1, s1 = (S >> 1) & 1, s2 = (S >> 2) & 1, s3 = (S >> 3) & 1;
        if (!La.single) w = __dmul_rn(w, fsig(La.far_dn ^ s0, ea_dn));
        if (!Lb.single) w = __dmul_rn(w, fsig(Lb.far_dn ^ s1, eb_dn));
        w = __dmul_rn(w, La.single ? fsig(s2 ^ s0, ea_up) : fsig(s2 ^ La.far_up, ea_up));
        w = __dmul_rn(w, Lb.single ? fsig(s3 ^ s1, eb_up) : fsig(s3 ^ Lb.far_up, eb_up));
      }
      wS = w;
    }
    // running sums in the order S = 0..15 over the states of non-zero
    // weight only (adding +0.0 changes no sum, so this is the sequential
    // sum over all 16); a zero-weight state keeps cumS = 0 and is never hit
    const unsigned pos = __ballot_sync(0xffffffffu, lane < 16 && wS > 0.0);
    if (!pos) return PMWA_EINVARIANT;
    double tot = 0.0, cumS = 0.0;
    for (unsigned m = pos; m; m &= m - 1) {
      const int S = __ffs(int(m)) - 1;
      tot = __dadd_rn(tot, __shfl_sync(0xffffffffu, wS, S));
      if (lane == S) cumS = tot;
    }
    const int lastS = 31 - __clz(int(pos));
    const double u = __dmul_rn(__dmul_rn(__ull2double_rn(wu >> 11), 0x1p-53), tot);
    const unsigned hit = __ballot_sync(0xffffffffu, lane < 16 && u < cumS);
    Sn = hit ? (__ffs(int(hit)) - 1) : lastS;
    }
    const int s0 = Sn & 1, s1 = (Sn >> 1) & 1, s2 = (Sn >> 2) & 1, s3 = (Sn >> 3) & 1;
    KA[ka] = (KA[ka] & ~3ull) | (uint64_t(s0) << 1) | uint64_t(s2);
    KB[kb] = (KB[kb] & ~3ull) | (uint64_t(s1) << 1) | uint64_t(s3);
    // the worms of v's four intervals anew: below on the lower and the upper
    // site, then above (the worm counts of the legs were taken before any
    // redraw; a redraw below v adds worms only below v, so the counts above v
    // still hold).  One body for the four: inlined four times it takes the
    // registers of two more warps.
    const int nA0 = nA, nB0 = nB;
    for (int e = 0; e < 4 && !rc; ++e) {
      const bool onB = e & 1, above = e >= 2;
      if (e == 2) {
        ia = (!La.single && La.plo < pv && pv < La.phi) ? ka + nA - nA0 : 0;
        ib = (!Lb.single && Lb.plo < pv && pv < Lb.phi) ? kb + nB - nB0 : 0;
      }
      const int single = onB ? Lb.single : La.single;
      if (single && !above) continue;
      const int bot = onB ? s1 : s0, top = onB ? s3 : s2;
      const uint64_t far = above ? (onB ? Lb.phi : La.phi) : (onB ? Lb.plo : La.plo);
      const uint64_t lo = above ? pv : far, hi = above ? (single ? pv : far) : pv;
      const int p = above ? top : (onB ? Lb.far_dn : La.far_dn);
      const int q = above ? (single ? bot : (onB ? Lb.far_up : La.far_up)) : bot;
      const int worms = above ? (onB ? Lb.wup : La.wup) : (onB ? Lb.wdn : La.wdn);
      int n = onB ? nB : nA;
      rc = regen_interval(d, Z, st, onB ? KB : KA, n, lo, hi, p, q, worms > 0);
      if (onB) nB = n; else nA = n;
    }
    if (rc) return rc;
  }
  if (st.s.pos >= (uint64_t(1) << 33)) return PMWA_ETIMEOUT;
  // states at the start of the circles after Step 2 (used if a list empties)
  if (nA) baseA = kab(KA[nA - 1]);
  if (nB) baseB = kab(KB[nB - 1]);
  // Step 3 on this bond: erase its diagonal vertices, lay new ones
  const bool otf = d.win_half > 0;
  {
    // (the windows do not move: the compaction drops only diagonal legs, so
    // while it runs every worm of both lists is still found in their first
    // nA / nB slots, some of them twice, which the window test does not mind)
    auto diag = [&](uint64_t key) {
      return ktag(key) == tag && kab(key) == kbl(key) &&
             (!otf || in_win_lists(KA, nA, KB, nB, kpk(key) >> 3, d.win_half));
    };
    const int wa = warp_compact(KA, nA, diag);
    const int wb = warp_compact(KB, nB, diag);
    const int removed = nA - wa, gone = nB - wb;
    nA = wa;
    nB = wb;
    if (gone != removed) return PMWA_EINVARIANT;
  }
  if (!d.has_vertices) return PMWA_OK;
  WarpDraws sv;
  sv.init(d.key0, d.key1, uint32_t(bid), c2_word(kVertex, 0, d.replica), d.sweep, d.SVs);
  uint64_t pos = 0;
  bool first = true;
  int bad = 0, xa = 0, xb = 0;  // events of the lists below the last candidate
  for (;;) {
    uint64_t g = sv.gap(Z);
    if (g) {
      ++sv.s.pos;
    } else {
      DrawWords words{sv, Z};
      const uint64_t E = zig_exp(Z, words, &bad);
      if (bad) return bad;
      g = grid_gap(E, d.SVs);
    }
    const uint64_t nxt = first ? g - 1 : pos + g;
    first = false;
    if (nxt >= kTwo59) break;
    pos = nxt;
    const uint64_t pk = (pos << 3) | uint64_t(tag), key = pk << 2;
    if (otf && !in_win_lists(KA, nA, KB, nB, pos, d.win_half)) continue;
    xa = warp_lower(KA, nA, xa & ~31, key);
    if (xa < nA && kpk(KA[xa]) == pk) continue;
    xb = warp_lower(KB, nB, xb & ~31, key);
    const int na = nA ? kab(KA[(xa ? xa : nA) - 1]) : baseA, nb = nB ? kab(KB[(xb ? xb : nB) - 1]) : baseB;
    const int si = na | (nb << 1);
    if (d.TV[si] < kTwo32) {
      const uint64_t w = sv.word(Z);
      if ((w >> 32) >= d.TV[si]) continue;
    }
    if (nA >= d.cap || nB >= d.cap) return PMWA_ECAPACITY;
    aslot_insert(KA, nA, xa, key | (uint64_t(na) << 1) | uint64_t(na));
    ++nA;
    aslot_insert(KB, nB, xb, key | (uint64_t(nb) << 1) | uint64_t(nb));
    ++nB;
  }
  return PMWA_OK;
}

// One warp per boundary bond.  The warp copies the bond's two site lists
// into its shared-memory stage (coalesced), every lane then runs the same
// update on the same data (so nothing diverges; lanes split only the
// heat-bath arithmetic), and the warp copies the lists back.  stage: 2 * cap
// event keys for this warp.
__device__ void boundary_warp(const Dev& d, int dir, int t, uint64_t* stage, const ZigTab& Z) {
  const int lane = threadIdx.x & 31;
  if (t >= boundary_count(d, dir)) return;
  const int a = boundary_site(d, dir, t);
  const int b = site_step(d, a, dir, +1);
  const uint32_t ca = d.cntA[a], cb = d.cntA[b];
  int nA = cnt_n(ca), baseA = cnt_base(ca), nB = cnt_n(cb), baseB = cnt_base(cb);
  const uint64_t* ga = d.keyA + size_t(a) * d.cap;
  const uint64_t* gb = d.keyA + size_t(b) * d.cap;
  uint64_t* sa = stage;
  uint64_t* sb = stage + d.cap;
  for (int k = lane; k < nA; k += 32) sa[k] = ga[k];
  for (int k = lane; k < nB; k += 32) sb[k] = gb[k];
  __syncwarp();
  const int rc = boundary_bond_update(d, a, dir, sa, nA, baseA, sb, nB, baseB, Z);
  __syncwarp();
  if (rc) {
    if (lane == 0) set_err(d.err, rc, 2);
    return;
  }
  uint64_t* wa = d.keyA + size_t(a) * d.cap;
  uint64_t* wb = d.keyA + size_t(b) * d.cap;
  for (int k = lane; k < nA; k += 32) wa[k] = sa[k];
  for (int k = lane; k < nB; k += 32) wb[k] = sb[k];
  if (lane == 0) {
    d.cntA[a] = cnt_make(nA, nA ? kab(sa[nA - 1]) : baseA);
    d.cntA[b] = cnt_make(nB, nB ? kab(sb[nB - 1]) : baseB);
  }
}

// One bond (warp) a block.  A bond is one chain of its vertices and their
// lengths differ, so a block of several warps keeps its place on the SM for the
// longest; and what bounds the kernel is the number of such chains an SM can
// interleave (every lane runs the same scalar step, 11 cycles an instruction
// with 7 warps a scheduler): 28 one-warp blocks an SM, 72 registers.  A launch,
// against blocks of four warps and bisections, draws and list searches done
// step by step: 256x256 beta t = 4 0.112 -> 0.066 ms, 512x512 beta t = 16 1.05 ->
// 0.62 ms, 4x4 domains at V/t = 3 1.02 -> 0.52 ms; with 12 / 16 / 20 / 24 blocks
// an SM 256x256 took 0.090 / 0.081 / 0.076 / 0.073 ms.  Likewise Step 1's sites
// (32 blocks: 128x128 in 4 slabs 0.119 -> 0.085 ms).
//
// Registers, spill stores and loads (bytes): k_boundary 72, 24 and 24,
// k_temporal 56 without spills.  The batched forms have the instance's record
// in shared memory instead of the constant bank and its fields in registers; a
// spill is costly, as beside 200 KB of shared memory the L1 has no room for
// the blocks' local memory.  They take 20 (96 registers, 244 and 176) and 24 blocks
// (80, 76 and 128): at 28 and 32, where the spills are 612 / 460 and 360 / 276, most
// replica sets were slower, at 16 those of long lists.  Against 28 and 32 blocks
// with the round keys kept in registers and the record copied by one lane
// (684 / 940 and 372 / 352), 400 replicas of 32x32 sites: 8x8 domains at beta t
// = 4, eta = 0.2 0.597 -> 0.483 ms a launch (blocks of four warps: 0.504), four
// slabs at beta t = 8 1.78 -> 1.36 ms of Step 1 (1.62).
constexpr int kBatchBlocks = 20;

__global__ void __launch_bounds__(32, 28) k_boundary(const __grid_constant__ Dev d, int dir) {
  extern __shared__ __align__(16) unsigned char bsm[];
  if (instance_failed(d.err)) return;
  const ZigTab Z = zig_stage(bsm, d.zig_cap, d.worm_tries);
  __syncthreads();
  boundary_warp(d, dir, int(blockIdx.x), reinterpret_cast<uint64_t*>(bsm + kZigBytes), Z);
}

// Batched form: each block serves a bond of one instance, when that instance's
// boundary step is due at iteration `it`.
__global__ void __launch_bounds__(32, kBatchBlocks) k_boundary_batch(const Dev* __restrict__ devs,
                                                                     const BatchBase* __restrict__ base,
                                                                     const int2* __restrict__ work, int it, int dir) {
  extern __shared__ __align__(16) unsigned char bsm[];
  __shared__ Dev sd;
  const int2 w = work[blockIdx.x];
  const BatchBase bb = base[w.x];
  if (!bb.active) return;
  stage_record(&sd, devs + w.x, bb, it);
  ZigTab Z = zig_stage(bsm);
  __syncthreads();
  Z.zcap = sd.zig_cap;
  Z.wtries = sd.worm_tries;
  if (instance_failed(sd.err)) return;
  if (sd.ndom < 2 || sd.sweep % uint32_t(sd.exchange_every) != 0) return;
  boundary_warp(sd, dir, w.y, reinterpret_cast<uint64_t*>(bsm + kZigBytes), Z);
}

// ---------------------------------------------------------------------------
// Step 1 (temporal-boundary update, Eq. 3), one warp per site, in place on
// the current configuration.  Boundary k lies in the interval I = I2 + I1
// between the nearest delimiters below and above it (vertex legs or other
// temporal boundaries, worms ignored): I2 from the lower delimiter (state p
// just above it) up to the boundary, I1 from the boundary up to the upper one
// (state q just below it).  The new state s' is drawn with P(s') =
// f_{q s'}(I1) f_{s' p}(I2) / f_{q p}(I); with f_{ab}(x) = e^x F(a ^ b, x) / 2,
// F(0, x) = 2 + expm1(-2x), F(1, x) = -expm1(-2x), the e^x / 2 are common to
// both s' and drop out.  The worms of I2 and then I1 are drawn anew (Eq. 1).
// The boundaries of a site go in order k = 0, 1, ..., each a heat bath given
// the current states of the others; sites are independent.  Every lane runs
// the same update on the staged list, as in the spatial boundary step.

// the nearest delimiter of boundary k going down (up = false) or up: its pk
// and the state on the side facing the boundary
__device__ __forceinline__ void tb_delim(const Dev& d, const uint64_t* K, int n, int base, int k, bool up,
                                         uint64_t* pk, int* st) {
  const uint64_t B = tb_pk(d, k);
  const int kb = up ? (k + 1) % d.ntau : (k + d.ntau - 1) % d.ntau;
  uint64_t best = tb_pk(d, kb);
  int leg = -1;
  if (n > 0) {
    // the nearest vertex leg in that direction, cyclic (worms skipped)
    const int i0 = slot_lower(K, n, B);  // first event above B
    for (int c = 0; c < n; ++c) {
      const int i = up ? (i0 + c) % n : (i0 + n - 1 - c) % n;
      if (kworm(K[i])) continue;
      const uint64_t q = kpk(K[i]);
      if (up ? up_dist(B, q) < up_dist(B, best) : up_dist(q, B) < up_dist(best, B)) { best = q; leg = i; }
      break;
    }
  }
  *pk = best;
  *st = (leg >= 0) ? (up ? kbl(K[leg]) : kab(K[leg])) : slot_state(K, n, base, best);
}

__device__ __forceinline__ int temporal_site(const Dev& d, int s, uint64_t* K, int& n, int& base, const ZigTab& Z) {
  WarpDraws st;
  st.init(d.key0, d.key1, uint32_t(s), c2_word(kTemporal, 0, d.replica), d.sweep, d.SWs);
  for (int k = 0; k < d.ntau; ++k) {
    const uint64_t B = tb_pk(d, k);
    uint64_t lo, hi;
    int p, q;
    tb_delim(d, K, n, base, k, false, &lo, &p);
    tb_delim(d, K, n, base, k, true, &hi, &q);
    const uint64_t I1 = wpts(B, hi), I2 = wpts(lo, B);
    const uint64_t wu = st.word(Z);
    // decided in binary32 when the uniform lies more than 2^-12 from the
    // fraction w0 / (w0 + w1) (two leg factors: the binary32 fraction is
    // within 2^-18 of the binary64 one), else in binary64
    int sn;
    {
      auto f = [](int sg, float e) { return sg ? -e : 2.0f + e; };
      const float g1 = expm1f(-2.0f * __ull2float_rn(I1) * d.XWf), g2 = expm1f(-2.0f * __ull2float_rn(I2) * d.XWf);
      const float v0 = f(q, g1) * f(p, g2), v1 = f(q ^ 1, g1) * f(1 ^ p, g2);
      const float r = __ull2float_rn(wu >> 11) * 0x1p-53f, fr = v0 / (v0 + v1);
      sn = (v0 + v1 > 0x1p-100f && fabsf(r - fr) > 0x1p-12f && r > 0x1p-12f) ? (r < fr ? 0 : 1) : -1;
    }
    if (sn < 0) {
      const double e1 = em1_of(I1, d.XW), e2 = em1_of(I2, d.XW);
      const double w0 = __dmul_rn(fsig(q, e1), fsig(p, e2));
      const double w1 = __dmul_rn(fsig(q ^ 1, e1), fsig(1 ^ p, e2));
      const double tot = __dadd_rn(w0, w1);
      if (!(tot > 0.0)) return PMWA_EINVARIANT;
      const double u = __dmul_rn(__dmul_rn(__ull2double_rn(wu >> 11), 0x1p-53), tot);
      sn = (u < w0) ? 0 : 1;
    }
    int rc = PMWA_OK;
    for (int e = 0; e < 2 && !rc; ++e)
      rc = regen_interval(d, Z, st, K, n, e ? B : lo, e ? hi : B, e ? sn : p, e ? q : sn, true);
    if (rc) return rc;
    if (n == 0) base = sn;
  }
  if (st.s.pos >= (uint64_t(1) << 33)) return PMWA_ETIMEOUT;
  return PMWA_OK;
}

constexpr int kBatchSiteBlocks = 24;

// one warp: stage site s's list (cap keys at K), update its boundaries, and
// write it back
__device__ void temporal_warp(const Dev& d, int s, uint64_t* K, const ZigTab& Z) {
  const int lane = threadIdx.x & 31;
  if (s >= d.N) return;
  const uint32_t c = d.cntA[s];
  int n = cnt_n(c), base = cnt_base(c);
  const uint64_t* g = d.keyA + size_t(s) * d.cap;
  for (int k = lane; k < n; k += 32) K[k] = g[k];
  __syncwarp();
  const int rc = temporal_site(d, s, K, n, base, Z);
  __syncwarp();
  if (rc) {
    if (lane == 0) set_err(d.err, rc, 1);
    return;
  }
  uint64_t* w = d.keyA + size_t(s) * d.cap;
  for (int k = lane; k < n; k += 32) w[k] = K[k];
  if (lane == 0) d.cntA[s] = cnt_make(n, n ? kab(K[n - 1]) : base);
}

__global__ void __launch_bounds__(32, 32) k_temporal(const __grid_constant__ Dev d) {
  extern __shared__ __align__(16) unsigned char tsm[];
  if (instance_failed(d.err)) return;
  const ZigTab Z = zig_stage(tsm, d.zig_cap, d.worm_tries);
  __syncthreads();
  temporal_warp(d, int(blockIdx.x), reinterpret_cast<uint64_t*>(tsm + kZigBytes), Z);
}

// Batched form: each block serves a site of one instance, when that instance
// has temporal domains and its Step 1 is due at iteration `it`.
__global__ void __launch_bounds__(32, kBatchSiteBlocks) k_temporal_batch(const Dev* __restrict__ devs,
                                                                         const BatchBase* __restrict__ base,
                                                                         const int2* __restrict__ work, int it) {
  extern __shared__ __align__(16) unsigned char tsm[];
  __shared__ Dev sd;
  const int2 w = work[blockIdx.x];
  const BatchBase bb = base[w.x];
  if (!bb.active) return;
  stage_record(&sd, devs + w.x, bb, it);
  ZigTab Z = zig_stage(tsm);
  __syncthreads();
  Z.zcap = sd.zig_cap;
  Z.wtries = sd.worm_tries;
  if (instance_failed(sd.err)) return;
  if (sd.ntau < 2 || sd.sweep % uint32_t(sd.exchange_every) != 0) return;
  temporal_warp(sd, w.y, reinterpret_cast<uint64_t*>(tsm + kZigBytes), Z);
}

static size_t temporal_smem(int cap) { return size_t(kZigBytes) + size_t(cap) * 8; }

int launch_temporal(const Dev& d, void* stream) {
  if (d.ntau < 2) return 0;
  const size_t smem = temporal_smem(d.cap);
  cudaError_t e = cudaFuncSetAttribute(k_temporal, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e) return int(e);
  k_temporal<<<d.N, 32, smem, cudaStream_t(stream)>>>(d);
  return int(cudaGetLastError());
}

// (the batch sets the kernel's shared-memory allowance once, before any
// capture: prepare_temporal)
int prepare_temporal(int cap) {
  return int(cudaFuncSetAttribute(k_temporal_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  int(temporal_smem(cap))));
}

int launch_temporal_batch(const Dev* devs, const BatchBase* base, const int2* work, int n_work, int it, int cap,
                          void* stream) {
  if (n_work <= 0) return 0;
  k_temporal_batch<<<n_work, 32, temporal_smem(cap), cudaStream_t(stream)>>>(devs, base, work, it);
  return int(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Launchers.

int upload_zig(const Zig& z) { return upload_constants(z); }

// advance every instance's batch state by S sweeps (the tail of a captured
// sequence of S sweeps, so that the next replay continues where it ended)
__global__ void k_advance(BatchBase* base, int n, int S) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || !base[i].active) return;
  base[i].sweep0 += uint32_t(S);
  base[i].row0 += S;
  base[i].flip ^= (S & 1);
}

int launch_advance(BatchBase* base, int n, int S, void* stream) {
  k_advance<<<blocks_for(n, 128), 128, 0, cudaStream_t(stream)>>>(base, n, S);
  return int(cudaGetLastError());
}

size_t boundary_smem(int cap) { return size_t(kZigBytes) + 2 * size_t(cap) * 8; }

int prepare_boundary(int cap) {
  cudaError_t e = cudaFuncSetAttribute(k_boundary, cudaFuncAttributeMaxDynamicSharedMemorySize, int(boundary_smem(cap)));
  if (e) return int(e);
  return int(cudaFuncSetAttribute(k_boundary_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  int(boundary_smem(cap))));
}

int launch_boundary_batch(const Dev* devs, const BatchBase* base, const int2* work, int n_work, int it, int dir,
                          int cap, void* stream) {
  if (n_work <= 0) return 0;
  k_boundary_batch<<<n_work, 32, boundary_smem(cap), cudaStream_t(stream)>>>(devs, base, work, it, dir);
  return int(cudaGetLastError());
}

int launch_boundary(const Dev& d, int dir, void* stream) {
  const long long n = dir == 0 ? (long long)d.ndx * d.Ly : (long long)d.ndy * d.Lx;
  if ((dir == 0 && d.ndx < 2) || (dir == 1 && d.ndy < 2)) return 0;
  cudaError_t e = cudaFuncSetAttribute(k_boundary, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       int(boundary_smem(d.cap)));
  if (e) return int(e);
  k_boundary<<<unsigned(n), 32, boundary_smem(d.cap), cudaStream_t(stream)>>>(d, dir);
  return int(cudaGetLastError());
}

// Scratch of pmwa_rho_slices_static: the rho values of one call live here
// between the kernel and the copy to the host, instead of in the caller's
// arena.  Every GPU that loads the library holds this array until the
// process exits.  Calls that overlap on the GPU share it and race; each call
// overwrites all N*K values it returns, so nothing needs clearing between
// calls (the array keeps the last call's contents).
constexpr size_t kRhoStaticMax = size_t(1) << 20;  // doubles (8 MiB)
static __device__ __align__(256) double g_rho_scratch[kRhoStaticMax];

// Device address of g_rho_scratch on the current device, looked up once per
// device (in host code the symbol is only a host-side stand-in).
static double* rho_scratch_address(int* status) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static double* addr[kMaxDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { *status = PMWA_ECUDA; return nullptr; }
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_rho_scratch) != cudaSuccess || !p) { *status = PMWA_ECUDA; return nullptr; }
    addr[dev] = static_cast<double*>(p);
  }
  *status = PMWA_OK;
  return addr[dev];
}

int rho_slices_static(const Dev& d, int K, double* host_out, void* stream) {
  if (K < 1 || !host_out) return PMWA_EINVAL;
  if (size_t(d.N) * size_t(K) > kRhoStaticMax) return PMWA_EINVAL;
  int st = PMWA_OK;
  double* scratch = rho_scratch_address(&st);
  if (!scratch) return st;
  run_rho(d, K, scratch, cudaStream_t(stream));
  if (cudaGetLastError() != cudaSuccess) return PMWA_ECUDA;
  if (cudaMemcpyAsync(host_out, scratch, size_t(d.N) * size_t(K) * sizeof(double), cudaMemcpyDeviceToHost,
                      cudaStream_t(stream)) != cudaSuccess)
    return PMWA_ECUDA;
  if (cudaStreamSynchronize(cudaStream_t(stream)) != cudaSuccess) return PMWA_ECUDA;
  return PMWA_OK;
}

// Supplement S-I equal-time correlators from the worm densities rho[i*K+k]:
// sum_{i,k} rho_i rho_{i+r x} into sums[r-1], rho_i rho_{i+r y} into
// sums[rmax + r - 1] (r = 1..rmax), and the plaquette product rho_i rho_{i+x}
// rho_{i+y} rho_{i+x+y} into sums[2 rmax].  A row of the lattice is Lx K
// consecutive doubles and a shift by r sites is a cyclic shift by r K of it,
// so every load is coalesced; a block takes kGreenR values of r (blockIdx.y;
// the last one the plaquette), which share the row's own densities, and pieces
// of kGreenSteps elements a thread: of a row, or of several rows shorter than
// the block.  There are as many blocks as the machine holds at once: with one a
// row, a lattice of few rows left it idle, and blocks of short rows spent their
// time on the sums' reduction.  The call, a thread a site (a line a lane and load)
// -> a block a row -> now: 256x256 sites, rmax = 128 with K = 16 1.57 -> 0.82 ->
// 0.71 ms and with K = 1 0.211 -> 0.288 -> 0.114 ms; 65536x2 sites, K = 16, rmax = 1
// 0.49 -> 2.40 -> 0.41 ms.  Two fused multiply-adds a site, slice and r, on a
// binary64 pipe of two lanes a cycle and SM, bound the first.
constexpr int kGreenR = 4, kGreenSteps = 4;
// elements of a row that a block takes side by side; pieces of the lattice
__host__ __device__ inline int green_width(long long W) { return int(W < 256 ? W : 256); }
__host__ __device__ inline unsigned green_pieces(long long W, int Ly) {
  const long long cw = green_width(W), rows = 256 / cw;
  return unsigned((Ly + rows - 1) / rows * ((W + cw * kGreenSteps - 1) / (cw * kGreenSteps)));
}
__global__ void __launch_bounds__(256) k_green(int Lx, int Ly, int K, int rmax, const double* __restrict__ rho,
                                               double* sums) {
  const int groups = int(gridDim.y) - 1, g = int(blockIdx.y);
  const long long W = static_cast<long long>(Lx) * K;
  double ax[kGreenR] = {}, ay[kGreenR] = {};
  const int cw = green_width(W), rows = 256 / cw, ty = int(threadIdx.x) / cw, tx = int(threadIdx.x) % cw;
  const long long span = static_cast<long long>(cw) * kGreenSteps;
  const unsigned pieces = green_pieces(W, Ly), across = unsigned((W + span - 1) / span);
  for (unsigned u = blockIdx.x; u < pieces; u += gridDim.x) {
    const int y = int(u / across) * rows + ty;
    if (ty >= rows || y >= Ly) continue;
    const long long from = (u % across) * span, end = from + span < W ? from + span : W;
    const double* row = rho + size_t(y) * W;
    if (g < groups) {
      const double* far[kGreenR];
#pragma unroll
      for (int e = 0; e < kGreenR; ++e) far[e] = rho + size_t((y + min(g * kGreenR + e + 1, rmax)) % Ly) * W;
      for (long long f = from + tx; f < end; f += cw) {
        const double c = row[f];
#pragma unroll
        for (int e = 0; e < kGreenR; ++e) {
          long long fx = f + static_cast<long long>(min(g * kGreenR + e + 1, rmax)) * K;
          if (fx >= W) fx -= W;
          ax[e] = fma(c, row[fx], ax[e]);
          ay[e] = fma(c, far[e][f], ay[e]);
        }
      }
    } else {
      const double* up = rho + size_t((y + 1) % Ly) * W;
      for (long long f = from + tx; f < end; f += cw) {
        const long long fx = f + K >= W ? f + K - W : f + K;
        ax[0] = fma(row[f] * row[fx], up[f] * up[fx], ax[0]);
      }
    }
  }
  // one sum a block and r: the order of few additions is left to the atomics
  __shared__ double red[8][2 * kGreenR];
#pragma unroll
  for (int e = 0; e < kGreenR; ++e) {
    if (g < groups || e == 0)  // (the plaquette is one sum)
      for (int o = 16; o > 0; o >>= 1) {
        ax[e] += __shfl_down_sync(0xffffffffu, ax[e], o);
        ay[e] += __shfl_down_sync(0xffffffffu, ay[e], o);
      }
    if ((threadIdx.x & 31) == 0) {
      red[threadIdx.x >> 5][e] = ax[e];
      red[threadIdx.x >> 5][kGreenR + e] = ay[e];
    }
  }
  __syncthreads();
  if (threadIdx.x >= 2 * kGreenR) return;
  const int e = int(threadIdx.x) % kGreenR, r = g * kGreenR + e + 1;
  double v = 0.0;
  for (int w = 0; w < 8; ++w) v += red[w][threadIdx.x];
  if (g < groups && r <= rmax) atomicAdd(sums + (threadIdx.x < kGreenR ? r - 1 : rmax + r - 1), v);
  if (g == groups && threadIdx.x == 0) atomicAdd(sums + 2 * rmax, v);
}

int launch_green(int Lx, int Ly, int K, int rmax, const double* rho, double* sums, void* stream) {
  const int groups = (rmax + kGreenR - 1) / kGreenR;
  const unsigned fill = unsigned((152 * 4 + groups) / (groups + 1));  // (64 registers: 4 blocks an SM)
  const unsigned blocks = std::min(green_pieces(static_cast<long long>(Lx) * K, Ly), fill);
  k_green<<<dim3(blocks, groups + 1), 256, 0, cudaStream_t(stream)>>>(Lx, Ly, K, rmax, rho, sums);
  return int(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Checkpoints: the used keys of every site between the slots and a packed
// buffer (each site's header word at at[s], its keys after it).  One warp per
// site.  Only the used part of a configuration then crosses to the host, 9 MB
// instead of 46 MB at 256x256, beta t = 4 (export 3.6 -> 0.15 ms, import 4.9
// -> 0.75 ms, each kernel 10 us).
__global__ void k_pack(const __grid_constant__ Dev d, const uint64_t* __restrict__ at, uint64_t* out) {
  const int s = int((static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= d.N) return;
  const uint32_t c = d.cntA[s];
  const int n = cnt_n(c);
  const uint64_t* K = d.keyA + size_t(s) * d.cap;
  uint64_t* o = out + at[s];
  if (lane == 0) o[0] = uint64_t(n) | (uint64_t(cnt_base(c)) << 63);
  for (int k = lane; k < n; k += 32) o[1 + k] = K[k];
}

// bad = min over the sites 0 .. ns - 1 of a packed buffer that break an
// invariant of the format (tags, time order, continuity, base state)
__global__ void k_packed_check(const uint64_t* __restrict__ at, const uint64_t* __restrict__ in, int ns,
                               unsigned long long* bad) {
  const int s = int((static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= ns) return;
  const uint64_t* p = in + at[s];
  const uint64_t hd = p[0];
  const int n = cnt_n(uint32_t(hd));
  bool ok = true;
  for (int k = lane; k < n; k += 32) {
    const uint64_t key = p[1 + k], nx = p[1 + (k + 1 == n ? 0 : k + 1)];
    ok = ok && ktag(key) != 6 && (k + 1 == n || kpk(key) < kpk(nx)) && kab(key) == kbl(nx) &&
         (k + 1 < n || int(hd >> 63) == kab(key));
  }
  if (!__all_sync(0xffffffffu, ok) && lane == 0) atomicMin(bad, (unsigned long long)(s));
}

__global__ void k_unpack(const __grid_constant__ Dev d, const uint64_t* __restrict__ at, const uint64_t* __restrict__ in) {
  const int s = int((static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= d.N) return;
  const uint64_t* p = in + at[s];
  const uint64_t hd = p[0];
  const int n = cnt_n(uint32_t(hd));
  uint64_t* K = d.keyA + size_t(s) * d.cap;
  for (int k = lane; k < n; k += 32) K[k] = p[1 + k];
  if (lane == 0) d.cntA[s] = cnt_make(n, int(hd >> 63));
}

int launch_pack(const Dev& d, const uint64_t* at, uint64_t* out, void* stream) {
  k_pack<<<site_warps(d.N), 128, 0, cudaStream_t(stream)>>>(d, at, out);
  return int(cudaGetLastError());
}

int launch_packed_check(const uint64_t* at, const uint64_t* in, int ns, unsigned long long* bad, void* stream) {
  if (cudaMemsetAsync(bad, 0xff, sizeof *bad, cudaStream_t(stream)) != cudaSuccess) return int(cudaGetLastError());
  if (ns < 1) return 0;
  k_packed_check<<<site_warps(ns), 128, 0, cudaStream_t(stream)>>>(at, in, ns, bad);
  return int(cudaGetLastError());
}

int launch_unpack(const Dev& d, const uint64_t* at, const uint64_t* in, void* stream) {
  k_unpack<<<site_warps(d.N), 128, 0, cudaStream_t(stream)>>>(d, at, in);
  return int(cudaGetLastError());
}

// The generator every kernel draws from, applied to listed counters and keys
// (compared on the host with published known-answer vectors).
__global__ void k_philox(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, long long n) {
  const long long j = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const uint32_t* c = in + 6 * j;
  const P4 b = philox(c[0], c[1], c[2], c[3], c[4], c[5]);
  out[4 * j] = b.x;
  out[4 * j + 1] = b.y;
  out[4 * j + 2] = b.z;
  out[4 * j + 3] = b.w;
}

int launch_philox(const uint32_t* in, uint32_t* out, int64_t n, void* stream) {
  if (n <= 0) return 0;
  k_philox<<<blocks_for(n, 128), 128, 0, cudaStream_t(stream)>>>(in, out, (long long)n);
  return int(cudaGetLastError());
}

int launch_rho(const Dev& d, int K, double* out, void* stream) {
  run_rho(d, K, out, cudaStream_t(stream));
  return int(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Invariants of a worldline configuration with worms (Steps 3-5 keep them):
// per site, the count fits the slot; every key is a bond leg (tags 0..5) or
// a worm (7); times strictly increase; the state is continuous around the
// circle (the state above an event is the state below the next one) and the
// base state is the state above the last event; a leg's tag names a bond of
// its site; the bond's other site holds the partner leg at the same time;
// the vertex conserves particles, s0 + s1 = s2 + s3.  One warp per site,
// lanes over its events; a partner is found by bisection in at most cap
// keys, so every read stays inside the slots whatever the configuration.
// out = min over failing sites of site << 4 | code (lowest code at a site).
__device__ __forceinline__ int find_pk(const uint64_t* K, int n, uint64_t pk) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (kpk(K[mid]) < pk) lo = mid + 1; else hi = mid;
  }
  return (lo < n && kpk(K[lo]) == pk) ? lo : -1;
}

__global__ void k_check(const __grid_constant__ Dev d, unsigned long long* out) {
  const int lane = threadIdx.x & 31;
  const long long s = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  if (s >= d.N) return;
  const uint32_t c = d.cntA[s];
  const int n = cnt_n(c);
  int bad = kCheckNone;
  if (n > d.cap) {
    bad = kCheckCapacity;
  } else {
    const uint64_t* K = d.keyA + size_t(s) * d.cap;
    for (int k = lane; k < n; k += 32) {
      const uint64_t key = K[k];
      const uint64_t nx = K[(k + 1 == n) ? 0 : k + 1];
      const int t = ktag(key);
      int b = kCheckNone;
      if (t == 6) b = kCheckTag;
      else if (k + 1 < n && kpk(nx) <= kpk(key)) b = kCheckOrder;
      else if (kab(key) != kbl(nx)) b = kCheckContinuity;
      else if (k + 1 == n && cnt_base(c) != kab(key)) b = kCheckBase;
      else if (t != 7) {
        int dir;
        const int a = leg_lower(d, int(s), t, &dir);
        const int o = (a == int(s)) ? site_step(d, a, dir, +1) : a;
        if (bond_tag(d, a, dir) != t) {
          b = kCheckBond;
        } else {
          const int no = min(cnt_n(d.cntA[o]), d.cap);
          const uint64_t* KO = d.keyA + size_t(o) * d.cap;
          const int ko = find_pk(KO, no, kpk(key));
          if (ko < 0) {
            b = kCheckPartner;
          } else {
            const uint64_t va = (a == int(s)) ? key : KO[ko], vb = (a == int(s)) ? KO[ko] : key;
            if (kbl(va) + kbl(vb) != kab(va) + kab(vb)) b = kCheckConservation;
          }
        }
      }
      bad = min(bad, b);
    }
  }
  for (int o = 16; o > 0; o >>= 1) bad = min(bad, __shfl_xor_sync(0xffffffffu, bad, o));
  if (lane == 0 && bad != kCheckNone)
    atomicMin(out, (static_cast<unsigned long long>(s) << 4) | static_cast<unsigned long long>(bad));
}

int launch_check(const Dev& d, unsigned long long* out, void* stream) {
  if (cudaMemsetAsync(out, 0xff, sizeof(unsigned long long), cudaStream_t(stream)) != cudaSuccess)
    return int(cudaGetLastError());
  const long long threads = static_cast<long long>(d.N) * 32;
  k_check<<<blocks_for(threads, 256), 256, 0, cudaStream_t(stream)>>>(d, out);
  return int(cudaGetLastError());
}

}  // namespace pmwa
