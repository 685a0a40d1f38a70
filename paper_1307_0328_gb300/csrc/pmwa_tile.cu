// pmwa_tile.cu -- Steps 3-6 of one MC sweep in a single kernel: one CTA per
// domain, the domain's vertex legs and worms resident in shared memory.
//
//   phase 1  Step 3 candidates, one thread per bond of the domain, written to
//            a shared pool (the current configuration is read from a staged
//            copy in shared memory where it fits, else from HBM/L2, prefetched
//            into L2 by bulk copies at kernel start)
//   phase 2  per site, or per part of a site's circle: the kept vertex legs of
//            the current configuration merged in time order with the new ones
//            into the shared leg array
//   phase 3  Step 4, one thread per site, a random word a step: worms of every
//            interval (Eq. 1) into the shared worm table; each worm records its
//            site and the index of the vertex leg just below it (its interval)
//   phase 4  Step 5, N_cycle passes of the shifted sub-block schedule: the
//            worms of a sub-block move in label order (Eq. 2); a move waits
//            only for the earlier ones whose intervals meet its own, which
//            gives the moves made one by one; vertex legs never move in
//            Step 5, so a move is a handful of shared-memory reads and two
//            bit flips.  What bounds it is the length of one move's dependent
//            chain times the few moves that follow one another in a pass
//            (3 to 12 of a CTA's warps have work, 0.3 instructions a cycle),
//            so a pass has one barrier, lengths are 32-bit differences where
//            these decide, and a worm looks for its next vertex while others
//            still move.  One 16x16-site domain, cycles a pass: 10.1k -> 6.4k
//            at beta t = 4 (95 worms), 19.6k -> 10.9k at beta t = 16 (381
//            worms); an 8x8 domain of one group (22 worms): 19.0k -> 5.4k
//   phase 5  legs and worms, each at its counted place, into the next
//            configuration in HBM, with the Step-6 counters and the Supplement S-I estimator
//
// The arithmetic and the order of every random draw are those of the
// deterministic specification, so the result is bit-identical to the CPU
// reference for every domain layout.
#include <cuda_runtime.h>

#include <algorithm>

#include "pmwa_device.cuh"

namespace pmwa {

namespace {

constexpr int kMaxCandPerBond = 128;
constexpr int kMaxWormsPerInterval = 128;
constexpr uint16_t kNone = 0xFFFF;
constexpr uint32_t kCntMask = 0x7fffffffu;
constexpr uint64_t kMask62 = kTwo62 - 1;
constexpr int kSms = 152;
constexpr int kSmemLimit = 232448;  // opt-in shared memory per block on sm_103a

struct WormRec {
  uint64_t key;
  uint64_t lab;   // label (Step 4)
  uint16_t site;  // local site index
  uint16_t leg;   // leg array index of the delimiter just below (kNone: site without legs)
  uint16_t slab;  // temporal slab (0 without temporal domains); fixed through Step 5
  uint16_t pad;
};

struct Misc {
  int pool_used;
  int nworms;
  int err;
  int where;
  int wslab[64];  // worms of each temporal slab of the domain
};

__device__ __forceinline__ int cnt_n(uint32_t c) { return int(c & kCntMask); }

// bulk prefetch of `bytes` (a multiple of 16) from a 16-byte aligned global
// address into L2 (TMA engine; no registers, no completion to wait for)
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %0;\n\tcp.async.bulk.prefetch.L2.global [ga], %1;\n\t}"
               :: "l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ int cnt_base(uint32_t c) { return int(c >> 31); }

__device__ __forceinline__ void tile_fail(Misc* m, int code, int where) {
  if (atomicCAS(&m->err, 0, code) == 0) m->where = where;
}

// item of thread tid when n <= NT items are spread over the warps (n: none);
// tid when there are more
__device__ __forceinline__ int spread(int tid, int NT, int n) {
  if (n >= NT) return tid;
  const int warps = NT >> 5, per = (n + warps - 1) / warps, lane = tid & 31;
  return lane < per ? (tid >> 5) * per + lane : n;
}

// exclusive scan of a[0..n) in place (a[n] receives the total); all threads
__device__ int block_scan(int* a, int n, int* wsum) {
  const int t = threadIdx.x, T = blockDim.x, lane = t & 31, wid = t >> 5, nw = T >> 5;
  const int chunk = (n + T - 1) / T;
  const int lo = min(n, t * chunk), hi = min(n, lo + chunk);
  int sum = 0;
  for (int i = lo; i < hi; ++i) sum += a[i];
  int v = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) wsum[wid] = v;
  __syncthreads();
  if (wid == 0) {
    int w = (lane < nw) ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += u;
    }
    if (lane < nw) wsum[lane] = w;
  }
  __syncthreads();
  int run = v - sum + (wid ? wsum[wid - 1] : 0);
  for (int i = lo; i < hi; ++i) { const int x = a[i]; a[i] = run; run += x; }
  const int total = wsum[nw - 1];
  __syncthreads();
  if (t == 0) a[n] = total;
  __syncthreads();
  return total;
}

struct Tile {
  const Dev* d;
  uint32_t* th;    // [256] directed-loop thresholds, 2^32 held as 2^32 - 1
  int* off;        // [nds + 1] start of each site's legs in leg[]
  uint8_t* base;   // [nds] state of a site without legs
  int* bcnt;       // [2 nds] candidates per bond of the domain
  uint32_t* rng;   // [nds] (bcnt, once the legs are merged) first leg | end << 16 of each site
  int* boff;       // [2 nds] their start in pool[]
  int* perr;       // [2] (boff, once the legs are merged) a status found in an even / odd pass of Step 5
  Misc* misc;
  uint64_t* leg;   // [legcap]
  uint8_t* wcnt;   // [legcap] worms in the interval just above each leg
  uint16_t* part;  // [legcap] index of the partner leg of each leg's vertex (kNone: none in the domain)
  uint64_t* pool;  // [poolcap] (aliases the worm table)
  WormRec* W;      // [wcap]
  uint16_t* idx;   // [wcap] (nxt) worms by label bucket before Step 5, by site after it
  uint16_t* ord;   // [wcap] worm indices in label order (lab, site, key)
  uint16_t* dn;    // [wcap] stamp of the last pass in which the k-th worm in label order has moved
  // (two buffers each, for even and odd passes)
  uint16_t* nxt;   // [2 wcap] the worm after the k-th one in its group's list
  uint32_t* fp;    // [2 wcap] the vertex the k-th worm's move reaches
  uint32_t* hd;    // [hstride + groups] (bkt, fill) head of each group's list: pass stamp << 16 | worm
  int hstride;     // from the even passes' heads to the odd ones'
  uint16_t* cell;  // [2 groups x 8] the first members of each group
  uint32_t* hash;  // [2 ghash] heads of the chains of worms by leg: pass stamp << 16 | entry
  int* gcnt;       // [3 groups] members of each group (three passes in turn)
  int* bkt;        // [max(nsub, nds) + 1]
  int* fill;       // [max(nsub, nds)]
  uint16_t* nbr;   // [6 nds] per leg tag: the bond's other site (0 when it leaves the domain)
  uint8_t* tinfo;  // [6 nds] per leg tag: 1 = lower site of the bond, 2 = bond leaves the domain,
                   // 4 << q = both sites in one sub-block in pass pattern q
  uint16_t* sub;   // [4 nds] sub-block of each site for offset pattern pass & 3
  int* soff;       // [nds + 1] start of each site's events in old[] (when staged)
  uint64_t* old;   // [oldcap] the domain's current configuration (when staged)
  int* wmo;        // [nds + 1] on-the-fly windows: start of each site's old worms in wm[]
  uint64_t* wm;    // [wcap] grid points of the current configuration's worms, by site
  bool staged;     // the current configuration is in old[]
  bool early;      // it is in leg[] (from off[li] on for site li) until the merge
  int x0, y0, nds, nsub;
  int ngrp;  // Step-5 chains: sub-blocks x temporal slabs

  __device__ int gsite(int li) const { return (x0 + li % d->dom_x) + d->Lx * (y0 + li / d->dom_x); }
  // current events of local site li (global site s): the staged copy or HBM
  __device__ const uint64_t* okeys(int li, int s) const {
    return staged ? old + soff[li] : d->keyA + size_t(s) * d->cap;
  }
  // the same before the merge writes legs: the copy in the leg table too
  __device__ const uint64_t* okeys_early(int li, int s) const { return early ? leg + off[li] : okeys(li, s); }
  __device__ int lsite(int s) const { return (s % d->Lx - x0) + d->dom_x * (s / d->Lx - y0); }
  __device__ int sub_of(int li, int pass) const {
    const int B = d->sub_block;
    const int ox = (B && B < d->dom_x) ? (pass & 1) * (B / 2) : 0;
    const int oy = (B && B < d->dom_y) ? ((pass >> 1) & 1) * (B / 2) : 0;
    const int bx = sb_axis(li % d->dom_x, d->dom_x, B, d->ndx, ox);
    const int by = sb_axis(li / d->dom_x, d->dom_y, B, d->ndy, oy);
    return bx + sb_slots(d->dom_x, B, d->ndx) * by;
  }
};

// On-the-fly vertex generation (the paper's closing discussion of
// extensions): with d.win_half > 0 the vertex phase of a bond is confined to
// the grid points within win_half of a worm of the current configuration on
// either of its two sites (cyclic).  R depends on the worms alone, which
// Step 3 does not move, so the restricted heat bath keeps the distribution.
__device__ __forceinline__ bool in_win(const Tile& T, int li, uint64_t pos) {
  const uint64_t half = T.d->win_half;
  for (int k = T.wmo[li]; k < T.wmo[li + 1]; ++k) {
    const uint64_t a = (pos - T.wm[k]) & (kTwo59 - 1), b = (T.wm[k] - pos) & (kTwo59 - 1);
    if (min(a, b) <= half) return true;
  }
  return false;
}

// ---------------------------------------------------------------------------
// phase 1: Step 3 candidates of bond (a, dir) from the current configuration
// (with OTF, only inside the windows of the bond's local sites la, lb)
template <bool OTF>
__device__ int bond_candidates(const Dev& d, const ZigTab& z, int a, int dir, const uint64_t* KA, const uint64_t* KB,
                               uint64_t* buf, int cap, int* bad, const Tile* T, int la, int lb) {
  const int b = site_step(d, a, dir, +1);
  const uint64_t tag = uint64_t(bond_tag(d, a, dir));
  const uint32_t ca = d.cntA[a], cb = d.cntA[b];
  const int nA = cnt_n(ca), nB = cnt_n(cb);
  Stream s;
  s.init(d.key0, d.key1, uint32_t(2 * a + dir), c2_word(kVertex, 0, d.replica), d.sweep);
  int n = 0, ia = 0, ib = 0;
  uint64_t pos = 0;
  bool first = true;
  for (;;) {
    const uint64_t E = zig_exp(z, s, bad);
    if (*bad) break;
    const uint64_t g = grid_gap(E, d.SVs);
    const uint64_t nxt = first ? g - 1 : pos + g;
    first = false;
    if (nxt >= kTwo59) break;
    pos = nxt;
    if (OTF && !(in_win(*T, la, pos) || in_win(*T, lb, pos))) continue;
    const uint64_t pk = (pos << 3) | tag;
    while (ia + 4 <= nA && kpk(KA[ia + 3]) < pk) ia += 4;
    while (ia < nA && kpk(KA[ia]) < pk) ++ia;
    while (ib + 4 <= nB && kpk(KB[ib + 3]) < pk) ib += 4;
    while (ib < nB && kpk(KB[ib]) < pk) ++ib;
    if (ia < nA && kpk(KA[ia]) == pk && kab(KA[ia]) != kbl(KA[ia])) continue;  // a kink holds the point
    const int na = nA ? kab(KA[ia ? ia - 1 : nA - 1]) : cnt_base(ca);
    const int nb = nB ? kab(KB[ib ? ib - 1 : nB - 1]) : cnt_base(cb);
    const int si = na | (nb << 1);
    if (d.TV[si] < kTwo32) {
      const uint64_t w = s.word();
      if ((w >> 32) >= d.TV[si]) continue;
    }
    if (n >= cap) { *bad = PMWA_ECAPACITY; break; }
    buf[n++] = (pk << 2) | uint64_t(na) | (uint64_t(nb) << 1);
  }
  return n;
}

// old event of local site li kept by Step 3: a kink, any leg of a bond
// between domains, and (OTF) a diagonal leg outside the windows of its bond
template <bool OTF>
__device__ __forceinline__ bool kept_leg(const Tile& T, int li, uint64_t k) {
  if (kworm(k)) return false;
  if (kab(k) != kbl(k)) return true;
  if (T.tinfo[li * 6 + ktag(k)] & 2) return true;
  if (OTF) {
    const uint64_t pos = kpk(k) >> 3;
    return !(in_win(T, li, pos) || in_win(T, T.nbr[li * 6 + ktag(k)], pos));
  }
  return false;
}

// the four bonds of local site li: (s,x) (s,y) with s the lower site, then
// (s-x,x) (s-y,y) with s the upper site; local bond id or -1 (between domains)
__device__ __forceinline__ void site_bonds(const Tile& T, int li, int lb[4]) {
  const Dev& d = *T.d;
  const int s = T.gsite(li);
  for (int j = 0; j < 4; ++j) {
    const int dir = j & 1;
    const int a = (j < 2) ? s : site_step(d, s, dir, -1);
    lb[j] = boundary_bond(d, a, dir) ? -1 : 2 * T.lsite(a) + dir;
  }
}

// ---------------------------------------------------------------------------
// phase 4: Step-5 moves.
//
// index of the leg at time point pv on site x (-1: none).  A step tells apart
// four parts by three loads that do not wait for one another: half the
// dependent steps of a bisection.
__device__ __forceinline__ int leg_index(const Tile& T, int x, uint64_t pv) {
  const int en = T.off[x + 1];
  const uint64_t key = pv << 2;  // (kpk(k) < pv exactly when k < pv << 2)
  int lo = T.off[x], n = en - lo;
  while (n > 3) {
    const int q = n >> 2;
    const uint64_t k1 = T.leg[lo + q], k2 = T.leg[lo + 2 * q], k3 = T.leg[lo + 3 * q];
    // the first leg not below pv lies behind the last of the three that is below it, and not
    // behind the next one
    const int j = int(k1 < key) + int(k2 < key) + int(k3 < key);
    n = (j == 0) ? q : (j == 3) ? n - 3 * q - 1 : q - 1;
    lo += j * q + (j ? 1 : 0);
  }
  while (n > 0 && T.leg[lo] < key) { ++lo; --n; }
  return (lo < en && kpk(T.leg[lo]) == pv) ? lo : -1;
}

// A worm's vertex as the two legs of it, iv | ip << 16, or kTurn | its own
// interval when it turns round whatever the others do (no leg has index 2^16 - 1)
constexpr uint32_t kTurn = 0xffff0000u;
__device__ __forceinline__ bool turns(uint32_t fp) { return fp >= kTurn; }

// What a Step-5 move reaches: the vertex v ahead of the worm, on the worm's
// own site and on the bond's other site.  Legs never move in Step 5, so all
// of it but the vertex's states can be formed before the moves the worm waits
// for have run.
//
// Lengths here are differences of the high words of the keys, in units of
// 2^-32 of the circle (they wrap as the circle does): within one unit of the
// true length unless they come out as 0 (which is a length below one unit, or
// the whole circle but less than one unit).
struct Ahead {
  uint32_t fp;        // v's legs on the own and the other site, iv | ip << 16 (kTurn: none)
  uint32_t dns, ups;  // the legs below and above v on both sites: i_dn | p_dn << 16, i_up | p_up << 16
                      // (an interval is named by its lower leg: the four round v are dns and fp)
  uint64_t kv;        // v's leg on the own site
  uint32_t id, iu, pd, pu;      // lengths of v's legs down and up, own and other site, with no worm on them
  uint32_t lid, liu, lpd, lpu;  // low words of the keys that end them
  int pl, b;                    // the other site; 1 when the worm's site is the upper one of the bond
};

// The vertex that the Step-5 move of a worm (key, local site li, interval
// L) reaches in pass pattern q.  fp >= kTurn: the worm turns round whatever
// the other worms do (a site without legs, a temporal boundary, a bond to
// another domain or sub-block).  Returns PMWA_EINVARIANT when the vertex has
// no partner leg on the other site.
__device__ __forceinline__ int look_ahead(const Tile& T, uint64_t key, int li, int L, int q, Ahead& o) {
  o.fp = kTurn | uint32_t(L);
  const uint32_t rs = T.rng[li];
  const int st = rs & 0xffff, en = rs >> 16;
  if (st == en) return PMWA_OK;
  const int iv = kdir(key) ? ((L + 1 == en) ? st : L + 1) : L;
  const uint64_t kv = T.leg[iv];
  const int tag = ktag(kv);
  if (tag == 6) return PMWA_OK;
  const int info = T.tinfo[li * 6 + tag], pl = T.nbr[li * 6 + tag];
  if (!((info >> (q + 2)) & 1)) return PMWA_OK;
  const uint32_t rp = T.rng[pl];
  const int ip = T.d->use_part ? (T.part[iv] == kNone ? -1 : int(T.part[iv])) : leg_index(T, pl, kpk(kv));
  if (ip < 0) return PMWA_EINVARIANT;
  const int sp = rp & 0xffff, ep = rp >> 16;
  const int i_dn = (iv == st ? en : iv) - 1, i_up = (iv + 1 == en) ? st : iv + 1;
  const int p_dn = (ip == sp ? ep : ip) - 1, p_up = (ip + 1 == ep) ? sp : ip + 1;
  const uint64_t kid = T.leg[i_dn], kiu = T.leg[i_up], kpd = T.leg[p_dn], kpu = T.leg[p_up];
  const uint32_t hv = uint32_t(kv >> 32);
  const bool i1 = i_dn == iv, p1 = p_dn == ip;  // v alone on its site: its legs are the whole circle
  o.id = i1 ? ~0u : hv - uint32_t(kid >> 32);
  o.iu = i1 ? ~0u : uint32_t(kiu >> 32) - hv;
  o.pd = p1 ? ~0u : hv - uint32_t(kpd >> 32);
  o.pu = p1 ? ~0u : uint32_t(kpu >> 32) - hv;
  o.lid = uint32_t(kid);
  o.liu = uint32_t(kiu);
  o.lpd = uint32_t(kpd);
  o.lpu = uint32_t(kpu);
  o.fp = uint32_t(iv) | (uint32_t(ip) << 16);
  o.kv = kv;
  o.dns = uint32_t(i_dn) | (uint32_t(p_dn) << 16);
  o.ups = uint32_t(i_up) | (uint32_t(p_up) << 16);
  o.pl = pl;
  o.b = (info & 1) ^ 1;
  return PMWA_OK;
}

// What a Step-5 move decides and the exact lengths of v's legs (own site down,
// other site down, own up, other up), in full words, for a move whose 32-bit
// lengths leave a doubt: worm k at (key, interval L), nw worms.  Only worms of v's
// four intervals count, and the interval's leg names them, so all of the domain's
// are looked at.  Out of line, as it is rare and a move's code long.
struct Exact {
  bool blocked, enter;
  uint64_t E0, E1, E2, E3;
};
__device__ __noinline__ Exact exact_lengths(const uint64_t* leg, const WormRec* W, int k, int nw, uint32_t fp,
                                            uint32_t dns, uint32_t ups, uint64_t kv, uint64_t key, int L,
                                            uint32_t z1) {
  const int iv = int(fp & 0xffff), ip = int(fp >> 16), i_dn = int(dns & 0xffff), p_dn = int(dns >> 16);
  const bool up = kdir(key);
  const uint64_t pv = kpk(kv), my = up ? (pv - kpk(key)) & kMask62 : (kpk(key) - pv) & kMask62;
  Exact x;
  x.E0 = wpts(kpk(leg[i_dn]), pv);
  x.E1 = wpts(kpk(leg[p_dn]), pv);
  x.E2 = wpts(pv, kpk(leg[ups & 0xffff]));
  x.E3 = wpts(pv, kpk(leg[ups >> 16]));
  x.blocked = false;
  for (int e = 0; e < nw; ++e) {
    if (e == k) continue;
    const int lg = W[e].leg;
    const uint64_t po = kpk(W[e].key);
    if (lg == L && (up ? ((pv - po) & kMask62) < my : ((po - pv) & kMask62) < my)) x.blocked = true;
    if (lg == iv) x.E2 = min(x.E2, wpts(pv, po));
    if (lg == ip) x.E3 = min(x.E3, wpts(pv, po));
    if (lg == i_dn) x.E0 = min(x.E0, wpts(po, pv));
    if (lg == p_dn) x.E1 = min(x.E1, wpts(po, pv));
  }
  // enter iff z1 * L_i < L_min * 2^32 (96-bit comparison)
  const uint64_t Li = up ? x.E0 : x.E2, lo = uint64_t(z1) * (Li & 0xffffffffull);
  x.enter = uint64_t(z1) * (Li >> 32) + (lo >> 32) < min(min(x.E0, x.E1), min(x.E2, x.E3));
  return x;
}

// The Step-5 move of worm k of nw (key, site li, interval L; updated here) to
// the vertex v of `o`.  each(f) calls f(leg, key) for (at least) every other
// worm in v's four intervals; it is used only when there is one.  The worm
// reverses at another worm ahead of it in its interval; otherwise it enters v
// with probability L_min / L_i (w0 >> 32 against the exact ratio), leaves by
// leg j (threshold table, low half of w0) and lands on a uniform worm grid
// point of leg j (mulhi of w1) heading away from v.  Leg l of v runs from v
// to the nearest event on its site and side (another vertex leg or worm, the
// moving worm excluded; the whole circle if none).
//
// The order of the worms, L_min and the enter test are decided on the 32-bit
// lengths wherever these leave no doubt (each within one unit of the exact
// one); a doubt -- two times with one high word, a test within three units
// -- costs the 64-bit computation (legs of 2^32 / n units on sites of n legs, four
// of which and the test leave a doubt within a few units each: about 20 n / 2^32
// of the moves, 1 in 10^7 at beta t = 4, 1 in 10^6 at 188 legs).  Only the landing
// point needs the exact length, of leg j alone.  A domain's passes keep few
// warps busy, so a move is one dependent chain and its cost is latency: the
// branches are the rare cases only, the loads stand together up front.
template <class Each>
__device__ __forceinline__ void make_move(const Tile& T, const Ahead& o, uint64_t& key, int& li, int& L, uint64_t w0,
                                          uint64_t w1, int k, int nw, Each each) {
  const int iv = int(o.fp & 0xffff), ip = int(o.fp >> 16), i_dn = int(o.dns & 0xffff), p_dn = int(o.dns >> 16);
  const uint64_t vi = T.leg[iv], vp = T.leg[ip];
  const int c0 = T.wcnt[i_dn], c1 = T.wcnt[p_dn], c2 = T.wcnt[iv], c3 = T.wcnt[ip];
  const bool up = kdir(key);
  const uint32_t hv = uint32_t(o.kv >> 32);
  uint32_t id = o.id, iu = o.iu, pd = o.pd, pu = o.pu;
  uint32_t lid = o.lid, liu = o.liu, lpd = o.lpd, lpu = o.lpu;
  int ends = 0;  // legs ended by a worm: 1 own down, 2 own up, 4 other down, 8 other up
  bool blocked = false, doubt = false;
  // legs by number: 0 / 1 the lower / upper site below v, 2 / 3 above
  const int i = o.b | (up ? 0 : 2);
  const uint32_t sa = uint32_t(o.b ? vp : vi), sb = uint32_t(o.b ? vi : vp);
  const int S = int((sa >> 1) & 1) | int(sb & 2) | (int(sa & 1) << 2) | (int(sb & 1) << 3);
  const uint4 th = reinterpret_cast<const uint4*>(T.th)[S * 4 + i];
  const bool others = c2 + c3 + (i_dn != iv ? c0 : 0) + (p_dn != ip ? c1 : 0) > 1;
  if (others) {
    const uint32_t my = up ? hv - uint32_t(key >> 32) : uint32_t(key >> 32) - hv;  // from the worm to v
    doubt = my == 0;
    each([&](int lg, uint64_t ko) {
      const uint32_t x = uint32_t(ko >> 32) - hv, y = 0u - x, lo = uint32_t(ko);  // from v up and down to the worm
      const uint32_t z = up ? y : x;
      blocked |= lg == L && z < my;
      doubt |= lg == L && z == my;
      if (lg == iv && x <= iu) { doubt |= x == iu; iu = x; liu = lo; ends |= 2; }
      if (lg == ip && x <= pu) { doubt |= x == pu; pu = x; lpu = lo; ends |= 8; }
      if (lg == i_dn && y <= id) { doubt |= y == id; id = y; lid = lo; ends |= 1; }
      if (lg == p_dn && y <= pd) { doubt |= y == pd; pd = y; lpd = lo; ends |= 4; }
    });
  }
  const uint32_t z1 = uint32_t(w0 >> 32), z0 = uint32_t(w0);
  const uint32_t lmin = min(min(id, iu), min(pd, pu));
  // z1 L_i / 2^32 against L_min, each side within 2 units below or above
  const long long slack = (long long)lmin - (long long)__umulhi(z1, up ? id : iu);
  bool enter = slack >= 3;
  doubt |= lmin < 4 || (slack < 3 && slack > -2);
  int j = int(z0 >= th.x) + int(z0 >= th.y) + int(z0 >= th.z);
  if (z0 == ~0u) {  // (the table holds thresholds up to 2^32 - 1: a 2^32 counts from the full one)
    const uint64_t* t = T.d->TH + (S * 4 + i) * 4;
    j = int(z0 >= t[0]) + int(z0 >= t[1]) + int(z0 >= t[2]);
  }
  const bool ju = j >= 2, jo = ((j ^ o.b) & 1) == 0;  // leg j goes up; lies on the worm's own site
  const int dn = jo ? i_dn : p_dn, x = jo ? iv : ip;
  const int wj = (ends >> ((jo ? 0 : 2) + (ju ? 1 : 0))) & 1;
  // exact length of leg j: the high-word difference and the low words, grid points times 32
  const uint32_t hj = jo ? (ju ? iu : id) : (ju ? pu : pd), lj = (jo ? (ju ? liu : lid) : (ju ? lpu : lpd)) & ~31u;
  const uint32_t lv = uint32_t(o.kv) & ~31u;
  const uint64_t dj = (uint64_t(hj) << 32) + (ju ? uint64_t(lj) - lv : uint64_t(lv) - lj);
  uint64_t Lj = (dj >> 5) - (ju ? 0 : wj);
  if (dn == x && !wj) Lj = kTwo59;
  if (doubt) {
    const Exact x = exact_lengths(T.leg, T.W, k, others ? nw : 0, o.fp, o.dns, o.ups, o.kv, key, L, z1);
    blocked = x.blocked;
    enter = x.enter;
    Lj = jo ? (ju ? x.E2 : x.E0) : (ju ? x.E3 : x.E1);
  }
  const uint64_t at = __umul64hi(w1, Lj);
  // the worm leaves leg i and takes leg j: flip their states
  const uint64_t ni = vi ^ (up ? 2u : 1u) ^ (jo ? (ju ? 1u : 2u) : 0u), np = vp ^ (jo ? 0u : (ju ? 1u : 2u));
  const uint32_t vx = uint32_t(jo ? ni : np);
  const uint64_t tv = o.kv & ~31ull;  // (sums of grid points times 32 wrap round the circle by themselves)
  const uint64_t to = ju ? ((tv + (at << 5)) | 30u | ((vx & 1u) ^ 1u)) : ((tv - ((at + 1) << 5)) | 28u | ((vx >> 1) & 1u));
  if (blocked || !enter) { key ^= 2u; return; }
  key = to;
  T.leg[iv] = ni;
  T.leg[ip] = np;
  const int nl = ju ? x : dn;
  if (nl != L) {
    T.wcnt[L] = uint8_t((L == iv ? c2 : c0) - 1);
    T.wcnt[nl] = uint8_t((ju ? (jo ? c2 : c3) : (jo ? c0 : c1)) + 1);
    L = nl;
  }
  li = jo ? li : o.pl;
}

// per-phase cycle counters (profiling only): thread 0 adds the cycles since
// the last tick to counter k
__device__ __forceinline__ void phase_tick(const Dev& d, int k, long long& t) {
  if (d.phase_cycles && threadIdx.x == 0) {
    const long long now = clock64();
    atomicAdd(d.phase_cycles + k, (unsigned long long)(now - t));
    t = now;
  }
}

// Step-5 chain of a worm in pass pattern q: its sub-block times N_beta plus
// its temporal slab (a worm never leaves its slab: it turns round at the
// boundaries and every leg ends there)
__device__ __forceinline__ int worm_group(const Tile& T, int site, int slab, int q) {
  return int(T.sub[site * 4 + q]) * T.d->ntau + slab;
}

// ---------------------------------------------------------------------------
// Independent moves.  In a pass the worms of one sub-block move one
// after another in label order, and a move reads and writes nothing but its
// own worm and the four intervals round the vertex it reaches: their worm
// counts, the worms in them and the states of the vertex's two legs.  A worm
// that turns round whatever the others do changes nothing another move
// reads.  So a move need wait only for the earlier moves of its sub-block
// whose intervals meet its own: running every move as soon as its such
// predecessors have run gives exactly the configuration of the moves made
// one by one.
// Do the intervals round another worm's vertex meet those round this one's?
// On a site they share one iff the other vertex is this one or one of its
// two neighbours there, so both legs of the other (either half of g) are held
// against the legs below, at and above this vertex on both sites, two at a
// time: some half word of x is zero iff (x - 0x00010001) & ~x has a half
// word's top bit set.  For a worm that turns round, g holds its own interval
// and the answer covers every case where that is one of the four.
struct Meet {
  uint32_t a0, a1, a2, c0, c1, c2;
  __device__ __forceinline__ explicit Meet(const Ahead& o) {
    a0 = o.dns; a1 = o.fp; a2 = o.ups;
    c0 = (a0 << 16) | (a0 >> 16); c1 = (a1 << 16) | (a1 >> 16); c2 = (a2 << 16) | (a2 >> 16);  // halves swapped
  }
  __device__ __forceinline__ bool operator()(uint32_t g) const {
    auto z = [](uint32_t x) { return (x - 0x00010001u) & ~x; };
    return ((z(a0 ^ g) | z(a1 ^ g) | z(a2 ^ g) | z(c0 ^ g) | z(c1 ^ g) | z(c2 ^ g)) & 0x80008000u) != 0;
  }
};

__device__ __forceinline__ bool worm_less(const WormRec& a, const WormRec& b) {
  if (a.lab != b.lab) return a.lab < b.lab;
  if (a.site != b.site) return a.site < b.site;
  return a.key < b.key;
}

__device__ __forceinline__ void add128(uint64_t& lo, uint64_t& hi, uint64_t blo, uint64_t bhi) {
  const uint64_t s = lo + blo;
  hi += bhi + (s < lo ? 1 : 0);
  lo = s;
}

// Label order of the nw worms of the domain, (lab, site, key) ascending,
// into ord[]: a counting sort on the top bits of the (uniform 63-bit)
// labels into nbk <= max(nsub, nds) buckets, then each worm's rank inside
// its bucket.  Uses bkt/fill as bucket counters and idx as scratch.
__device__ void label_order(const Tile& T, int nw, int* wsum) {
  const int tid = threadIdx.x, NT = blockDim.x;
  const int cap = max(T.ngrp, T.nds);
  int B = 0;
  while ((2 << B) <= cap && (1 << B) < nw) ++B;
  const int nbk = 1 << B;
  for (int i = tid; i <= nbk; i += NT) T.bkt[i] = 0;
  __syncthreads();
  for (int w = tid; w < nw; w += NT) atomicAdd(&T.bkt[B ? int(T.W[w].lab >> (63 - B)) : 0], 1);
  __syncthreads();
  block_scan(T.bkt, nbk, wsum);
  for (int i = tid; i < nbk; i += NT) T.fill[i] = T.bkt[i];
  __syncthreads();
  for (int w = tid; w < nw; w += NT)
    T.idx[atomicAdd(&T.fill[B ? int(T.W[w].lab >> (63 - B)) : 0], 1)] = uint16_t(w);
  __syncthreads();
  for (int w = tid; w < nw; w += NT) {
    const int b = B ? int(T.W[w].lab >> (63 - B)) : 0;
    const int lo = T.bkt[b], hi = T.bkt[b + 1];
    int r = 0;
    for (int j = lo; j < hi; ++j) r += worm_less(T.W[T.idx[j]], T.W[w]);
    T.ord[lo + r] = uint16_t(w);
  }
  __syncthreads();
}

// The groups of a pass.  A worm that looks ahead for pass p joins its group u:
// it takes the next place of the group's table of kGroupSlots worm numbers
// (numbers in label order), or, when those are taken, puts itself at the head
// of the group's linked list (hd[u] = stamp << 16 | k, the stamp being p + 1,
// so that the heads need no clearing; nxt[k] the worm it found there).
// Two-by-two sub-blocks hold one to five worms: the table brings a group's
// members in one go, where a list is one dependent load after the other.
// Tables and lists alternate between two buffers, the counts between three
// (a pass clears the one that the pass after the next fills).
__device__ __forceinline__ void join_list(const Tile& T, int k, int u, int pass) {
  const uint32_t stamp = uint32_t(pass + 1);
  const uint32_t was = atomicExch(T.hd + (pass & 1) * T.hstride + u, (stamp << 16) | uint32_t(k));
  T.nxt[(pass & 1) * T.d->wcap + k] = (was >> 16) == stamp ? uint16_t(was) : kNone;
}

// a worm's site and interval in one store: a move that runs beside this
// one's reads either the old or the new pair
__device__ __forceinline__ void store_place(WormRec& w, int li, int L) {
  *reinterpret_cast<uint32_t*>(&w.site) = uint32_t(li) | (uint32_t(L) << 16);
}

constexpr int kSpinLimit = 1 << 20;  // polls of a predecessor before the pass gives up (never reached)
constexpr int kNeighbours = 64;      // neighbours that a worm holds one by one
constexpr int kGroupSlots = 8;       // worms of a group's table (16 bits each) at least
// up to so many groups, of more worms on average: scans and chains by leg
constexpr int kScanGroups = 9, kScanMembers = 12;
// worms of a thread at most: a plan of 227 KB and 48 bytes a worm holds 4842,
// 19 for each of 256 threads, and smaller CTAs run domains of fewer worms
// (tile_class: the table of 48 expected worms holds 286, that of 384 825)
constexpr int kMaxTurns = 24;

// All N_cycle passes of a domain of more than 32 worms (called by all
// threads); W[] is in label order.  With at most blockDim.x worms a thread
// keeps its worm k in registers throughout, and the worms are spread over the
// warps, at least 16 a warp: a warp's loops run as long as its slowest lane's,
// but more warps issue more instructions.
//
// With more a thread takes its worms k = tid, tid + blockDim.x, ... in
// turns within each pass and looks ahead anew at a turn's start.  A worm waits
// for smaller k alone, which belong to its own turn or an earlier one of other
// warps, and an earlier turn waits for no later one: every wait ends.
//
// A pass has one barrier.  Behind it every worm goes through its group once,
// for its rank r (the members with a smaller k) and for the members whose
// intervals meet its own (nn of them, four in `mem`, 16 bits each),
// draws its Philox block and moves as soon as the earlier ones of those (bits
// of `deps`) have set their flag dn[] -- no round waits for the slowest worm
// of the domain.  What it reaches in the next pass depends on its own place
// and on leg times alone, so it looks ahead and joins its next group right
// after its move, while other worms still move.
//
// The members of up to kNeighbours neighbours beyond four are listed by the
// thread itself (local memory, in a second round through the group); a worm with
// more looks at every worm of the domain.  Walking the group anew at each poll
// and in the move, and a form for more worms than threads that looked ahead anew
// every round, had made domains of many worms an interval up to 4.0 times
// slower than rounds of precomputed waits (8x8 sites at beta t = 2, eta = 3,
// now 1.8 times as fast as those; 24x24 at beta t = 4, eta = 0.5 in 4x4 blocks
// 2.14 -> 5.02 -> 0.91 ms a sweep).
//
// The groups' tables hold the expected members and three standard deviations
// where the plan has room.  In a domain of few large groups (sub_block 0: one)
// going through a group costs more than the moves; there (kScanGroups,
// kScanMembers: at more groups, lists of tens of members were the faster by up
// to 4) the worms enter their vertex's two legs (one that turns: its interval)
// in a hash table of chains, entry 2 k + side with its successors in W[k].lab,
// and a worm looks up the six legs whose owners' intervals can meet its own.
// Its rank is k with one group, else counted over the group numbers in nxt[].
template <bool kSeveral>
__device__ void block_passes(const Tile& T, int dom, int nw, long long& tclk) {
  const Dev& d = *T.d;
  const int NT = int(blockDim.x), nwarps = NT >> 5, lane = threadIdx.x & 31;
  const int per = kSeveral ? 32 : max(16, (nw + nwarps - 1) / nwarps);
  const int first = (int(threadIdx.x) >> 5) * per + lane;
  const int slots = d.gslots;
  const bool scan = T.ngrp <= kScanGroups && nw > kScanMembers * T.ngrp;
  const bool table = d.gtab && !scan, hash = scan && d.ghash;
  int k = first;
  bool act = lane < per && k < nw;
  uint64_t key = 0;
  int li = 0, L = 0, slab = 0, u = 0, u_old = 0;
  Ahead o;
  o.fp = kTurn;
  // (a status found while pass p is prepared or run is read after the next
  // barrier by all threads alike: two flags in turn)
  auto fail = [&](int pass, int rc) { T.perr[pass & 1] = rc; };
  auto prepare = [&](int pass, int b3) {
    u = worm_group(T, li, slab, pass & 3);
    const int at = table ? atomicAdd(T.gcnt + b3 * T.ngrp + u, 1) : slots;
    const int rc = look_ahead(T, key, li, L, pass & 3, o);
    if (rc) fail(pass, rc);
    T.fp[(pass & 1) * d.wcap + k] = o.fp;
    if (hash) {
      const uint32_t stamp = uint32_t(pass + 1);
      uint32_t* hh = T.hash + (pass & 1) * d.ghash;
      uint16_t* next = reinterpret_cast<uint16_t*>(&T.W[k].lab) + 2 * (pass & 1);
      for (int e = 0; e < (turns(o.fp) ? 1 : 2); ++e) {
        const uint32_t leg = (e ? o.fp >> 16 : o.fp) & 0xffffu;
        const uint32_t was = atomicExch(hh + (leg & (d.ghash - 1)), (stamp << 16) | uint32_t(2 * k + e));
        next[e] = (was >> 16) == stamp ? uint16_t(was) : kNone;
      }
    }
    if (at < slots) T.cell[((pass & 1) * T.ngrp + u) * slots + at] = uint16_t(k);
    else if (scan) T.nxt[(pass & 1) * d.wcap + k] = uint16_t(u);
    else join_list(T, k, u, pass);
  };
  auto load = [&] {
    const WormRec& w = T.W[k];
    key = w.key;
    li = w.site;
    L = w.leg;
    slab = w.slab;
  };
  for (; k < nw && lane < per; k += NT) {
    load();
    prepare(0, 0);
    if (!kSeveral) break;
  }
  volatile uint16_t* dn = T.dn;
  uint16_t more[kNeighbours];
  int b3 = 0;  // pass % 3
  for (int pass = 0; pass < d.n_cycle; ++pass) {
    __syncthreads();
    if (const int rc = T.perr[pass & 1]) {
      tile_fail(T.misc, rc, 5);
      return;
    }
    const int stamp = pass + 1;
    const uint32_t* fp = T.fp + (pass & 1) * d.wcap;
    const uint16_t* nxt = T.nxt + (pass & 1) * d.wcap;
    const int b3n = b3 == 2 ? 0 : b3 + 1, b3p = b3 == 0 ? 2 : b3 - 1;
    if (kSeveral && table)
      for (int i = threadIdx.x; i < T.ngrp; i += NT) T.gcnt[b3p * T.ngrp + i] = 0;
    for (int t0 = 0; t0 < (kSeveral ? nw : 1); t0 += NT) {
      if (kSeveral) {
        k = t0 + first;
        act = k < nw;
        o.fp = kTurn;
        if (act) {
          load();
          u = worm_group(T, li, slab, pass & 3);
          look_ahead(T, key, li, L, pass & 3, o);  // (its status was seen when the pass was prepared)
        }
      }
      const uint16_t* cell = T.cell + ((pass & 1) * T.ngrp + u) * slots;
      const Meet meet(o);
      bool moved = !act;
      int r = 0, nn = 0, n = 0;  // n: members in the table
      bool list = false;         // some members are in the list
      uint32_t deps = 0;
      uint64_t mem = 0, waits = 0, w0 = 0, w1 = 0;
      if (act && turns(o.fp)) {
        key ^= 2u;
        if (kSeveral) *reinterpret_cast<uint32_t*>(&T.W[k].key) = uint32_t(key);  // (the word that holds the direction)
        moved = true;
      }
      auto neighbour = [&](bool m, int j, uint32_t g) {
        nn += m ? 1 : 0;
        mem = m ? (mem << 16) | uint64_t(j) : mem;
        deps = m ? (deps << 1) | (j < k && !turns(g) ? 1u : 0u) : deps;
      };
      auto look_at = [&](int j, uint32_t g) {
        r += j < k ? 1 : 0;
        neighbour(meet(g) && j != k, j, g);
      };
      if (!moved) {
        if (table) {
          const int c = T.gcnt[b3 * T.ngrp + u];
          n = min(c, slots);
          list = c > slots;
        } else {
          list = !scan;
        }
        for (int e0 = 0; e0 < n; e0 += 4) {
          const uint2 four = *reinterpret_cast<const uint2*>(cell + e0);
  #pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = int(((e < 2 ? four.x : four.y) >> (16 * (e & 1))) & 0xffff);
            if (e0 + e < n) look_at(j, fp[j]);
          }
        }
        if (list)
          for (int j = int(T.hd[(pass & 1) * T.hstride + u] & 0xffff); j != kNone; j = nxt[j]) look_at(j, fp[j]);
        if (hash) {
          const uint32_t* hh = T.hash + (pass & 1) * d.ghash;
          r = k;
          if (T.ngrp > 1) {
            r = 0;
            for (int j = 0; j < k; ++j) r += nxt[j] == u ? 1 : 0;
          }
          mem = ~0ull;
          for (int s = 0; s < 6; ++s) {
            const uint32_t pair = s < 2 ? o.dns : s < 4 ? o.fp : o.ups, leg = (s & 1) ? pair >> 16 : pair & 0xffffu;
            const uint32_t h = hh[leg & (d.ghash - 1)];
            int e = (h >> 16) == uint32_t(stamp) ? int(h & 0xffff) : kNone;
            while (e != kNone) {
              const int j = e >> 1;
              const uint32_t g = fp[j];
              if (((e & 1) ? g >> 16 : g & 0xffffu) == leg && j != k) {
                // (a worm can be found by both of its legs)
                const uint64_t x = mem ^ (uint64_t(j) * 0x0001000100010001ull);
                if (!((x - 0x0001000100010001ull) & ~x & 0x8000800080008000ull)) neighbour(true, j, g);
              }
              e = reinterpret_cast<const uint16_t*>(&T.W[j].lab)[2 * (pass & 1) + (e & 1)];
            }
          }
        } else if (scan) {
          for (int j = 0; j < nw; ++j)
            if (nxt[j] == u) look_at(j, fp[j]);
        }
        if (nn > 4) {  // more than mem holds: all of them into the list
          nn = 0;
          auto add = [&](int j) {
            const uint32_t g = fp[j];
            if (j == k || !meet(g)) return;
            if (nn < kNeighbours) {
              more[nn] = uint16_t(j);
              waits |= uint64_t(j < k && !turns(g) ? 1 : 0) << nn;
            }
            ++nn;
          };
          if (scan)
            for (int j = 0; j < nw; ++j)
              if (nxt[j] == u) add(j);
          for (int e = 0; e < n; ++e) add(int(cell[e]));
          if (list)
            for (int j = int(T.hd[(pass & 1) * T.hstride + u] & 0xffff); j != kNone; j = nxt[j]) add(j);
          // (a worm found by both of its legs counted twice: the list stays longer than mem, by this worm itself)
          while (nn < 5) more[nn++] = uint16_t(k);
        }
        const P4 b = philox(uint32_t(r), uint32_t(dom * T.ngrp + u), c2_word(kScatter, uint32_t(pass), d.replica),
                            d.sweep, d.key0, d.key1);
        w0 = uint64_t(b.x) | (uint64_t(b.y) << 32);
        w1 = uint64_t(b.z) | (uint64_t(b.w) << 32);
      }
      if (!kSeveral && act && table && pass > 0) T.gcnt[b3p * T.ngrp + u_old] = 0;
      u_old = u;
      phase_tick(d, 5, tclk);
      int spin = 0, seen = 0;
      while (!__all_sync(0xffffffffu, moved)) {
        if (!moved) {
          bool ready = true;
          if (nn <= 4) {
            for (uint32_t m = deps; m; m &= m - 1)
              ready = ready && dn[(mem >> (16 * (__ffs(int(m)) - 1))) & 0xffff] == stamp;
          } else if (nn <= kNeighbours) {
            for (; waits; waits &= waits - 1)
              if (dn[more[__ffsll((long long)waits) - 1]] != stamp) { ready = false; break; }
          } else {  // (worms of other groups meet none of this one's intervals)
            for (; seen < k; ++seen)
              if (dn[seen] != stamp && !turns(fp[seen]) && meet(fp[seen])) { ready = false; break; }
          }
          if (ready) {
            __threadfence_block();
            make_move(T, o, key, li, L, w0, w1, k, nw, [&](auto f) {
              if (nn <= 4) {
                for (int e = 0; e < nn; ++e) {
                  const WormRec& w = T.W[(mem >> (16 * e)) & 0xffff];
                  f(int(w.leg), w.key);
                }
              } else {  // (the list, or every worm of the domain)
                const bool listed = nn <= kNeighbours;
                for (int e = 0; e < (listed ? nn : nw); ++e) {
                  const int j = listed ? int(more[e]) : e;
                  if (j != k) f(int(T.W[j].leg), T.W[j].key);
                }
              }
            });
            WormRec& w = T.W[k];
            w.key = key;
            store_place(w, li, L);
            __threadfence_block();
            dn[k] = uint16_t(stamp);
            moved = true;
          }
        }
        if (++spin > kSpinLimit) { fail(pass + 1, PMWA_ETIMEOUT); break; }
      }
      if (d.phase_cycles && threadIdx.x == 0) atomicAdd(d.phase_cycles + 7, (unsigned long long)spin);
      phase_tick(d, 6, tclk);
      if (act && pass + 1 < d.n_cycle) prepare(pass + 1, b3n);
    }
    b3 = b3n;
  }
  __syncthreads();
  if (const int rc = T.perr[d.n_cycle & 1]) tile_fail(T.misc, rc, 5);
  if (!kSeveral && act) T.W[k].key = key;
}

// All N_cycle passes of a domain holding nw <= 32 worms, run by one warp
// (lane = threadIdx.x < 32) with no block barrier.  Lane k holds worm k of the
// label order (W[] is in that order).  __match_any_sync over the groups gives
// the lanes of its group and its rank r (the r-th move of a group draws Philox
// block r, as in the block-wide passes); the vertices go through fp[lane] and
// tell a lane which of them meet its own intervals.  It waits for those of
// lower rank, and rounds move every lane whose waits are over (at most 32
// rounds: the first waiting lane of each group waits for nobody), which gives
// each group's moves made one by one in rank order.  Returns a status (the
// same for all lanes).
__device__ int small_passes(const Tile& T, int dom, int nw, int lane) {
  const Dev& d = *T.d;
  const unsigned lt = (1u << lane) - 1u;
  const bool act = lane < nw;
  uint64_t key = 0;
  int li = 0, L = 0, slab = 0, rc = PMWA_OK;
  if (act) {
    const WormRec& w = T.W[lane];
    key = w.key;
    li = w.site;
    L = w.leg;
    slab = w.slab;
  }
  for (int pass = 0; pass < d.n_cycle; ++pass) {
    const int q = pass & 3;
    int u = -1 - lane;
    Ahead o;
    o.fp = kTurn;
    if (act) {
      u = worm_group(T, li, slab, q);
      rc = look_ahead(T, key, li, L, q, o);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, u);
    uint32_t* fp = T.fp + (pass & 1) * d.wcap;  // (two buffers: a slow lane may still read the last pass's)
    if (act) fp[lane] = o.fp;
    const bool turn = turns(o.fp);
    const Meet meet(o);
    const unsigned turning = __ballot_sync(0xffffffffu, turn);
    __syncwarp();
    unsigned near = 0;  // lanes whose intervals meet this one's, two at a time
    if (!turn)
      for (unsigned m = peers & ~(1u << lane); m;) {
        const int j = __ffs(int(m)) - 1;
        m &= m - 1;
        const int i = m ? __ffs(int(m)) - 1 : j;
        m &= m - 1;
        const uint32_t gj = fp[j], gi = fp[i];
        near |= (meet(gj) ? 1u : 0u) << j | (meet(gi) ? 1u : 0u) << i;
      }
    bool moved = turn;
    uint64_t w0 = 0, w1 = 0;
    if (!turn) {
      const P4 b = philox(uint32_t(__popc(peers & lt)), uint32_t(dom * T.ngrp + u),
                          c2_word(kScatter, uint32_t(pass), d.replica), d.sweep, d.key0, d.key1);
      w0 = uint64_t(b.x) | (uint64_t(b.y) << 32);
      w1 = uint64_t(b.z) | (uint64_t(b.w) << 32);
    } else {
      key ^= 2u;
    }
    const unsigned wait = near & lt & ~turning;
    unsigned done = turning;
    while (done != 0xffffffffu) {
      if (!moved && (wait & ~done) == 0) {
        make_move(T, o, key, li, L, w0, w1, lane, nw, [&](auto f) {
          for (unsigned m = near; m; m &= m - 1) {
            const int j = __ffs(int(m)) - 1;
            f(int(T.W[j].leg), T.W[j].key);
          }
        });
        WormRec& w = T.W[lane];
        w.key = key;
        store_place(w, li, L);
        moved = true;
      }
      __syncwarp();
      done = __ballot_sync(0xffffffffu, moved);
    }
    const unsigned bad = __ballot_sync(0xffffffffu, rc != PMWA_OK);
    if (bad) return __shfl_sync(0xffffffffu, rc, __ffs(int(bad)) - 1);
  }
  if (act) T.W[lane].key = key;
  return PMWA_OK;
}

}  // namespace

// Step 4 (Eq. 1) on every site of the domain (all threads): thread tid takes
// sites tid, tid + NT, ...  A site's words come from one stream, interval
// after interval, so a site is one chain; what a word is used for depends on
// the words before it (a gap of the rate-eta process, its wedge test, the
// parity sampler's two extra words, a new worm's label).  The lanes of a warp
// take one word each a step, whatever their state, so that the Philox blocks
// -- most of the arithmetic -- are evaluated by all lanes together and the
// common state, a gap longer than its interval, is shared; a loop of draws per
// interval had the lanes in different places of nested loops.  The sampler
// and the order of the words are sample_worms'.  Cycles a sweep, loop of draws
// -> steps -> steps with the binary32 wedge test: 16x16 sites 92k -> 79k -> 66k
// at beta t = 4, 273k -> 225k -> 188k at beta t = 16; 4x4 sites with 188 legs
// each 380k -> 337k -> 287k.
__device__ __forceinline__ void create_worms(const Tile& T, const ZigTab& Z, int tid, int NT) {
  const Dev& d = *T.d;
  enum { kDone, kState, kGap, kKeep, kExtra, kLabel };
  uint64_t offs[kMaxWormsPerInterval];
  int li = spread(tid, NT, T.nds), state = kDone, bad = 0;
  uint32_t unit = 0, block = 0;
  int st = 0, nl = 0, k = 0;            // the site's legs, its current interval
  uint64_t lo = 0, M = 0, pos = 0;      // interval: lower leg, worm grid points; last proposal
  int sigma = 0, p = 0, n = 0, tries = 0, o = 0, j = 0;
  bool first = true;
  ZigDraw zd;
  zd.start();
  auto attempt = [&] { n = 0; first = true; state = kGap; zd.start(); };
  auto retry = [&] {
    if (++tries >= Z.wtries) bad = PMWA_ETIMEOUT;
    attempt();
  };
  // the interval from leg st + k on (or the next one with grid points), else
  // the end of the site
  auto enter = [&] {
    for (;;) {
      if (k == nl) { state = kDone; li += NT; return; }
      lo = T.leg[st + k];
      const uint64_t hi = T.leg[st + (k + 1 == nl ? 0 : k + 1)];
      M = wpts(kpk(lo), kpk(hi));
      p = kab(lo);
      sigma = p ^ kbl(hi);
      if (M) break;
      if (sigma) { bad = PMWA_EINVARIANT; return; }
      T.wcnt[st + k] = 0;
      ++k;
    }
    tries = 0;
    attempt();
  };
  auto begin = [&] {
    const int s = T.gsite(li);
    st = T.off[li];
    nl = T.off[li + 1] - st;
    unit = uint32_t(s);
    block = 0;
    k = 0;
    if (nl == 0) { state = kState; return; }
    // (the state of a site whose delimiters are temporal boundaries only and
    // which keeps no worm: all its boundary states are equal)
    T.base[li] = uint8_t(kab(T.leg[st]));
    enter();
  };
  // the interval has its n worms
  auto accept = [&] {
    if (nl) T.wcnt[st + k] = uint8_t(n);  // (n <= kMaxWormsPerInterval)
    if (n == 0) { ++k; if (nl) enter(); else { state = kDone; li += NT; } return; }
    o = atomicAdd(&T.misc->nworms, n);
    const int sl = nl ? slab_of_m(d, wm_above(kpk(lo))) : 0;  // an interval lies inside one temporal slab
    atomicAdd(&T.misc->wslab[sl], n);
    if (o + n > d.wcap) { bad = PMWA_ECAPACITY; return; }
    j = 0;
    state = kLabel;
  };
  auto step = [&](uint64_t w) {
    if (state == kGap) {
      uint64_t E;
      if (zd.step(Z, w, E, &bad)) {
        const uint64_t g = grid_gap(E, d.SWs), nxt = first ? g - 1 : pos + g;
        first = false;
        zd.start();
        if (nxt < M) {
          pos = nxt;
          if (n >= kMaxWormsPerInterval) bad = PMWA_ECAPACITY; else offs[n++] = pos;
        } else if (sigma == 1 && M <= d.SWI) {
          if (n & 1) retry(); else state = kKeep;
        } else if ((n & 1) == sigma) {
          accept();
        } else {
          retry();
        }
      }
    } else if (state == kKeep) {
      if (__umul64hi(w, uint64_t(n + 1)) != 0) retry(); else state = kExtra;
    } else if (state == kExtra) {
      const uint64_t extra = __umul64hi(w, M);
      int at = n;
      bool clash = false;
      for (int e = 0; e < n; ++e) {
        if (offs[e] == extra) { clash = true; break; }
        if (offs[e] > extra) { at = e; break; }
      }
      if (clash) {
        retry();
      } else if (n >= kMaxWormsPerInterval) {
        bad = PMWA_ECAPACITY;
      } else {
        for (int e = n; e > at; --e) offs[e] = offs[e - 1];
        offs[at] = extra;
        ++n;
        accept();
      }
    } else if (state == kLabel) {
      const uint64_t m0 = nl ? wm_above(kpk(lo)) : 0;
      T.W[o + j] = WormRec{wkey((m0 + offs[j]) & (kTwo59 - 1), int(w & 1), p ^ 1 ^ (j & 1)), w >> 1, uint16_t(li),
                           nl ? uint16_t(st + k) : kNone, uint16_t(nl ? slab_of_m(d, m0) : 0), 0};
      if (++j == n) { ++k; if (nl) enter(); else { state = kDone; li += NT; } }
    } else if (state == kState) {  // a site without legs: its state, then one interval round the circle
      p = int(w >> 63);
      T.base[li] = uint8_t(p);
      M = kTwo59;
      sigma = 0;
      tries = 0;
      attempt();
    }
  };
  for (;;) {
    if (state == kDone && li < T.nds && !bad) begin();
    const bool run = state != kDone && !bad;
    if (!__any_sync(0xffffffffu, run)) {
      if (__any_sync(0xffffffffu, state == kDone && li < T.nds && !bad)) continue;
      break;
    }
    const P4 b = philox(block, unit, c2_word(kRegen, 0, d.replica), d.sweep, d.key0, d.key1);
    ++block;
    uint64_t w = uint64_t(b.x) | (uint64_t(b.y) << 32);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      if (run && state != kDone && !bad) step(w);
      w = uint64_t(b.z) | (uint64_t(b.w) << 32);
    }
  }
  if (bad) tile_fail(T.misc, bad, 4);
}

// ---------------------------------------------------------------------------
// Where the sources of a site's Step-3 merge start and end for one part of
// its circle: the old events [o0, o1), the new legs of its four bonds
// [s_j, e_j) of each run, the temporal boundaries [t0, t1).  Part h of P (a
// power of two) holds the time keys from h 2^62 / P up to the next part's.
// o0 >= 0: the first old event, known from before (else it is looked up).
struct MergeRange {
  int o0, o1, s0, e0, s1, e1, s2, e2, s3, e3, t0, t1;
};

__device__ __forceinline__ MergeRange merge_range(const Tile& T, const uint64_t* KO, int nO, const int lb[4],
                                                  int h, int P, int o0, int o1) {
  const Dev& d = *T.d;
  const int n0 = lb[0] >= 0 ? T.bcnt[lb[0]] : 0, n1 = lb[1] >= 0 ? T.bcnt[lb[1]] : 0;
  const int n2 = lb[2] >= 0 ? T.bcnt[lb[2]] : 0, n3 = lb[3] >= 0 ? T.bcnt[lb[3]] : 0;
  const int NB = d.ntau > 1 ? d.ntau : 0;
  MergeRange R{0, nO, 0, n0, 0, n1, 0, n2, 0, n3, 0, NB};
  if (P == 1) return R;
  const uint64_t part = kTwo62 / uint64_t(P);
  // (a candidate c of the pool has the time key c >> 2 = kpk(c))
  if (h > 0) {
    const uint64_t cut = part * uint64_t(h);
    R.o0 = o0 >= 0 ? o0 : slot_lower(KO, nO, cut);
    R.s0 = n0 ? slot_lower(T.pool + T.boff[lb[0]], n0, cut) : 0;
    R.s1 = n1 ? slot_lower(T.pool + T.boff[lb[1]], n1, cut) : 0;
    R.s2 = n2 ? slot_lower(T.pool + T.boff[lb[2]], n2, cut) : 0;
    R.s3 = n3 ? slot_lower(T.pool + T.boff[lb[3]], n3, cut) : 0;
    while (R.t0 < NB && tb_pk(d, R.t0) < cut) ++R.t0;
  }
  if (h + 1 < P) {
    const uint64_t cut = part * uint64_t(h + 1);
    R.o1 = o1 >= 0 ? o1 : slot_lower(KO, nO, cut);
    R.e0 = n0 ? slot_lower(T.pool + T.boff[lb[0]], n0, cut) : 0;
    R.e1 = n1 ? slot_lower(T.pool + T.boff[lb[1]], n1, cut) : 0;
    R.e2 = n2 ? slot_lower(T.pool + T.boff[lb[2]], n2, cut) : 0;
    R.e3 = n3 ? slot_lower(T.pool + T.boff[lb[3]], n3, cut) : 0;
    R.t1 = 0;
    while (R.t1 < NB && tb_pk(d, R.t1) < cut) ++R.t1;
  }
  return R;
}

// The Step-3 merge of one part of site li's circle into the leg table from
// position o: the kept old events, the new legs of its four bonds and the
// temporal boundaries (tag-6 delimiters), in time order.  A new leg's and a
// boundary's states above and below are the worldline's state there, that of
// the last old event passed (Step 3 changes no state).
//
// A chain of as many steps as the site has old events and new legs, one
// thread a site: each step takes the earliest of the six heads, kept or not,
// by selects -- no lane waits for another's branch -- and the old list, which
// is read from L2, is fetched four keys ahead.  Cycles of the whole phase a
// sweep: 16x16 sites 108k -> 76k at beta t = 4, 175k -> 101k at beta t = 16; 4x4
// sites with 188 legs each 532k -> 228k.
template <bool OTF>
__device__ __forceinline__ void merge_site(const Tile& T, int li, const uint64_t* KO, int nO, int base0,
                                           const int lb[4], const MergeRange& R, int o) {
  const Dev& d = *T.d;
  unsigned out = 0;  // leg tags of the site whose bonds leave the domain: their legs all stay
#pragma unroll
  for (int t = 0; t < 6; ++t) out |= (T.tinfo[li * 6 + t] & 2) ? 1u << t : 0u;
  // each run's next candidate (h), its place in the pool (i) and the run's end (e)
  int i0 = (lb[0] >= 0 ? T.boff[lb[0]] : 0), i1 = (lb[1] >= 0 ? T.boff[lb[1]] : 0);
  int i2 = (lb[2] >= 0 ? T.boff[lb[2]] : 0), i3 = (lb[3] >= 0 ? T.boff[lb[3]] : 0);
  const int e0 = i0 + R.e0, e1 = i1 + R.e1, e2 = i2 + R.e2, e3 = i3 + R.e3;
  i0 += R.s0; i1 += R.s1; i2 += R.s2; i3 += R.s3;
  const uint64_t none = ~0ull;
  uint64_t h0 = i0 < e0 ? T.pool[i0] : none, h1 = i1 < e1 ? T.pool[i1] : none;
  uint64_t h2 = i2 < e2 ? T.pool[i2] : none, h3 = i3 < e3 ? T.pool[i3] : none;
  int io = R.o0, ib = R.t0;
  const int on = R.o1;
  uint64_t r0 = io < on ? KO[io] : none, r1 = io + 1 < on ? KO[io + 1] : none;
  uint64_t r2 = io + 2 < on ? KO[io + 2] : none, r3 = io + 3 < on ? KO[io + 3] : none;
  uint64_t tb = ib < R.t1 ? tb_pk(d, ib) << 2 : none;
  uint64_t cur = nO ? uint64_t(kab(KO[(io ? io : nO) - 1])) : uint64_t(base0);
  for (;;) {
    // (times differ, so whole words compare as times do)
    const bool s01 = h1 < h0, s23 = h3 < h2;
    const uint64_t a = s01 ? h1 : h0, b = s23 ? h3 : h2;
    const bool sb = b < a;
    const uint64_t c = sb ? b : a, t = min(r0, tb);
    const bool fresh = c < t, bound = !fresh && tb < r0;
    const uint64_t best = fresh ? c : t;
    if (best == none) break;
    if (fresh || bound) {
      T.leg[o++] = (best & ~3ull) | (cur * 3);
    } else {
      const int tag = ktag(r0);
      bool keep = tag != 7 && (kab(r0) != kbl(r0) || ((out >> tag) & 1));
      if (OTF && !keep && tag != 7) {
        const uint64_t pos = kpk(r0) >> 3;
        keep = !(in_win(T, li, pos) || in_win(T, T.nbr[li * 6 + tag], pos));
      }
      if (keep) T.leg[o++] = r0;
      cur = uint64_t(kab(r0));
      r0 = r1; r1 = r2; r2 = r3;
      r3 = io + 4 < on ? KO[io + 4] : none;
      ++io;
    }
    if (bound) tb = ++ib < R.t1 ? tb_pk(d, ib) << 2 : none;
    if (fresh) {
      const int run = sb ? (s23 ? 3 : 2) : (s01 ? 1 : 0);
      const int at = 1 + (run == 0 ? i0 : run == 1 ? i1 : run == 2 ? i2 : i3);
      const int end = run == 0 ? e0 : run == 1 ? e1 : run == 2 ? e2 : e3;
      const uint64_t nx = at < end ? T.pool[at] : none;
      if (run == 0) { h0 = nx; i0 = at; }
      if (run == 1) { h1 = nx; i1 = at; }
      if (run == 2) { h2 = nx; i2 = at; }
      if (run == 3) { h3 = nx; i3 = at; }
    }
  }
}

// the term of a site without legs (out of line: the series' code is long)
__device__ __noinline__ bool xg_fix_circle(GridScale XQ, uint64_t& v) { return xg_fix(0, kTwo59, XQ, v); }

template <bool OTF>
__device__ __forceinline__ void tile_body(const Dev& d, const int dom, const int stop, unsigned char* sm,
                                          int* wsum) {
  Tile T;
  T.d = &d;
  T.th = reinterpret_cast<uint32_t*>(sm + d.sm_th);
  T.off = reinterpret_cast<int*>(sm + d.sm_off);
  T.base = reinterpret_cast<uint8_t*>(sm + d.sm_base);
  T.bcnt = reinterpret_cast<int*>(sm + d.sm_bcnt);
  T.rng = reinterpret_cast<uint32_t*>(T.bcnt);
  T.boff = reinterpret_cast<int*>(sm + d.sm_boff);
  T.perr = T.boff;
  T.misc = reinterpret_cast<Misc*>(sm + d.sm_misc);
  T.leg = reinterpret_cast<uint64_t*>(sm + d.sm_leg);
  T.wcnt = reinterpret_cast<uint8_t*>(sm + d.sm_wcnt);
  T.part = reinterpret_cast<uint16_t*>(sm + d.sm_part);
  T.pool = reinterpret_cast<uint64_t*>(sm + d.sm_pool);
  T.W = reinterpret_cast<WormRec*>(sm + d.sm_worm);
  T.idx = reinterpret_cast<uint16_t*>(sm + d.sm_idx);
  T.ord = reinterpret_cast<uint16_t*>(sm + d.sm_ord);
  T.dn = reinterpret_cast<uint16_t*>(sm + d.sm_dn);
  T.nxt = reinterpret_cast<uint16_t*>(sm + d.sm_nxt);
  T.fp = reinterpret_cast<uint32_t*>(sm + d.sm_fp);
  T.bkt = reinterpret_cast<int*>(sm + d.sm_bkt);
  T.fill = reinterpret_cast<int*>(sm + d.sm_fill);
  T.gcnt = reinterpret_cast<int*>(sm + d.sm_gcnt);
  T.hash = reinterpret_cast<uint32_t*>(sm + d.sm_hash);
  T.cell = reinterpret_cast<uint16_t*>(sm + d.sm_cell);
  T.hd = reinterpret_cast<uint32_t*>(T.bkt);
  T.hstride = (d.sm_fill - d.sm_bkt) / int(sizeof(int));
  T.nbr = reinterpret_cast<uint16_t*>(sm + d.sm_nbr);
  T.tinfo = reinterpret_cast<uint8_t*>(sm + d.sm_tinfo);
  T.sub = reinterpret_cast<uint16_t*>(sm + d.sm_sub);
  T.soff = reinterpret_cast<int*>(sm + d.sm_soff);
  T.old = reinterpret_cast<uint64_t*>(sm + d.sm_old);
  T.staged = T.early = false;
  T.x0 = (dom % d.ndx) * d.dom_x;
  T.y0 = (dom / d.ndx) * d.dom_y;
  T.nds = d.dom_x * d.dom_y;
  T.nsub = sb_slots(d.dom_x, d.sub_block, d.ndx) * sb_slots(d.dom_y, d.sub_block, d.ndy);
  T.ngrp = T.nsub * d.ntau;
  const int tid = threadIdx.x, NT = blockDim.x, nds = T.nds;
  Misc* misc = T.misc;

  long long tclk = clock64();
  // the domain's current event lists on their way into L2 before the scans
  // of Step 3 reach them: one bulk prefetch per site of its used slots (a
  // list starts 64-byte aligned; its length rounded up to 16 bytes stays
  // within the site's cap, a multiple of 8 keys)
  for (int li = tid; li < nds; li += NT) {
    const int s = T.gsite(li), n = cnt_n(d.cntA[s]);
    if (n) prefetch_l2(d.keyA + size_t(s) * d.cap, uint32_t((n * 8 + 15) & ~15));
  }
  const ZigTab Z = zig_stage(sm + d.sm_zig, d.zig_cap, d.worm_tries);
  for (int k = tid; k < 256; k += NT) T.th[k] = d.TH[k] >> 32 ? ~0u : uint32_t(d.TH[k]);
  if (tid == 0) { misc->pool_used = 0; misc->nworms = 0; misc->err = 0; misc->where = 0; }
  for (int k = tid; k < d.ntau; k += NT) misc->wslab[k] = 0;
  // per-site tables: bond partners by leg tag, sub-blocks by offset pattern
  for (int li = tid; li < nds; li += NT)
    for (int q = 0; q < 4; ++q) T.sub[li * 4 + q] = uint16_t(T.sub_of(li, q));
  __syncthreads();
  for (int li = tid; li < nds; li += NT) {
    for (int t = 0; t < 6; ++t) { T.nbr[li * 6 + t] = 0; T.tinfo[li * 6 + t] = 0; }
    const int s = T.gsite(li);
    for (int j = 0; j < 4; ++j) {
      const int dir = j & 1;
      const int a = (j < 2) ? s : site_step(d, s, dir, -1);
      const int tg = bond_tag(d, a, dir);
      const bool out = boundary_bond(d, a, dir);
      int info = (j < 2 ? 1 : 0) | (out ? 2 : 0);
      if (!out) {
        const int lo = T.lsite((j < 2) ? site_step(d, s, dir, +1) : a);
        T.nbr[li * 6 + tg] = uint16_t(lo);
        for (int q = 0; q < 4; ++q) info |= T.sub[li * 4 + q] == T.sub[lo * 4 + q] ? 4 << q : 0;
      }
      T.tinfo[li * 6 + tg] = uint8_t(info);
    }
  }
  __syncthreads();

  // stage the domain's current configuration in shared memory (one warp per
  // site, coalesced), so that the scans of phases 1-2 do not wait on HBM/L2
  if (d.oldcap > 0) {
    for (int li = tid; li < nds; li += NT) T.soff[li] = cnt_n(d.cntA[T.gsite(li)]);
    __syncthreads();
    if (block_scan(T.soff, nds, wsum) <= d.oldcap) {
      const int lane = tid & 31;
      for (int li = tid >> 5; li < nds; li += NT >> 5) {
        const uint64_t* KO = d.keyA + size_t(T.gsite(li)) * d.cap;
        const int st = T.soff[li], n = T.soff[li + 1] - st;
        for (int k = lane; k < n; k += 32) T.old[st + k] = KO[k];
      }
      T.staged = true;
    }
    __syncthreads();
  }
  // Else the leg table, empty until the merge, holds the lists for phase 1 and
  // the merge's counts where they fit: every bond reads two of them key by
  // key, 29 cycles a key instead of L2's several hundred.  (The counts of the
  // merge then go through the worm-count bytes: 8 a site.)  Cycles of the
  // candidate phase a sweep: 254k -> 146k at 16x16 sites and beta t = 16, 598k
  // -> 340k at 4x4 sites with 188 legs each; 94k -> 97k at beta t = 4, which the
  // counts win back.
  if (!T.staged && d.legcap >= 8 * nds) {
    for (int li = tid; li < nds; li += NT) T.off[li] = cnt_n(d.cntA[T.gsite(li)]);
    __syncthreads();
    T.early = block_scan(T.off, nds, wsum) <= d.legcap;
    if (T.early) {
      const int lane = tid & 31;
      for (int li = tid >> 5; li < nds; li += NT >> 5) {
        const uint64_t* KO = d.keyA + size_t(T.gsite(li)) * d.cap;
        const int st = T.off[li], n = T.off[li + 1] - st;
        for (int k = lane; k < n; k += 32) T.leg[st + k] = KO[k];
      }
    }
    __syncthreads();
  }

  if (OTF) {
    // the worms of the current configuration, by site: the windows of the
    // on-the-fly vertex phase
    T.wmo = reinterpret_cast<int*>(sm + d.sm_wmo);
    T.wm = reinterpret_cast<uint64_t*>(sm + d.sm_wm);
    for (int li = tid; li < nds; li += NT) {
      const int s = T.gsite(li), n = cnt_n(d.cntA[s]);
      const uint64_t* KO = T.okeys_early(li, s);
      int c = 0;
      for (int k = 0; k < n; ++k) c += kworm(KO[k]) ? 1 : 0;
      T.wmo[li] = c;
    }
    __syncthreads();
    if (block_scan(T.wmo, nds, wsum) > d.wcap) { if (tid == 0) tile_fail(misc, PMWA_ECAPACITY, 35); }
    __syncthreads();
    if (misc->err) goto fail;
    for (int li = tid; li < nds; li += NT) {
      const int s = T.gsite(li), n = cnt_n(d.cntA[s]);
      const uint64_t* KO = T.okeys_early(li, s);
      int o = T.wmo[li];
      for (int k = 0; k < n; ++k) if (kworm(KO[k])) T.wm[o++] = kpk(KO[k]) >> 3;
    }
    __syncthreads();
  }

  // ---- phase 1: Step 3 candidates per bond
  // (the bonds, sites and parts of sites of these phases are spread evenly over
  // the warps: a warp's loops run as long as its slowest lane's)
  for (int lb = spread(tid, NT, 2 * nds); lb < 2 * nds; lb += NT) {
    const int li = lb >> 1, dir = lb & 1;
    const int a = T.gsite(li);
    uint64_t buf[kMaxCandPerBond];
    int n = 0, bad = 0;
    if (d.has_vertices && !boundary_bond(d, a, dir)) {
      const int b = site_step(d, a, dir, +1);
      n = bond_candidates<OTF>(d, Z, a, dir, T.okeys_early(li, a), T.okeys_early(T.lsite(b), b), buf,
                               min(d.capb, kMaxCandPerBond), &bad, &T, li, T.lsite(b));
    }
    if (bad) { tile_fail(misc, bad, 31); n = 0; }
    int o = 0;
    if (n) {
      o = atomicAdd(&misc->pool_used, n);
      if (o + n > d.poolcap) { tile_fail(misc, PMWA_ECAPACITY, 32); n = 0; }
      else for (int k = 0; k < n; ++k) T.pool[o + k] = buf[k];
    }
    T.bcnt[lb] = n;
    T.boff[lb] = o;
  }
  __syncthreads();
  phase_tick(d, 0, tclk);
  if (misc->err) goto fail;

  // ---- phase 2: kept legs + new legs per site, merged in time order.  With
  // P threads a site to spare (two in the 512-thread CTA of a 16x16 domain,
  // eight in a 4x4 domain's of 128) each site's circle is cut into P parts at equal
  // times that P threads count and merge; each part is in time order and the
  // parts follow one another, so the leg table is the one a single thread
  // writes.  The parts' counts and first old events go through the (not yet
  // used) worm-count bytes.
  {
    int P = 1;
    while (2 * P * nds <= NT && P < 8 && d.legcap >= 16 * P * nds) P *= 2;
    const int units = P * nds;
    const bool scratch = P > 1 || T.early;
    int* hc = reinterpret_cast<int*>(T.wcnt);  // [P][nds] legs of a part
    int* ho = hc + units;                      // [P][nds] its first old event
    for (int un = spread(tid, NT, units); un < units; un += NT) {
      const int li = un % nds, h = un / nds;
      const int s = T.gsite(li);
      const uint64_t* KO = T.okeys_early(li, s);
      const int nO = cnt_n(d.cntA[s]);
      int lb[4];
      site_bonds(T, li, lb);
      const MergeRange R = merge_range(T, KO, nO, lb, h, P, -1, -1);
      int c = 0;
      for (int k = R.o0; k < R.o1; ++k) c += kept_leg<OTF>(T, li, KO[k]);
      c += (R.e0 - R.s0) + (R.e1 - R.s1) + (R.e2 - R.s2) + (R.e3 - R.s3) + (R.t1 - R.t0);
      if (scratch) hc[un] = c;
      else T.off[li] = c;
      if (P > 1) ho[un] = R.o0;
    }
    if (scratch) {
      __syncthreads();
      for (int li = tid; li < nds; li += NT) {
        int c = 0;
        for (int h = 0; h < P; ++h) c += hc[h * nds + li];
        T.off[li] = c;
      }
    }
    __syncthreads();
    if (block_scan(T.off, nds, wsum) > d.legcap) { if (tid == 0) tile_fail(misc, PMWA_ECAPACITY, 33); }
    __syncthreads();
    if (misc->err) goto fail;
    for (int un = spread(tid, NT, units); un < units; un += NT) {
      const int li = un % nds, h = un / nds;
      const int s = T.gsite(li);
      const uint64_t* KO = T.okeys(li, s);
      const int nO = cnt_n(d.cntA[s]);
      int lb[4];
      site_bonds(T, li, lb);
      int o = T.off[li];
      for (int e = 0; e < h; ++e) o += hc[e * nds + li];
      const MergeRange R = merge_range(T, KO, nO, lb, h, P, P > 1 ? ho[un] : -1, h + 1 < P ? ho[un + nds] : -1);
      merge_site<OTF>(T, li, KO, nO, cnt_base(d.cntA[s]), lb, R, o);
    }
  }
  __syncthreads();
  if (stop >= 5 && d.use_part) {
    // the partner leg of every vertex leg whose bond lies in the domain: the
    // leg with the same time on the bond's other site (legs keep their
    // places through Step 5; only their states change)
    // (legs split evenly over the threads; each vertex once, from its lower site)
    const int total = T.off[nds];
    for (int j = tid; j < total; j += NT) T.part[j] = kNone;
    __syncthreads();
    const int chunk = (total + NT - 1) / NT;
    int j = tid * chunk;
    const int jend = min(total, j + chunk);
    if (j < jend) {
      int a = 0, b = nds;  // the site of leg j: off[a] <= j < off[a + 1]
      while (a + 1 < b) {
        const int m = (a + b) >> 1;
        if (T.off[m] <= j) a = m; else b = m;
      }
      int li = a;
      for (; j < jend; ++j) {
        while (T.off[li + 1] <= j) ++li;
        const uint64_t key = T.leg[j];
        if (ktag(key) == 6) continue;  // a temporal boundary
        if ((T.tinfo[li * 6 + ktag(key)] & 3) != 1) continue;  // (inside the domain, seen from its lower site)
        const int ip = leg_index(T, T.nbr[li * 6 + ktag(key)], kpk(key));
        if (ip < 0) { tile_fail(misc, PMWA_EINVARIANT, 34); continue; }
        T.part[j] = uint16_t(ip);
        T.part[ip] = uint16_t(j);
      }
    }
    __syncthreads();
  }
  phase_tick(d, 1, tclk);

  if (stop >= 4) {
    // ---- phase 3: Step 4, worms of every interval (the pool is dead now)
    create_worms(T, Z, tid, NT);
    __syncthreads();
    phase_tick(d, 2, tclk);
    if (misc->err) goto fail;

    // ---- phase 4: Step 5
    if (stop >= 5) {
      const int nw = misc->nworms;
      if (nw > 0) label_order(T, nw, wsum);
      // The shifted sub-block schedule: in pass p every worm moves once,
      // inside the sub-block of offset pattern p & 3 that holds its site, in
      // label order; the r-th move of sub-block u draws Philox block r of
      // stream (unit = domain * n_sub + u, scatter | pass).
      for (int u = tid; u < T.ngrp; u += NT) T.hd[u] = T.hd[T.hstride + u] = 0;  // stamp 0: no pass
      for (int i = tid; i < 2 * d.ghash; i += NT) T.hash[i] = 0;
      if (d.gtab)
        for (int u = tid; u < 3 * T.ngrp; u += NT) T.gcnt[u] = 0;
      for (int li = tid; li < nds; li += NT) T.rng[li] = uint32_t(T.off[li]) | (uint32_t(T.off[li + 1]) << 16);
      for (int k = tid; k < nw; k += NT) T.dn[k] = 0;
      if (tid < 2) T.perr[tid] = PMWA_OK;
      if (nw > kMaxTurns * NT) {
        if (tid == 0) tile_fail(misc, PMWA_EINVARIANT, 7);
      } else if (nw > NT) {  // the worms into label order, several a thread
        WormRec w[kMaxTurns];
        for (int k = tid, t = 0; k < nw; k += NT, ++t) w[t] = T.W[T.ord[k]];
        __syncthreads();
        for (int k = tid, t = 0; k < nw; k += NT, ++t) T.W[k] = w[t];
      } else if (nw > 0) {  // one a thread
        WormRec w{};
        if (tid < nw) w = T.W[T.ord[tid]];
        __syncthreads();
        if (tid < nw) T.W[tid] = w;
      }
      __syncthreads();
      if (misc->err) goto fail;
      if (nw > NT) {
        block_passes<true>(T, dom, nw, tclk);
      } else if (nw > 32) {
        block_passes<false>(T, dom, nw, tclk);
      } else if (nw > 0 && tid < 32) {  // few worms: one warp, no barrier
        const int rc = small_passes(T, dom, nw, tid);
        if (rc && tid == 0) tile_fail(misc, rc, 5);
      }
      __syncthreads();
      if (misc->err) goto fail;
      phase_tick(d, 3, tclk);
    }
  }

  // ---- phase 5: next configuration + Step 6.  An event's place in its site's
  // list follows from counts alone: a leg's from its index and the site's
  // worms below it, a worm's from its interval and the site's worms below it.
  // So legs and worms are laid over the threads, not sites (a site's merge is
  // one chain, and sites are half or an eighth of the threads in the larger
  // and smaller CTAs), and consecutive lanes write consecutive keys.  The
  // occupied time of a site is 2^62 when its state at the origin is 1, plus
  // the times where the state falls and minus those where it rises.  Cycles a
  // sweep, with xg_series: 16x16 sites 75k -> 60k at beta t = 4, 153k -> 112k
  // at beta t = 16; 4x4 sites with 188 legs each 165k -> 91k.
  {
    const int nw = (stop >= 4) ? misc->nworms : 0;
    const int NB = d.ntau > 1 ? d.ntau : 0;  // temporal boundaries in the leg table: no events
    uint64_t nv = 0, nk = 0, nwc = 0, olo = 0, ohi = 0, qlo = 0, qhi = 0;
    double q = 0.0;
    // +t at a fall, -t at a rise of the state (128-bit two's complement)
    auto flip = [&](uint64_t pk, int above) {
      if (above) add128(olo, ohi, ~pk + 1, pk ? ~0ull : 0);
      else add128(olo, ohi, pk, 0);
    };
    if (stop >= 4) {
      for (int li = tid; li <= nds; li += NT) T.bkt[li] = 0;
      __syncthreads();
      for (int w = tid; w < nw; w += NT) atomicAdd(&T.bkt[T.W[w].site], 1);
      __syncthreads();
      block_scan(T.bkt, nds, wsum);
      for (int li = tid; li < nds; li += NT) T.fill[li] = T.bkt[li];
      __syncthreads();
      for (int w = tid; w < nw; w += NT) T.idx[atomicAdd(&T.fill[T.W[w].site], 1)] = uint16_t(w);
      __syncthreads();
      // worms of site li below `key`
      auto below = [&](int li, uint64_t key) {
        int r = 0;
        for (int p = T.bkt[li]; p < T.bkt[li + 1]; ++p) r += T.W[T.idx[p]].key < key ? 1 : 0;
        return r;
      };
      for (int w = tid; w < nw; w += NT) {
        const uint64_t key = T.W[w].key;
        const int li = T.W[w].site, L = T.W[w].leg;
        int at = below(li, key);
        // (a worm of the interval round the origin may lie before the first leg)
        if (L != kNone && key > T.leg[L]) at += L - T.off[li] + 1 - (NB ? slab_of_m(d, key >> 5) + 1 : 0);
        if (at >= d.cap) { tile_fail(misc, PMWA_ECAPACITY, 6); continue; }
        d.keyB[size_t(T.gsite(li)) * d.cap + at] = key;
        flip(kpk(key), kab(key));
        ++nwc;
      }
      const int total = T.off[nds], warps = NT >> 5;
      const int chunk = ((total + warps - 1) / warps + 31) & ~31;  // legs a warp
      int j = (tid >> 5) * chunk + (tid & 31);
      const int jend = min(total, (tid >> 5) * chunk + chunk);
      if (j < jend) {
        int a = 0, b = nds;  // the site of leg j: off[a] <= j < off[a + 1]
        while (a + 1 < b) {
          const int m = (a + b) >> 1;
          if (T.off[m] <= j) a = m; else b = m;
        }
        int li = a, en = T.off[a + 1];
        size_t slot = size_t(T.gsite(li)) * d.cap;
        for (; j < jend; j += 32) {
          if (en <= j) {
            do en = T.off[++li + 1]; while (en <= j);
            slot = size_t(T.gsite(li)) * d.cap;
          }
          const int st = T.off[li];
          const uint64_t lo = T.leg[j];
          const int tag = ktag(lo);
          if (tag < 6) {
            const uint64_t m = lo >> 5;
            const int at = j - st + below(li, lo) - (NB && m ? slab_of_m(d, m - 1) + 1 : 0);
            if (at >= d.cap) tile_fail(misc, PMWA_ECAPACITY, 6);
            else d.keyB[slot + at] = lo;
          }
          if (stop < 6) continue;
          // Step 6, per interval: vertex and kink counts, and the improved <Q>
          // sum of x g_sigma(x), in fixed point (exact sum) where x < 1/2,
          // else in binary64
          const bool kink = tag < 6 && kab(lo) != kbl(lo);
          if (kink) flip(kpk(lo), kab(lo));
          if (tag < 6 && (T.tinfo[li * 6 + tag] & 1)) { ++nv; if (kink) ++nk; }
          const uint64_t hi = T.leg[j + 1 == en ? st : j + 1];
          const uint64_t I = wpts(kpk(lo), kpk(hi));
          const int sg = kab(lo) ^ kbl(hi);
          uint64_t v;
          if (xg_fix(sg, I, d.XQ, v)) add128(qlo, qhi, v, 0);
          else q += xg_sigma(sg, __ull2double_rn(I) * d.XW);
        }
      }
    }
    for (int li = tid; li < nds; li += NT) {
      const int s = T.gsite(li);
      const int st = T.off[li], nl = T.off[li + 1] - st;
      int no, base;
      if (stop >= 4) {
        no = nl - (nl ? NB : 0) + T.bkt[li + 1] - T.bkt[li];
        base = T.base[li];
        if (nl) {  // the state at the origin: above the last leg, and past the worms behind it
          const uint64_t top = T.leg[st + nl - 1];
          base = kab(top);
          for (int p = T.bkt[li]; p < T.bkt[li + 1]; ++p) base ^= T.W[T.idx[p]].key > top ? 1 : 0;
        }
        if (no > d.cap) continue;  // (reported above)
      } else {
        // Step 3 alone: the legs merged with the current configuration's worms
        uint64_t* OUT = d.keyB + size_t(s) * d.cap;
        const uint64_t* KO = d.keyA + size_t(s) * d.cap;
        const int nO = cnt_n(d.cntA[s]);
        int il = 0, io = 0;
        no = 0;
        bool bad = false;
        for (;;) {
          while (io < nO && !kworm(KO[io])) ++io;
          while (il < nl && ktag(T.leg[st + il]) == 6) ++il;  // a temporal boundary is no event
          const uint64_t wk = io < nO ? KO[io] : ~0ull, lk = il < nl ? T.leg[st + il] : ~0ull;
          if (lk == ~0ull && wk == ~0ull) break;
          if (no >= d.cap) { bad = true; break; }
          if (lk < wk) { OUT[no++] = lk; ++il; } else { OUT[no++] = wk; ++io; }
        }
        if (bad) { tile_fail(misc, PMWA_ECAPACITY, 6); continue; }
        base = no ? kab(OUT[no - 1]) : cnt_base(d.cntA[s]);
      }
      d.cntB[s] = uint32_t(no) | (uint32_t(base) << 31);
      if (stop < 6) continue;
      if (base) add128(olo, ohi, kTwo62, 0);
      if (nl == 0) {  // a site without legs is one interval of sigma = 0
        uint64_t v;
        if (xg_fix_circle(d.XQ, v)) add128(qlo, qhi, v, 0);
        else q += xg_sigma(0, double(kTwo59) * d.XW);
      }
    }
    if (stop >= 6) {
      for (int o = 16; o > 0; o >>= 1) {
        nv += __shfl_down_sync(0xffffffffu, nv, o);
        nk += __shfl_down_sync(0xffffffffu, nk, o);
        nwc += __shfl_down_sync(0xffffffffu, nwc, o);
        const uint64_t blo = __shfl_down_sync(0xffffffffu, olo, o);
        const uint64_t bhi = __shfl_down_sync(0xffffffffu, ohi, o);
        add128(olo, ohi, blo, bhi);
        const uint64_t clo = __shfl_down_sync(0xffffffffu, qlo, o);
        const uint64_t chi = __shfl_down_sync(0xffffffffu, qhi, o);
        add128(qlo, qhi, clo, chi);
      }
      if (__any_sync(0xffffffffu, q != 0.0))  // (binary64 terms are rare)
        for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
      q += __ull2double_rn(qhi) * 4.0 + __ull2double_rn(qlo) * 0x1p-62;
      if ((tid & 31) == 0) {
        pmwa_row* r = d.rows + d.row;
        if (nv) atomicAdd(reinterpret_cast<unsigned long long*>(&r->n_v), (unsigned long long)nv);
        if (nk) atomicAdd(reinterpret_cast<unsigned long long*>(&r->n_k), (unsigned long long)nk);
        if (nwc) atomicAdd(reinterpret_cast<unsigned long long*>(&r->n_w), (unsigned long long)nwc);
        if (olo | ohi) {
          const unsigned long long old =
              atomicAdd(reinterpret_cast<unsigned long long*>(&r->occ_lo), (unsigned long long)olo);
          const uint64_t carry = (old + olo < old) ? 1 : 0;
          if (ohi + carry)
            atomicAdd(reinterpret_cast<unsigned long long*>(&r->occ_hi), (unsigned long long)(ohi + carry));
        }
        atomicAdd(&r->q_impr, q);
      }
      if (dom == 0 && tid == 0) d.rows[d.row].sweep = d.sweep;
      if (tid == 0) {
        // worms per (space-time) domain: the fewest (kept as a complement, so
        // that the zeroed row and an atomic maximum give the minimum) and the
        // empty ones
        pmwa_row* r = d.rows + d.row;
        unsigned wmin = ~0u, empty = 0;
        for (int k = 0; k < d.ntau; ++k) {
          wmin = min(wmin, unsigned(misc->wslab[k]));
          empty += misc->wslab[k] == 0 ? 1u : 0u;
        }
        atomicMax(&r->w_dom_min, ~wmin);
        if (empty) atomicAdd(&r->dom_empty, empty);
      }
    }
    __syncthreads();
    phase_tick(d, 4, tclk);
    if (misc->err) goto fail;
  }
  return;
fail:
  if (tid == 0) set_err(d.err, misc->err, misc->where);
}

// CTAs of NT threads may use up to 128 registers a thread (512 / NT CTAs per
// SM by registers)
template <int NT, bool OTF>
__global__ void __launch_bounds__(NT, 512 / NT) k_tile(const __grid_constant__ Dev d, int stop) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int wsum[32];
  if (instance_failed(d.err)) return;
  tile_body<OTF>(d, int(blockIdx.x), stop, sm, wsum);
}

// Batched form: one CTA per (instance, domain) work item; the instance's
// parameters are copied into shared memory and advanced to sweep iteration
// `it` of the current batch call (buffers, sweep index, row).
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_tile_batch(const Dev* __restrict__ devs,
                                                   const BatchBase* __restrict__ base,
                                                   const int2* __restrict__ work, int it, int stop) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int wsum[32];
  __shared__ Dev sd;
  const int2 w = work[blockIdx.x];
  if (!base[w.x].active) return;
  if (threadIdx.x == 0) sd = at_iteration(devs[w.x], base[w.x], it);
  __syncthreads();
  if (instance_failed(sd.err)) return;
  tile_body<false>(sd, w.y, stop, sm, wsum);
}

// ---------------------------------------------------------------------------
// Shared-memory plan of one domain.  Fixed tables, then the leg table
// (legcap legs and a worm count each), then a union that holds the Step-3
// candidate pool and, beside it, the staged current configuration (phases
// 1-2), later the worm table and the Step-5 arrays.  The configuration is
// staged only when that costs no CTA per SM (CTAs per SM: the 228 KB of
// shared memory of an SM over the per-CTA size plus its 1 KB reserve).
//
// What a plan offers (its size, its legs) is computed from the reserve below:
// 2 KB of thresholds, 48 bytes a worm, two words a site or group and two
// bytes a group for each warp.  The domain tuner picks shapes by these sizes
// and a tuned instance's chain follows from its domain shape, so the reserve
// is kept; what the kernel lays out fits inside it (40 bytes a worm, 1 KB of
// thresholds, and the groups' member tables where they fit).
bool plan_tile_smem(Dev* d, double legs_want) {
  const int nds = d->dom_x * d->dom_y;
  // Step-5 chains: sub-blocks x temporal slabs
  const int nsub = sb_slots_host(d->dom_x, d->sub_block, d->ndx) * sb_slots_host(d->dom_y, d->sub_block, d->ndy) *
                   std::max(1, d->ntau);
  const int nb = std::max(nsub, nds) + 1;
  auto up16 = [](size_t x) { return (x + 15) & ~size_t(15); };
  size_t o = 0;
  d->sm_th = int(o); o = up16(o + 256 * sizeof(uint32_t));
  d->sm_zig = int(o); o = up16(o + size_t(kZigBytes));
  d->sm_off = int(o); o = up16(o + size_t(nds + 1) * sizeof(int));
  d->sm_base = int(o); o = up16(o + size_t(nds));
  d->sm_bcnt = int(o); o = up16(o + size_t(2 * nds) * sizeof(int));
  d->sm_boff = int(o); o = up16(o + size_t(2 * nds) * sizeof(int));
  d->sm_misc = int(o); o = up16(o + sizeof(Misc));
  d->sm_nbr = int(o); o = up16(o + size_t(6 * nds) * sizeof(uint16_t));
  d->sm_sub = int(o); o = up16(o + size_t(4 * nds) * sizeof(uint16_t));
  d->sm_tinfo = int(o); o = up16(o + size_t(6 * nds));
  const size_t fixed = o + 1024;  // (the reserve of the fixed tables)
  // worm side of the union, as reserved
  const int warps = nds <= 32 ? 2 : (nds <= 96 ? 4 : 16);
  const size_t worm_bytes = up16(size_t(d->wcap) * 24) + 4 * up16(size_t(d->wcap) * 2) + up16(size_t(d->wcap) * 16) +
                            2 * up16(size_t(nb) * sizeof(int)) + up16(size_t(warps) * size_t(nsub) * 2);
  // (on-the-fly windows: the worms of the current configuration by site, beside the pool)
  const size_t otf_bytes = d->win_half ? up16(size_t(nds + 1) * sizeof(int)) + up16(size_t(d->wcap) * 8) : 0;
  const size_t pool_bytes = up16(size_t(d->poolcap) * sizeof(uint64_t)) + otf_bytes;
  const long long want = std::min<long long>((long long)legs_want, 65000);
  const long long limit = (long long)kSmemLimit - 1024;
  // CTAs per SM: shared memory (1 KB the hardware reserves a CTA and up to
  // 1 KB of static shared memory), registers (up to 128 a thread: 2, 4 or 8
  // CTAs of 256, 128 or 64 threads) and the 32-CTA limit
  const long long by_regs = nds <= 32 ? 8 : (nds <= 96 ? 4 : 2);
  auto per_sm = [&](long long bytes) { return std::min(std::min((228LL * 1024) / (bytes + 2048), by_regs), 32LL); };
  // without staging
  const long long uni0 = (long long)std::max(worm_bytes, pool_bytes);
  const long long room = limit - (long long)fixed - uni0;
  if (room < 8 * 64) return false;
  // legs, their worm counts and (optionally) their partner indices
  auto legs_bytes = [&](long long c, bool part) {
    return (long long)up16(size_t(c) * 8) + (long long)up16(size_t(c)) + (part ? (long long)up16(size_t(c) * 2) : 0);
  };
  const long long capn = std::min<long long>(want, room / 9 - 16);
  const long long totn = (long long)fixed + legs_bytes(capn, false) + uni0;
  const long long capp = std::min<long long>(want, room / 11 - 16);
  const long long totp = (long long)fixed + legs_bytes(capp, true) + uni0;
  // the partner table only when it shrinks neither the leg table nor occupancy
  const bool part = capp == capn && per_sm(totp) >= per_sm(totn);
  const long long cap0 = part ? capp : capn;
  const long long tot0 = part ? totp : totn;
  // with staging: room for as many events as legs
  const long long stage = (long long)up16(size_t(nds + 1) * sizeof(int)) + (long long)up16(size_t(want) * 8);
  const long long uni1 = std::max((long long)worm_bytes, (long long)pool_bytes + stage);
  const long long tot1 = (long long)fixed + legs_bytes(want, part) + uni1;
  const bool staged = cap0 == want && tot1 <= limit && per_sm(tot1) >= per_sm(tot0);
  d->legcap = int(cap0);
  d->oldcap = staged ? int(want) : 0;
  d->sm_plan = int(fixed + size_t(legs_bytes(cap0, part)) + size_t(staged ? uni1 : uni0));
  d->sm_leg = int(o); o = up16(o + size_t(d->legcap) * sizeof(uint64_t));
  d->sm_wcnt = int(o); o = up16(o + size_t(d->legcap));
  d->use_part = part ? 1 : 0;
  d->sm_part = int(o); if (part) o = up16(o + size_t(d->legcap) * 2);
  d->sm_pool = int(o);
  d->sm_wmo = int(o + up16(size_t(d->poolcap) * sizeof(uint64_t)));
  d->sm_wm = int(d->sm_wmo + up16(size_t(nds + 1) * sizeof(int)));
  d->sm_soff = int(o + pool_bytes);
  d->sm_old = int(o + pool_bytes + up16(size_t(nds + 1) * sizeof(int)));
  d->sm_worm = int(o);
  size_t w = o + up16(size_t(d->wcap) * sizeof(WormRec));
  d->sm_ord = int(w); w = up16(w + size_t(d->wcap) * 2);
  d->sm_dn = int(w); w = up16(w + size_t(d->wcap) * 2);
  d->sm_idx = d->sm_nxt = int(w); w = up16(w + size_t(d->wcap) * 4);
  d->sm_fp = int(w); w = up16(w + size_t(d->wcap) * 8);
  d->sm_bkt = int(w); w = up16(w + size_t(nb) * sizeof(int));
  d->sm_fill = int(w); w = up16(w + size_t(nb) * sizeof(int));
  // the groups' member tables, where the reserve has room for them
  auto cells = [&](int slots) { return up16(size_t(nsub) * 2 * size_t(slots) * sizeof(uint16_t)); };
  const size_t counts = up16(size_t(nsub) * 3 * sizeof(int));
  d->gtab = w + cells(kGroupSlots) + counts <= size_t(d->sm_plan) ? 1 : 0;
  d->gslots = kGroupSlots;
  const double root = std::sqrt(std::max(0.0, double(d->wcap) - 64.0)) - 8.0, mean = root * root / nsub;
  const int want_slots = nsub > kScanGroups || mean < kScanMembers ? int(mean + 3.0 * std::sqrt(mean)) : 0;
  while (d->gtab && d->gslots < std::min(want_slots, 64) && w + cells(d->gslots + 4) + counts <= size_t(d->sm_plan))
    d->gslots += 4;
  d->sm_cell = int(w); w += d->gtab ? cells(d->gslots) : 0;
  d->sm_gcnt = int(w); w += d->gtab ? counts : 0;
  // and chains of worms by leg: as many heads as fit, a power of two
  d->sm_hash = int(w);
  d->ghash = 0;
  for (int h = 64; nsub <= kScanGroups && h <= 1024 && w + 8 * size_t(h) <= size_t(d->sm_plan); h *= 2) d->ghash = h;
  w += 8 * size_t(d->ghash);
  d->sm_total = int(std::max(w, o + pool_bytes + (staged ? size_t(stage) : 0)));
  return d->sm_plan <= kSmemLimit - 1024 && d->sm_total <= d->sm_plan;
}

int upload_zig_tile(const Zig& z) { return upload_constants(z); }

// CTA sizes of the sweep kernel, `ctas` domains being launched together (class
// 0: 64 threads, 1: 128, 2: 256, 3: 512).  The least class follows from the
// sites, up to 32 / 96 / more, and from the bound on the mean of the worms, which
// Step 5 gives a thread each: up to 48 for 64 threads; for 128 up to 96 of a
// domain of 32 sites, and up to 384, three turns of a thread, of a larger one,
// whose other phases fill the 128 threads (8x8 sites at beta t = 4, eta = 0.6,
// 1600 domains: 1.33 ms with 256 threads, 1.21 with 128; 4x4 at eta = 2: 6.66 and 9.1).
// There is no such bound above.  Beyond the least class a CTA
// takes as many threads as cost no other CTA its place on the SM, which its
// shared memory or the number of domains limits: the work of Step 3, Step 4 and
// the output is then spread over more warps, and a merge cut into more parts.
// A sweep, with the sites' classes alone and now: one 8x8 domain 127 -> 116 us,
// 9 of 8x12 sites 251 -> 224 us, 16 of 16x16 sites 277 -> 251 us, 144 of 4x4 sites
// 156 -> 145 us.
int tile_class(const Dev& d, int ctas) {
  const int sites = d.dom_x * d.dom_y;
  const double worms = d.beta * d.eta * sites;
  int c = sites <= 32 && worms <= 48.0 ? 0 : sites <= 96 && worms <= (sites <= 32 ? 96.0 : 384.0) ? 1 : 2;
  // CTAs an SM has to hold (registers hold 8 >> c of class c)
  const int by_smem = std::max(1, int((228LL * 1024) / (static_cast<long long>(d.sm_total) + 2048)));
  const int held = std::min(by_smem, (ctas - 1) / kSms + 1);
  while (c < 3 && (8 >> (c + 1)) >= held) ++c;
  return c;
}

int prepare_tile_batch(int cls, int smem) {
  cudaError_t e;
  switch (cls) {
    case 0: e = cudaFuncSetAttribute(k_tile_batch<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
    case 1: e = cudaFuncSetAttribute(k_tile_batch<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
    case 2: e = cudaFuncSetAttribute(k_tile_batch<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
    default: e = cudaFuncSetAttribute(k_tile_batch<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
  }
  return int(e);
}

int launch_tile_batch(int cls, const Dev* devs, const BatchBase* base, const int2* work, int n_work, int smem,
                      int it, int stop, void* stream) {
  if (n_work <= 0) return 0;
  const cudaStream_t st = cudaStream_t(stream);
  switch (cls) {
    case 0: k_tile_batch<64><<<n_work, 64, smem, st>>>(devs, base, work, it, stop); break;
    case 1: k_tile_batch<128><<<n_work, 128, smem, st>>>(devs, base, work, it, stop); break;
    case 2: k_tile_batch<256><<<n_work, 256, smem, st>>>(devs, base, work, it, stop); break;
    default: k_tile_batch<512><<<n_work, 512, smem, st>>>(devs, base, work, it, stop); break;
  }
  return int(cudaGetLastError());
}

template <int NT, bool OTF>
static int launch_tile_k(const Dev& d, int stop, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(k_tile<NT, OTF>, cudaFuncAttributeMaxDynamicSharedMemorySize, d.sm_total);
  if (e) return int(e);
  k_tile<NT, OTF><<<d.ndom, NT, d.sm_total, st>>>(d, stop);
  return int(cudaGetLastError());
}

int launch_tile(const Dev& d, int stop, void* stream) {
  const int cls = tile_class(d, d.ndom);
  const cudaStream_t st = cudaStream_t(stream);
  const bool otf = d.win_half > 0;
  switch (cls) {
    case 0: return otf ? launch_tile_k<64, true>(d, stop, st) : launch_tile_k<64, false>(d, stop, st);
    case 1: return otf ? launch_tile_k<128, true>(d, stop, st) : launch_tile_k<128, false>(d, stop, st);
    case 2: return otf ? launch_tile_k<256, true>(d, stop, st) : launch_tile_k<256, false>(d, stop, st);
    default: return otf ? launch_tile_k<512, true>(d, stop, st) : launch_tile_k<512, false>(d, stop, st);
  }
}

}  // namespace pmwa
