// pmwa_green.cu -- Supplement S-I estimators resolved by the component of Q.
//
//   k_rho_alpha       rho_b and rho_b+ at K equal-time slices, a lane a slice
//   k_green_tau_site  the two-point densities of one site (r = 0), lanes over its slices
//   k_green_tau_r     products of one-point densities of two sites (r >= 1)
//
// For X inside the interval I between two vertex legs of a site (p the state
// above the lower leg, q the state below the upper one, I1 the part of I
// below X, I2 the part above) the density of worms of type a at X is
//   rho_a(X) = eta <q| e^{I2 eta Q} Q_a e^{I1 eta Q} |p> / <q| e^{I eta Q} |p>,
// with Q_b = b taking 1 to 0 and Q_b+ = b+ taking 0 to 1.  One site's
// <a| e^{x Q} |b> is cosh x (a = b) or sinh x (a != b) = e^x F(a ^ b, x) / 2
// with F(0, x) = 2 + expm1(-2x) and F(1, x) = -expm1(-2x); the factors e^x
// cancel because I1 + I2 = I, counted in worm grid points (x = count beta eta
// / 2^59).  A site without vertex legs has no reference point on its circle:
// its density is the trace form eta Tr[Q_a e^{x Q}] / Tr[e^{x Q}] over the
// whole circle.  Two points on one interval take both operators inside the
// interval's matrix element; on two intervals the densities multiply.
//
// Every value is a fixed sequence of binary64 operations (no contraction), so
// the per-slice densities are reproducible bit for bit.
#include <cuda_runtime.h>

#include <algorithm>

#include "pmwa_device.cuh"

namespace pmwa {

namespace {

constexpr uint32_t kCntMaskG = 0x7fffffffu;
constexpr uint64_t kMask62G = kTwo62 - 1;

struct SliceInfo {
  int iv;          // event index of the lower leg, -1: the site has no legs
  int p, q;        // state above the lower leg, below the upper one
  uint64_t M, M1;  // worm points of the interval, and below the slice
  uint64_t off;    // pk distance from the lower leg up to the slice
  uint64_t pt;     // the slice's pk
};

__device__ __forceinline__ uint64_t slice_pk(int K, int k) {
  const uint64_t q62 = kTwo62 / uint64_t(K), r62 = kTwo62 % uint64_t(K);
  return uint64_t(k) * q62 + (uint64_t(k) * r62) / uint64_t(K);
}

__device__ __forceinline__ double Fsig(int sigma, uint64_t M, double XW) {
  const double e = expm1_det(__dmul_rn(-2.0, __dmul_rn(__ull2double_rn(M), XW)));
  return sigma ? -e : __dadd_rn(2.0, e);
}
__device__ __forceinline__ int q_in(int a) { return 1 - a; }
__device__ __forceinline__ int q_out(int a) { return a; }

// the interval of the slice at pt on a site whose legs are known to exist
// (lo: the last leg with pk <= pt, or the last leg of the circle)
__device__ __forceinline__ void slice_at(const uint64_t* Kk, int n, int lo, uint64_t pt, SliceInfo* z) {
  int hi = lo;
  for (int i = 1; i <= n; ++i) { hi = (lo + i) % n; if (!kworm(Kk[hi])) break; }
  const uint64_t plo = kpk(Kk[lo]), phi = kpk(Kk[hi]);
  z->iv = lo;
  z->p = kab(Kk[lo]);
  z->q = kbl(Kk[hi]);
  z->M = wpts(plo, phi);
  z->M1 = (pt == plo) ? 0 : wpts(plo, pt);
  z->off = (pt - plo) & kMask62G;
  z->pt = pt;
}

// the one-point densities of b and b+ at a slice from the three exponentials
// they share: e_lo, e_hi = expm1(-2x) of the interval's parts below and above
// the slice, den = F of the whole interval
struct Parts {
  double elo, ehi, den;
};
__device__ __forceinline__ double em1_of(uint64_t M, double XW) {
  return expm1_det(__dmul_rn(-2.0, __dmul_rn(__ull2double_rn(M), XW)));
}
__device__ __forceinline__ double F_of(int sigma, double e) { return sigma ? -e : __dadd_rn(2.0, e); }
__device__ __forceinline__ Parts parts_of(const SliceInfo& z, double XW) {
  return Parts{em1_of(z.M1, XW), em1_of(z.M - z.M1, XW), F_of(z.q ^ z.p, em1_of(z.M, XW))};
}
__device__ __forceinline__ double rho_one(const SliceInfo& z, const Parts& e, int a, double eta, double XW) {
  if (z.iv < 0) return __dmul_rn(eta, __ddiv_rn(Fsig(1, kTwo59, XW), __dmul_rn(2.0, Fsig(0, kTwo59, XW))));
  const double num = __dmul_rn(F_of(z.q ^ q_out(a), e.ehi), F_of(q_in(a) ^ z.p, e.elo));
  return __dmul_rn(eta, __ddiv_rn(num, __dmul_rn(2.0, e.den)));
}

// Q_a1 at slice z1 and Q_a2 at slice z2 of a site without vertex legs: the
// trace over the whole circle
__device__ __forceinline__ double rho_two_ring(const SliceInfo& z1, int a1, const SliceInfo& z2, int a2, double eta,
                                               double XW) {
  const uint64_t Ib = wpts(z1.pt, z2.pt), Ic = kTwo59 - Ib;
  const double num = __dmul_rn(Fsig(q_in(a2) ^ q_out(a1), Ib, XW), Fsig(q_in(a1) ^ q_out(a2), Ic, XW));
  return __dmul_rn(__dmul_rn(eta, eta), __ddiv_rn(num, __dmul_rn(4.0, Fsig(0, kTwo59, XW))));
}

// the slice k of site s found by bisection: the last vertex leg with pk <= pt, else the last leg of the
// circle; `last` is the site's last vertex leg (-1: none)
__device__ __forceinline__ void slice_one(const uint64_t* Kk, int n, int last, int K, int k, SliceInfo* z) {
  const uint64_t pt = slice_pk(K, k);
  if (last < 0) { z->iv = -1; z->p = z->q = 0; z->M = kTwo59; z->M1 = 0; z->off = 0; z->pt = pt; return; }
  int a = 0, b = n;  // first event with pk > pt
  while (a < b) {
    const int mid = (a + b) >> 1;
    if (kpk(Kk[mid]) <= pt) a = mid + 1; else b = mid;
  }
  int lo = last;
  for (int j = a - 1; j >= 0; --j) if (!kworm(Kk[j])) { lo = j; break; }
  slice_at(Kk, n, lo, pt, z);
}

// the site's last vertex leg (-1: none); worms are few, so it is near the end
__device__ __forceinline__ int last_leg(const uint64_t* Kk, int n) {
  int i = n - 1;
  while (i >= 0 && kworm(Kk[i])) --i;
  return i;
}

// sites s0 <= s < s0 + ns: rho[((s - s0) K + k) 2 + a]; iv[(s - s0) K + k]
// when iv is not null.  2^sh threads a site, one a slice, each found by
// bisection: a thread a site walked list and slices in one chain and wrote a
// line a lane.  The two densities of a slice share three exponentials.
// 128x128 sites, K = 32: 0.42 -> 0.19 ms.
__global__ void __launch_bounds__(128) k_rho_alpha(const __grid_constant__ Dev d, int K, int sh, int s0, int ns,
                                                   double* rho, int32_t* iv) {
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if ((t >> sh) >= ns) return;
  const int u = int(t >> sh), s = s0 + u, step = 1 << sh;
  const uint64_t* Kk = d.keyA + size_t(s) * d.cap;
  const int n = min(int(d.cntA[s] & kCntMaskG), d.cap), last = last_leg(Kk, n);
  for (int k = int(t) & (step - 1); k < K; k += step) {
    SliceInfo z;
    slice_one(Kk, n, last, K, k, &z);
    const Parts e = parts_of(z, d.XW);
    const size_t o = size_t(u) * K + k;
    const double r0 = rho_one(z, e, 0, d.eta, d.XW), r1 = rho_one(z, e, 1, d.eta, d.XW);
    *reinterpret_cast<double2*>(rho + 2 * o) = make_double2(r0, r1);
    if (iv) iv[o] = z.iv;
  }
}

// sums[dk] += sum over sites and slices k of the density of b+ at slice k and
// b at slice k + dk (mod K) on the same site, dk = 1..K-1; the one-point
// densities as k_rho_alpha lays them out go to rho if it is not null.
//
// One warp per site at a time.  Lanes over the slices first: interval, parts
// and one-point densities of every slice go to shared memory once.  Then
//   - lanes over dk: two slices on different intervals multiply their
//     densities (a product and a sum, no exponential);
//   - two slices on one interval need one more exponential, of the piece
//     between them, and it serves both orders (dk and K - dk).  The slices of
//     an interval follow one another, so slice k has run[k] partners behind
//     it; the pairs are laid over the lanes without gaps, 32 at a time, and
//     handed to the lanes of their dk.
// The binary64 pipe (2 lanes a cycle and SM) bounds it: with every pair's
// seven exponentials 128x128 sites and K = 32 took 18.1 ms, now 0.62 ms.
//
// With K <= 16 slices and many sites a warp takes 32 >> sh of them, 2^sh >= K lanes
// each (else one).  The call for 256x256 sites at rmax = 8, a thread a site -> a warp
// -> now: K = 2 0.296 -> 0.939 -> 0.166 ms, K = 4 1.08 -> 1.07 -> 0.25, K = 8 4.36
// -> 1.56 -> 0.53, K = 16 17.4 -> 2.24 -> 1.30.
constexpr int kTauWarps = 4;
struct TauSlices {
  double rb[kMaxGreenSlices], rbd[kMaxGreenSlices];              // densities of b, b+
  double elo[kMaxGreenSlices], ehi[kMaxGreenSlices], den[kMaxGreenSlices];
  uint64_t M1[kMaxGreenSlices];
  int iv[kMaxGreenSlices];
  uint8_t pq[kMaxGreenSlices];
  short first[kMaxGreenSlices + 32];                             // pairs before slice k's
  double v[2][32];
  short dk[32];
};
__global__ void __launch_bounds__(32 * kTauWarps) k_green_tau_site(const __grid_constant__ Dev d, int K, int sh,
                                                                  double* sums, double* rho) {
  __shared__ TauSlices sm[kTauWarps];
  const int G = 1 << sh, lane = threadIdx.x & (G - 1), sub = (threadIdx.x & 31) >> sh, wid = threadIdx.x >> 5;
  TauSlices& t = sm[wid];
  const int s0 = sub * G, f0 = sub * (G + 1), per = 32 >> sh;  // this site's places in t (G < 32: K <= G)
  const double eta2 = __dmul_rn(d.eta, d.eta);
  double acc[2] = {0.0, 0.0};  // dk = lane, lane + 32
  const long long step = (long long)gridDim.x * kTauWarps * per;
  for (long long b = ((long long)blockIdx.x * kTauWarps + wid) * per; b < d.N; b += step) {
    const long long s = b + sub;
    const bool act = s < d.N;
    const uint64_t* Kk = d.keyA + size_t(act ? s : 0) * d.cap;
    const int n = act ? min(int(d.cntA[s] & kCntMaskG), d.cap) : 0, last = act ? last_leg(Kk, n) : -1;
    __syncwarp();
    for (int k = lane; act && k < K; k += G) {
      SliceInfo z;
      slice_one(Kk, n, last, K, k, &z);
      const Parts e = parts_of(z, d.XW);
      const double b0 = rho_one(z, e, 0, d.eta, d.XW), b1 = rho_one(z, e, 1, d.eta, d.XW);
      t.rb[s0 + k] = b0;
      t.rbd[s0 + k] = b1;
      if (rho) *reinterpret_cast<double2*>(rho + (size_t(s) * K + k) * 2) = make_double2(b0, b1);
      t.elo[s0 + k] = e.elo;
      t.ehi[s0 + k] = e.ehi;
      t.den[s0 + k] = e.den;
      t.M1[s0 + k] = z.M1;
      t.iv[s0 + k] = z.iv;
      t.pq[s0 + k] = uint8_t(z.p | (z.q << 1));
    }
    __syncwarp();
    // no legs: every pair by the trace over the circle; else different intervals
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int dk = lane + G * h;
      if (!act || dk == 0 || dk >= K) continue;
      double a = 0.0;
      int j = dk;
      for (int k = 0; k < K; ++k) {
        if (last < 0) {
          SliceInfo z1, z2;
          slice_one(Kk, n, last, K, k, &z1);
          slice_one(Kk, n, last, K, j, &z2);
          acc[h] = __dadd_rn(acc[h], rho_two_ring(z1, 1, z2, 0, d.eta, d.XW));
        } else if (t.iv[s0 + k] != t.iv[s0 + j]) {
          a = __dadd_rn(a, __dmul_rn(t.rbd[s0 + k], t.rb[s0 + j]));
        }
        if (++j == K) j = 0;
      }
      if (last >= 0) acc[h] = __dadd_rn(acc[h], a);
    }
    // one interval: slice k with the slices behind it up to the interval's end
    int mine[2], sum = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 2 * lane + h;
      int run = 0;
      if (last >= 0 && k < K) {
        int j = k + 1 == K ? 0 : k + 1;
        while (run < K - 1 && t.iv[s0 + j] == t.iv[s0 + k] && t.M1[s0 + j] >= t.M1[s0 + k]) {
          ++run;
          j = j + 1 == K ? 0 : j + 1;
        }
      }
      mine[h] = run;
      sum += run;
    }
    int before = sum;
    for (int o = 1; o < G; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, before, o, G);
      if (lane >= o) before += x;
    }
    const int total = __shfl_sync(0xffffffffu, before, G - 1, G);
    before -= sum;
    if (2 * lane <= K) t.first[f0 + 2 * lane] = short(before);
    if (2 * lane + 1 <= K) t.first[f0 + 2 * lane + 1] = short(before + mine[0]);
    if (lane == G - 1 && K == 2 * G) t.first[f0 + K] = short(total);
    __syncwarp();
    const int most = int(__reduce_max_sync(0xffffffffu, unsigned(total)));
    for (int p0 = 0; p0 < most; p0 += G) {
      const int p = p0 + lane;
      if (p < total) {
        int lo = 0, hi = K;  // the slice k with first[k] <= p < first[k + 1]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (t.first[f0 + mid] <= p) lo = mid; else hi = mid;
        }
        const int k = lo, dk = p - t.first[f0 + k] + 1, j = k + dk >= K ? k + dk - K : k + dk;
        const double eb = em1_of(t.M1[s0 + j] - t.M1[s0 + k], d.XW), den = __dmul_rn(4.0, t.den[s0 + k]);
        const int pp = t.pq[s0 + k] & 1, qq = t.pq[s0 + k] >> 1;
        // lower operator on k, upper on j: b+ on k and b on j, then the other way round
        auto v = [&](int aL, int aU) {
          const double num = __dmul_rn(__dmul_rn(F_of(qq ^ q_out(aU), t.ehi[s0 + j]), F_of(q_in(aU) ^ q_out(aL), eb)),
                                       F_of(q_in(aL) ^ pp, t.elo[s0 + k]));
          return __dmul_rn(eta2, __ddiv_rn(num, den));
        };
        t.v[0][s0 % 32 + lane] = v(1, 0);
        t.v[1][s0 % 32 + lane] = v(0, 1);
        t.dk[s0 % 32 + lane] = short(dk);
      }
      __syncwarp();
      for (int i = 0; i < min(G, total - p0); ++i) {
        const int dk = t.dk[s0 % 32 + i];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (lane + G * h == dk) acc[h] = __dadd_rn(acc[h], t.v[0][s0 % 32 + i]);
          if (lane + G * h == K - dk) acc[h] = __dadd_rn(acc[h], t.v[1][s0 % 32 + i]);
        }
      }
      __syncwarp();
    }
  }
  __syncwarp();
  t.rb[threadIdx.x & 31] = acc[0];  // (dk = lane of each of the warp's sites)
  t.rb[(threadIdx.x & 31) + 32] = acc[1];
  __syncthreads();
  const int dk = threadIdx.x;
  if (dk > 0 && dk < K) {  // (K <= 64 <= the block's threads)
    double v = 0.0;
    const int at = dk < G ? dk : dk - G + 32;  // (dk >= G: its second sum; one site a warp then, or K = 2 G)
    for (int w = 0; w < kTauWarps; ++w)
      for (int q = 0; q < per; ++q) v = __dadd_rn(v, sm[w].rb[at + q * G]);
    atomicAdd(sums + dk, v);
  }
}

// sums[(dir (rmax + 1) + r) K + dk] += sum_{i,k} rho_b(i + r e_dir, k + dk)
// rho_b+(i, k), dir = blockIdx.y, r = 8 blockIdx.z + 1 .. + 8 up to rmax.  One
// warp takes a site i: its K densities of b+ and, for each r, the K densities
// of b of site j go to shared memory (one coalesced row each), and lane dk
// runs over k with one fused multiply-add each and keeps the sums of its dk in
// registers from site to site: the binary64 pipe is the bound (N 2 rmax K^2
// multiply-adds; 128x128 sites, K = 32, rmax = 8: 0.43 ms of it; measured 0.47
// ms, 1.74 ms with a thread a site and two lines a lane for each product).
// Up to 16 slices a warp takes 32 >> sh sites, 2^sh lanes each.
constexpr int kTauRowWarps = 8, kTauRowR = 8;
__global__ void __launch_bounds__(32 * kTauRowWarps) k_green_tau_r(int Lx, int Ly, int K, int sh, int rmax,
                                                                  const double* __restrict__ rho, double* sums) {
  extern __shared__ __align__(16) double tsm[];
  const int G = 1 << sh, lane = threadIdx.x & (G - 1), group = threadIdx.x >> sh, groups = int(blockDim.x) >> sh;
  const int dir = int(blockIdx.y), r0 = int(blockIdx.z) * kTauRowR;
  double* bd = tsm + size_t(group) * 3 * K;  // K densities of b+, then 2 K of b (twice over)
  double* b = bd + K;
  double* part = tsm + size_t(groups) * 3 * K;  // the block's sums, [kTauRowR][K]
  for (int i = threadIdx.x; i < kTauRowR * K; i += blockDim.x) part[i] = 0.0;
  double acc[kTauRowR][2] = {};
  const long long N = (long long)Lx * Ly, step = (long long)gridDim.x * groups;
  for (long long i0 = (long long)blockIdx.x * groups; i0 < N; i0 += step) {
    const long long i = i0 + group;
    const bool act = i < N;
    const int x = int(act ? i % Lx : 0), y = int(act ? i / Lx : 0);
    if (act)
      for (int k = lane; k < K; k += G) bd[k] = rho[(size_t(i) * K + k) * 2 + 1];
#pragma unroll
    for (int e = 0; e < kTauRowR; ++e) {
      const int r = r0 + e + 1;
      if (r > rmax) break;
      const size_t j = dir == 0 ? size_t(y) * Lx + (x + r) % Lx : size_t((y + r) % Ly) * Lx + x;
      __syncwarp();
      if (act)
        for (int k = lane; k < K; k += G) b[k] = b[k + K] = rho[(j * K + k) * 2];
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int dk = lane + G * h;
        if (act && dk < K) {
          double a = 0.0;
          for (int k = 0; k < K; ++k) a = fma(b[k + dk], bd[k], a);
          acc[e][h] += a;
        }
      }
    }
    __syncwarp();
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < kTauRowR; ++e)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double v = acc[e][h];  // (the warp's sites first: their sums go to one address)
      for (int o = G; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (r0 + e + 1 <= rmax && lane + G * h < K && (threadIdx.x & 31) < G) atomicAdd(part + e * K + lane + G * h, v);
    }
  __syncthreads();
  const int nr = min(kTauRowR, rmax - r0);
  for (int i = threadIdx.x; i < nr * K; i += blockDim.x)
    atomicAdd(sums + (size_t(dir) * (rmax + 1) + r0 + 1) * K + i, part[i]);
}

// Supplement S-I n-point functions of distinct sites at equal time: tuple j
// holds n sites (sites[j n + c]); out[j] = (sum_k prod_c rho[s_c K + k] / K)
// / eta^n, the product in tuple order from 1.0, the sum over the slices in
// order, eta^n by n multiplications from 1.0.  Distinct sites never share an
// interval, so the densities multiply.
__global__ void k_npoint(int K, int n, int m, const double* __restrict__ rho, const int32_t* __restrict__ sites,
                         double eta, double* out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  const int32_t* t = sites + size_t(j) * n;
  double acc = 0.0;
  for (int k = 0; k < K; ++k) {
    double p = 1.0;
    for (int c = 0; c < n; ++c) p = __dmul_rn(p, rho[size_t(t[c]) * K + k]);
    acc = __dadd_rn(acc, p);
  }
  double etan = 1.0;
  for (int c = 0; c < n; ++c) etan = __dmul_rn(etan, eta);
  out[j] = __ddiv_rn(__ddiv_rn(acc, double(K)), etan);
}

// Joint density of g operators Q_a[0..g) at the points z[idx[0..g)] of one
// interval, in time order (Supplement S-I with every operator inserted in the
// interval's matrix element):
//   eta^g <q| e^{I_g Q} Q_a[g-1] ... Q_a[0] e^{I_0 Q} |p> / <q| e^{I Q} |p>
//     = eta^g F(in_a[0] ^ p, I_0) prod_j F(in_a[j] ^ out_a[j-1], I_j) F(q ^ out_a[g-1], I_g)
//       / (2^g F(q ^ p, I)),
// I_0 the worm points below the first point, I_j between points j-1 and j,
// I_g above the last; on a site without legs the cyclic trace
//   eta^g prod_j F(in_a[j+1] ^ out_a[j], I_j) / (2^g F(0, 2^59)),
// I_j between points j and j + 1 and the last piece closing the circle.
__device__ double rho_interval(const SliceInfo* z, const int* idx, const int* a, int g, double eta, double XW) {
  double num = 1.0, etag = 1.0, den = 1.0;
  for (int j = 0; j < g; ++j) { etag = __dmul_rn(etag, eta); den = __dmul_rn(den, 2.0); }
  const SliceInfo& z0 = z[idx[0]];
  if (z0.iv < 0) {
    uint64_t used = 0;
    for (int j = 0; j < g; ++j) {
      const int nx = (j + 1) % g;
      const uint64_t piece = (j + 1 < g) ? wpts(z[idx[j]].pt, z[idx[j + 1]].pt) : kTwo59 - used;
      used += piece;
      num = __dmul_rn(num, Fsig(q_in(a[nx]) ^ q_out(a[j]), piece, XW));
    }
    return __dmul_rn(etag, __ddiv_rn(num, __dmul_rn(den, Fsig(0, kTwo59, XW))));
  }
  num = Fsig(q_in(a[0]) ^ z0.p, z[idx[0]].M1, XW);
  for (int j = 1; j < g; ++j)
    num = __dmul_rn(num, Fsig(q_in(a[j]) ^ q_out(a[j - 1]), z[idx[j]].M1 - z[idx[j - 1]].M1, XW));
  num = __dmul_rn(num, Fsig(z0.q ^ q_out(a[g - 1]), z0.M - z[idx[g - 1]].M1, XW));
  return __dmul_rn(etag, __ddiv_rn(num, __dmul_rn(den, Fsig(z0.q ^ z0.p, z0.M, XW))));
}

// Supplement S-I n-point functions resolved by the component of Q at
// arbitrary times: tuple j holds n points (site, slice, component) at
// pts[(j n + c) 3 ..]; out[j] = (sum over the K cyclic shifts of the slices of
// the product over intervals of the joint density of their points) / K /
// eta^n.  The points are grouped by interval (site and lower vertex leg, or
// the whole circle of a site without legs) in order of first appearance, each
// group's points in time order (insertion sort by the offset from the lower
// leg, or by time point on a site without legs).
// 2^sh lanes a tuple, one a shift at a time, whose products are then added in
// order: the fewest that fill the machine (tuple_lanes).  A warp a tuple, few of
// whose lanes have a shift or whose lanes all add the 32 products, is bound by
// the instructions it issues once there are many tuples; a thread a tuple runs K
// dependent searches one after the other.  4096 tuples of 3, K = 32: a thread
// 0.74, a warp 0.14 ms; the call for 10^6 tuples of 1 at K = 1 / 8 / 32: a thread
// 1.79 / 3.93 / 11.4, a warp 11.2 / 13.4 / 15.1, now 1.77 / 3.87 / 11.2 ms.
__global__ void __launch_bounds__(64) k_npoint_alpha(const __grid_constant__ Dev d, int K, int sh, int n, int m,
                                                     const int32_t* __restrict__ pts, double* out) {
  const long long id = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> sh;
  const int lanes = 1 << sh, lane = threadIdx.x & (lanes - 1);
  const long long j = id < m ? id : m - 1;  // (the last warp's spare lanes repeat the last tuple)
  const int32_t* t = pts + size_t(j) * size_t(n) * 3;
  int last[kMaxNpoint], cnt[kMaxNpoint];
  for (int c = 0; c < n; ++c) {
    cnt[c] = min(int(d.cntA[t[3 * c]] & kCntMaskG), d.cap);
    last[c] = last_leg(d.keyA + size_t(t[3 * c]) * d.cap, cnt[c]);
  }
  double acc = 0.0;
  for (int k0 = 0; k0 < K; k0 += lanes) {
    const int k = k0 + lane;
    double prod = 1.0;
    if (k < K) {
      SliceInfo z[kMaxNpoint];
      for (int c = 0; c < n; ++c)
        slice_one(d.keyA + size_t(t[3 * c]) * d.cap, cnt[c], last[c], K, (t[3 * c + 1] + k) % K, &z[c]);
      unsigned done = 0;
      for (int c = 0; c < n; ++c) {
        if (done & (1u << c)) continue;
        int idx[kMaxNpoint], a[kMaxNpoint], g = 0;
        for (int e = c; e < n; ++e)
          if (!(done & (1u << e)) && t[3 * e] == t[3 * c] && z[e].iv == z[c].iv) { idx[g++] = e; done |= 1u << e; }
        const bool ring = z[c].iv < 0;
        for (int i = 1; i < g; ++i)
          for (int q = i; q > 0; --q) {
            const uint64_t ka = ring ? z[idx[q]].pt : z[idx[q]].off, kb = ring ? z[idx[q - 1]].pt : z[idx[q - 1]].off;
            if (ka < kb) { const int tmp = idx[q]; idx[q] = idx[q - 1]; idx[q - 1] = tmp; } else break;
          }
        for (int i = 0; i < g; ++i) a[i] = t[3 * idx[i] + 2];
        prod = __dmul_rn(prod, rho_interval(z, idx, a, g, d.eta, d.XW));
      }
    }
    if (sh == 0)
      acc = __dadd_rn(acc, prod);
    else
      for (int i = 0; i < min(lanes, K - k0); ++i) acc = __dadd_rn(acc, __shfl_sync(0xffffffffu, prod, i, lanes));
  }
  double etan = 1.0;
  for (int c = 0; c < n; ++c) etan = __dmul_rn(etan, d.eta);
  if (lane == 0 && id < m) out[j] = __ddiv_rn(__ddiv_rn(acc, double(K)), etan);
}

// log2 of a tuple's lanes: whole warps for few tuples (two in one warp wait for
// each other's branches), fewer as soon as the tuples have a thread for each of
// a full machine's 152 x 1024, and no more than there are slices once those fill
// half of it
int tuple_lanes(int K, int m) {
  const long long full = 152 * 1024, tuples = m;
  const int own = slice_lanes(K);
  int sh = 5;
  while (sh > 0 && (tuples << (sh - 1)) >= full) --sh;
  return sh > own && (tuples << own) >= full / 2 ? own : sh;
}

}  // namespace

int launch_npoint_alpha(const Dev& d, int K, int n, int m, const int32_t* pts, double* out, void* stream) {
  if (m <= 0) return 0;
  const int sh = tuple_lanes(K, m);
  k_npoint_alpha<<<unsigned(((static_cast<long long>(m) << sh) + 63) / 64), 64, 0, cudaStream_t(stream)>>>(d, K, sh, n, m,
                                                                                                      pts, out);
  return int(cudaGetLastError());
}

int launch_npoint(int K, int n, int m, const double* rho, const int32_t* sites, double eta, double* out,
                  void* stream) {
  if (m <= 0) return 0;
  k_npoint<<<(m + 127) / 128, 128, 0, cudaStream_t(stream)>>>(K, n, m, rho, sites, eta, out);
  return int(cudaGetLastError());
}

// this translation unit's copy of the constant tables (expm1_det reads them)
int upload_zig_green(const Zig& z) { return upload_constants(z); }

int launch_rho_alpha(const Dev& d, int K, int s0, int ns, double* rho, int32_t* iv, void* stream) {
  const int sh = slice_lanes(K);
  k_rho_alpha<<<unsigned((((long long)ns << sh) + 127) / 128), 128, 0, cudaStream_t(stream)>>>(d, K, sh, s0, ns, rho,
                                                                                             iv);
  return int(cudaGetLastError());
}

int launch_green_tau(const Dev& d, int K, int rmax, double* rho, double* sums, void* stream) {
  cudaStream_t st = cudaStream_t(stream);
  const size_t nsum = size_t(2) * size_t(rmax + 1) * size_t(K);
  if (cudaMemsetAsync(sums, 0, nsum * sizeof(double), st) != cudaSuccess) return int(cudaGetLastError());
  // (a warp a site while all sites run at once: two in a warp wait for each other)
  const int sh = d.N <= 152 * 4 * kTauWarps ? 5 : slice_lanes(K), per = 32 >> sh;
  if (K > 1) {
    const int bs = std::min((d.N + kTauWarps * per - 1) / (kTauWarps * per), 152 * 4);
    k_green_tau_site<<<bs, 32 * kTauWarps, 0, st>>>(d, K, sh, sums, rmax > 0 ? rho : nullptr);
    if (cudaGetLastError() != cudaSuccess) return PMWA_ECUDA;
  } else if (rmax > 0) {  // one slice: no pairs of slices on one site, the densities alone
    if (const int rc = launch_rho_alpha(d, K, 0, d.N, rho, nullptr, stream)) return rc;
  }
  if (rmax > 0) {
    const int groups = kTauRowWarps * per;
    const size_t smem = (size_t(3 * groups) + kTauRowR) * size_t(K) * sizeof(double);
    const dim3 grid(std::min((d.N + groups - 1) / groups, 152 * 3), 2, (rmax + kTauRowR - 1) / kTauRowR);
    k_green_tau_r<<<grid, 32 * kTauRowWarps, smem, st>>>(d.Lx, d.Ly, K, sh, rmax, rho, sums);
  }
  return int(cudaGetLastError());
}

}  // namespace pmwa
