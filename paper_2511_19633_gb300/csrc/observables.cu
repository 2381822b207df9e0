// Per-event observables (Section 4.1 of arXiv:2511.19633; e+e- event shapes
// as in GAPS 1) and weighted histograms. Each block takes chunks of up to 256
// events: per-event scalar work (the colourless final state, the boson
// kinematics, the output and the histogram bins) runs with one thread per
// event; the clusterings run four events a warp with eight lanes each and the
// event's final-state momenta in the warp's shared memory (a larger event,
// alone, with all lanes), the lanes sharing the pair scans and the thrust
// candidates. Every value is formed with the same operations, in the same
// order, as a plain one-thread evaluation, and every minimum is taken in the
// order of a plain scan (lowest index on ties), so the results do not depend on
// the number of lanes. Histograms are privatised per block in shared memory and
// merged with global atomics.
//
// Bound by FP32 issue and latency: a clustering is a chain of steps, each with
// a minimum over the lanes and a few functions of one pseudo-jet (log, atan2),
// and most events have fewer than 16 pseudo-jets. Four events a warp share the
// instructions of those steps, and warps that take events by size stay in step
// and end together; the minimum over candidates of the few pseudo-jets whose
// neighbour changed is shared by an event's lanes (all of them scanned by one
// lane each: 1.49 ms for 150 001 p p events, 1.04 ms shared, 0.58 ms with the
// events by size). One event a warp, 32 events a warp in turn: 1.55 ms, 1.24 ms
// for 4096 p p events (0.17 now), 8.6 ms for 30 000 p p events in FP64 (1.8). The
// division by R^2 in the distance is needed in place: comparing the dividends
// and dividing only on near ties took 0.69 ms (a branch in the scans).
#include "physics_fp64.cuh"

namespace gaps {


namespace {

constexpr int kMaxFinal = 128;
constexpr int kObsWarps = 8;  // warps per block, each on its own group of events
constexpr unsigned kFull = 0xffffffffu;
static_assert(GAPS_NOBS == 8, "the kernel writes eight observables per event");

// events that a warp clusters at a time, the lanes of each and the pseudo-jets
// it may have there
constexpr int kObsGroups = 4;
constexpr int kObsLanes = 32 / kObsGroups;
constexpr int kObsSmall = kMaxFinal / kObsGroups;
constexpr int kObsSizes = 2 * (kObsSmall + 1) + 1;  // alone, and each size of the two kinds
constexpr int kObsThreads = kObsWarps * 32;

// an event of up to N pseudo-jets: the coloured final state, its anti-kT
// kinematics and nearest neighbours
template <typename R, int N>
struct ObsEvent {
  static constexpr int kWords = N / 32;
  R ps[N][4];
  R ipt2[N], y[N], phi[N], nnd[N];  // (ipt2: 1 / pT^2)
  int nnj[N];
  uint32_t am[kWords];  // remaining pseudo-jets (the pair scans index it by word)
};
// a warp's events
template <typename R>
union ObsWarp {
  ObsEvent<R, kMaxFinal> one;
  ObsEvent<R, kObsSmall> four[kObsGroups];
};

// The GW lanes that work on an event. The teams of a warp go through a
// clustering in step (every collective names the whole warp), so that they
// share its instructions whatever their events' sizes.
template <int GW>
struct ObsTeam {
  int lane, shift;  // lane in the team, the team's first lane
  __device__ __forceinline__ explicit ObsTeam(int warp_lane)
      : lane(warp_lane & (GW - 1)), shift(warp_lane & ~(GW - 1) & 31) {}
  // the predicate of the team's lanes, lane 0 in bit 0
  __device__ __forceinline__ uint32_t ballot(bool p) const {
    const uint32_t all = __ballot_sync(kFull, p) >> shift;
    return GW == 32 ? all : all & ((1u << (GW & 31)) - 1u);
  }
};

template <typename R>
__device__ __forceinline__ R norm3(const R* p) {
  return sqrt(p[1] * p[1] + p[2] * p[2] + p[3] * p[3]);
}

// a team's lexicographic minimum of (v, k); v is never NaN
template <int GW, typename R>
__device__ __forceinline__ void team_argmin(const ObsTeam<GW>& T, R& v, int& k) {
#pragma unroll
  for (int off = GW / 2; off > 0; off >>= 1) {
    const R ov = __shfl_xor_sync(kFull, v, off);
    const int ok = __shfl_xor_sync(kFull, k, off);
    if (ov < v || (ov == v && ok < k)) { v = ov; k = ok; }
  }
}

template <int GW, typename R>
__device__ __forceinline__ R team_fmax(const ObsTeam<GW>& T, R v) {
#pragma unroll
  for (int off = GW / 2; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(kFull, v, off));
  return v;
}

// bits of word w of an index mask that stand for indices above i
__device__ __forceinline__ uint32_t above(int i, int w) {
  const int lo = 32 * w;
  if (i < lo) return kFull;
  if (i >= lo + 31) return 0u;
  return kFull << (i - lo + 1);
}

// |p| of the event's momenta (kept in nnd) and, in FP32, their directions, which
// the pair distances below use
template <typename R, int N>
__device__ __forceinline__ void keep_norm(ObsEvent<R, N>& W, int i) {
  const R n = norm3(W.ps[i]);
  W.nnd[i] = n;
  if constexpr (sizeof(R) == 4) {
    W.ipt2[i] = W.ps[i][1] / n;
    W.y[i] = W.ps[i][2] / n;
    W.phi[i] = W.ps[i][3] / n;
  }
}

// thrust: all 2^(n-1) subsets for n <= 12 (total momentum is zero), otherwise
// the exact construction from candidate axes p_i x p_j with the four sign
// choices of i and j; the lanes share the candidates, the maximum is exact
template <int GW, typename R, int N>
__device__ __forceinline__ R thrust(const ObsTeam<GW>& T, const ObsEvent<R, N>& W, int n) {
  R sum = 0;
  for (int i = 0; i < n; ++i) sum += W.nnd[i];
  const bool any = n >= 2 && sum > R(0);
  R best = 0;
  if (n <= 12) {
    const uint32_t subsets = any ? 1u << (n - 1) : 0u;
    for (uint32_t m = T.lane; m < subsets; m += GW) {
      R v0 = 0, v1 = 0, v2 = 0;
      for (int i = 0; i < n; ++i)
        if ((m >> i) & 1u) { v0 += W.ps[i][1]; v1 += W.ps[i][2]; v2 += W.ps[i][3]; }
      R l = sqrt(v0 * v0 + v1 * v1 + v2 * v2);
      best = fmax(best, l);
    }
  } else if (any) {
    for (int i = 0; i < n; ++i) {
      for (int j = i + 1 + T.lane; j < n; j += GW) {
        const R* pi = W.ps[i];
        const R* pj = W.ps[j];
        R ax0 = pi[2] * pj[3] - pi[3] * pj[2];
        R ax1 = pi[3] * pj[1] - pi[1] * pj[3];
        R ax2 = pi[1] * pj[2] - pi[2] * pj[1];
        R b0 = 0, b1 = 0, b2 = 0;
        for (int k = 0; k < n; ++k) {
          if (k == i || k == j) continue;
          R d = W.ps[k][1] * ax0 + W.ps[k][2] * ax1 + W.ps[k][3] * ax2;
          if (d > R(0)) { b0 += W.ps[k][1]; b1 += W.ps[k][2]; b2 += W.ps[k][3]; }
        }
        for (int si = 0; si < 2; ++si) {
          for (int sj = 0; sj < 2; ++sj) {
            R v0 = b0, v1 = b1, v2 = b2;
            if (si) { v0 += pi[1]; v1 += pi[2]; v2 += pi[3]; }
            if (sj) { v0 += pj[1]; v1 += pj[2]; v2 += pj[3]; }
            R l = sqrt(v0 * v0 + v1 * v1 + v2 * v2);
            best = fmax(best, l);
          }
        }
      }
    }
  }
  best = team_fmax(T, best);
  return any ? R(2) * best / sum : R(1);
}

// y_ij of the Durham algorithm from the kept norms and directions
template <typename R, int N>
__device__ __forceinline__ R durham_yij(const ObsEvent<R, N>& W, int i, int j, R evis2) {
  R omc;  // 1 - cos(theta_ij)
  if constexpr (sizeof(R) == 8) {
    omc = R(1) -
          (W.ps[i][1] * W.ps[j][1] + W.ps[i][2] * W.ps[j][2] + W.ps[i][3] * W.ps[j][3]) / (W.nnd[i] * W.nnd[j]);
  } else {
    // |n_i - n_j|^2 / 2 keeps the relative precision for collinear pairs
    R d0 = W.ipt2[i] - W.ipt2[j], d1 = W.y[i] - W.y[j], d2 = W.phi[i] - W.phi[j];
    omc = R(0.5) * (d0 * d0 + d1 * d1 + d2 * d2);
  }
  R emin = fmin(W.ps[i][0], W.ps[j][0]);
  return R(2) * emin * emin * omc / evis2;
}

// Durham clustering, E-scheme; y23, y34 = smallest y_ij when 3 -> 2, 4 -> 3.
// Each step takes the smallest y_ij over the remaining pairs in row-major
// order of the pair (lowest i, then lowest j, on ties); a merged pair keeps
// the slot of i, and j leaves. The lanes share the pairs of the remaining ones,
// which nnj lists in ascending order.
template <int GW, typename R, int N>
__device__ __forceinline__ void durham(const ObsTeam<GW>& T, ObsEvent<R, N>& W, int m, R& y23, R& y34) {
  const int lane = T.lane;
  R evis = 0;
  for (int i = 0; i < m; ++i) evis += W.ps[i][0];
  const R evis2 = evis * evis;
  y23 = 0; y34 = 0;
  for (int i = lane; i < m; i += GW) W.nnj[i] = i;
  __syncwarp();
  while (__any_sync(kFull, m > 2)) {
    R ymin = R(INFINITY);
    int key = INT_MAX;
    const int pairs = m > 2 ? m * (m - 1) / 2 : 0;
    for (int p = lane; p < pairs; p += GW) {
      // the pair a < b with p = b (b - 1) / 2 + a
      int b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);
      if (b * (b - 1) / 2 > p) --b;
      const int a = p - b * (b - 1) / 2, i = W.nnj[a], j = W.nnj[b];
      const R yij = durham_yij(W, i, j, evis2);
      const int k = i * kMaxFinal + j;
      if (yij < ymin || (yij == ymin && key != INT_MAX && k < key)) { ymin = yij; key = k; }
    }
    team_argmin(T, ymin, key);
    if (key == INT_MAX) m = 0;  // no finite y_ij (degenerate momenta)
    const bool on = m > 2;
    const int bi = on ? key / kMaxFinal : 0, bj = on ? key % kMaxFinal : 0;
    if (on) {
      if (m == 3) y23 = ymin;
      if (m == 4) y34 = ymin;
      if (lane < 4) W.ps[bi][lane] += W.ps[bj][lane];
    }
    __syncwarp();
    // bi's norm, and bj out of the list
    if (on && lane == 0) keep_norm(W, bi);
    for (int i0 = 0; __any_sync(kFull, on && i0 < m - 1); i0 += GW) {
      const int i = i0 + lane;
      const bool in = on && i < m - 1;
      const int here = in ? W.nnj[i] : 0, next = in ? W.nnj[i + 1] : 0;
      __syncwarp();
      if (in && here >= bj) W.nnj[i] = next;
      __syncwarp();
    }
    m -= 1;
    __syncwarp();
  }
}

template <typename R>
__device__ __forceinline__ void jet_kin(const R* p, R& ipt2, R& y, R& phi) {
  ipt2 = R(1) / (p[1] * p[1] + p[2] * p[2]);
  if constexpr (sizeof(R) == 8) y = R(0.5) * log((p[0] + p[3]) / (p[0] - p[3]));
  else y = R(0.5) * log(p[0] / p[3]);
  phi = atan2(p[2], p[1]);
}

template <typename R>
__device__ __forceinline__ R jet_pz(const R* p) {
  if constexpr (sizeof(R) == 8) return p[3];
  else return R(0.5) * (p[0] - p[3]);
}

// anti-kT distance of pseudo-jets i, j from their cached kinematics
template <typename R>
__device__ __forceinline__ R akt_dij(const R* ipt2, const R* y, const R* phi, int i, int j, R R2) {
  R dphi = fabs(phi[i] - phi[j]);
  if (dphi > R(kPi)) dphi = R(2.0 * kPi) - dphi;
  R dr2 = (y[i] - y[j]) * (y[i] - y[j]) + dphi * dphi;
  return fmin(ipt2[i], ipt2[j]) * dr2 / R2;
}

// nearest remaining neighbour of i among j > i (lowest j on ties)
template <typename R, int N>
__device__ __forceinline__ void akt_nn(ObsEvent<R, N>& W, int i, R R2) {
  R best = R(INFINITY);
  int bj = -1;
  for (int w = i >> 5; w < ObsEvent<R, N>::kWords; ++w) {
    uint32_t bits = W.am[w] & above(i, w);
    while (bits) {
      const int j = 32 * w + __ffs(bits) - 1;
      bits &= bits - 1;
      R d = akt_dij(W.ipt2, W.y, W.phi, i, j, R2);
      if (d < best) { best = d; bj = j; }
    }
  }
  W.nnd[i] = best;
  W.nnj[i] = bj;
}

// anti-kT R (Cacciari, Salam, Soyez 2008), E-scheme, rapidity-azimuth
// distance, over the m0 pseudo-jets of W.ps (those with zero transverse
// momentum are left out). Nearest-neighbour bookkeeping (O(n^2)): every
// remaining pseudo-jet keeps its nearest neighbour among the later ones, and
// each step takes the smallest of all beam and neighbour distances in the
// order of a full scan (beam distance of i, then its neighbour, i ascending),
// so the clustering sequence equals the brute-force one. Reports the number
// of jets with pT > 5 GeV and |eta| < 5 and the leading one's pT and eta.
template <int GW, typename R, int N>
__device__ __forceinline__ void antikt(const ObsTeam<GW>& T, ObsEvent<R, N>& W, int m0, R Rj, int& njets, R& lead,
                                       R& lead_eta) {
  const int lane = T.lane;
  int m = 0;
  uint32_t word = 0;
  for (int b = 0; b < N; b += GW) {
    const int i = b + lane;
    const bool keep = i < m0 && W.ps[i][1] * W.ps[i][1] + W.ps[i][2] * W.ps[i][2] > R(0);
    const uint32_t bits = T.ballot(keep);
    m += __popc(bits);
    if (keep) jet_kin(W.ps[i], W.ipt2[i], W.y[i], W.phi[i]);
    word |= bits << (b & 31);
    if (((b + GW) & 31) == 0) {
      if (lane == 0) W.am[b >> 5] = word;
      word = 0;
    }
  }
  const R R2 = Rj * Rj;
  __syncwarp();
  auto left = [&](int i) { return ((W.am[i >> 5] >> (i & 31)) & 1u) != 0; };
  for (int i = lane; i < m0; i += GW)
    if (left(i)) akt_nn(W, i, R2);
  __syncwarp();
  njets = 0;
  lead = 0;
  lead_eta = 0;
  while (__any_sync(kFull, m > 0)) {
    R dmin = R(INFINITY);
    int key = INT_MAX;  // 2 i for the beam distance of i, 2 i + 1 for its neighbour
    for (int i = m > 0 ? lane : m0; i < m0; i += GW) {
      if (!left(i)) continue;
      const R diB = W.ipt2[i];
      if (diB < dmin) { dmin = diB; key = 2 * i; }
      if (W.nnd[i] < dmin) { dmin = W.nnd[i]; key = 2 * i + 1; }
    }
    team_argmin(T, dmin, key);
    if (key == INT_MAX) m = 0;  // no finite distance (cannot happen for pT > 0)
    const bool on = m > 0;
    const int bi = on ? key >> 1 : 0;
    const int bj = on && (key & 1) ? W.nnj[bi] : -1;
    const int gone = bj < 0 ? bi : bj;
    if (on && bj < 0) {
      R jpt = sqrt(W.ps[bi][1] * W.ps[bi][1] + W.ps[bi][2] * W.ps[bi][2]);
      if (jpt > R(5)) {
        R jeta = asinh(jet_pz(W.ps[bi]) / jpt);
        if (fabs(jeta) < R(5)) {
          njets += 1;
          if (jpt > lead) { lead = jpt; lead_eta = jeta; }
        }
      }
    }
    if (bj >= 0 && lane < 4) W.ps[bi][lane] += W.ps[bj][lane];
    __syncwarp();
    if (on && lane == 0) {
      if (bj >= 0) jet_kin(W.ps[bi], W.ipt2[bi], W.y[bi], W.phi[bi]);
      W.am[gone >> 5] &= ~(1u << (gone & 31));
    }
    m -= 1;
    __syncwarp();
    // refresh the neighbours that pointed at a changed or removed pseudo-jet:
    // few, so the team scans each one's candidates together
    for (int w = 0; w < ObsEvent<R, N>::kWords; ++w) {
      uint32_t st = 0;
      for (int b = 32 * w; b < 32 * w + 32 && __any_sync(kFull, on && b < m0); b += GW) {
        const int i = b + lane;
        bool stale = false;
        if (on && i < m0 && left(i)) {
          const int nj = W.nnj[i];
          stale = (bj >= 0 && (i == bi || nj == bi)) || nj == gone;
          if (bj >= 0 && i < bi && !stale) {
            // a merged pseudo-jet may become i's nearest neighbour, or displace one
            R d = akt_dij(W.ipt2, W.y, W.phi, i, bi, R2);
            if (d < W.nnd[i] || (d == W.nnd[i] && bi < nj)) { W.nnd[i] = d; W.nnj[i] = bi; }
          }
        }
        st |= T.ballot(stale) << (b & 31);
      }
      while (__any_sync(kFull, st != 0)) {
        const int i = st ? 32 * w + __ffs(st) - 1 : m0;
        st &= st - 1;
        R best = R(INFINITY);
        int near = INT_MAX;
        for (int j = i + 1 + lane; j < m0; j += GW) {
          if (!left(j)) continue;
          const R d = akt_dij(W.ipt2, W.y, W.phi, i, j, R2);
          if (d < best) { best = d; near = j; }
        }
        team_argmin(T, best, near);
        if (lane == 0 && i < m0) { W.nnd[i] = best; W.nnj[i] = near == INT_MAX ? -1 : near; }
      }
    }
    __syncwarp();
  }
}

// the coloured final state of event e (the first N of it; np = 0: none) into W:
// its number
template <int GW, typename R, int N>
__device__ __forceinline__ int load_event(const ObsTeam<GW>& T, const DevEvents& E, uint64_t e, int np, bool pp,
                                          ObsEvent<R, N>& W) {
  int m = 0;
  for (int base = pp ? 2 : 0; __any_sync(kFull, base < np && m < N); base += GW) {
    const int i = base + T.lane;
    int fl = 0;
    const bool have = i < np && m < N;
    if (have) fl = E.F(i, e);
    const bool coloured = have && !(fl == 23 || fl == 11 || fl == -11);
    const uint32_t cm = T.ballot(coloured);
    const int at = m + __popc(cm & ((1u << T.lane) - 1u));
    if (coloured && at < N) {
      R* q = W.ps[at];
      if (sizeof(R) == 4 && pp) {
        const double en = E.P(0, i, e), pz = E.P(3, i, e);
        q[0] = (R)(en + pz);
        q[1] = (R)E.P(1, i, e);
        q[2] = (R)E.P(2, i, e);
        q[3] = (R)(en - pz);
      } else {
        for (int mu = 0; mu < 4; ++mu) q[mu] = (R)E.P(mu, i, e);
      }
    }
    m = min(m + __popc(cm), N);
  }
  __syncwarp();
  return m;
}

// an event's clusterings: the Durham scales, or the jets
template <int GW, typename R, int N>
__device__ __forceinline__ void cluster(const ObsTeam<GW>& T, ObsEvent<R, N>& W, int m, bool pp, R& a, R& b, R& c,
                                        int& jets) {
  if (__any_sync(kFull, !pp && m > 0)) {
    R y23, y34;
    durham(T, W, pp ? 0 : m, y23, y34);
    if (!pp) { b = y23; c = y34; }
  }
  if (__any_sync(kFull, pp && m > 0)) {
    R lead, eta;
    int n;
    antikt(T, W, pp ? m : 0, R(0.4), n, lead, eta);
    if (pp) { a = lead; b = eta; jets = n; }
  }
}

__device__ __forceinline__ int bin_of(const HistDef& H, int h, double v) {
  if (H.logx[h]) {
    if (!(v > 0.0)) return 0;
    v = log10(v);
  }
  if (!(v >= H.lo[h])) return 0;
  double f = (v - H.lo[h]) / (H.hi[h] - H.lo[h]);
  int b = (int)floor(f * H.nb[h]);
  if (b >= H.nb[h]) return H.nb[h] + 1;
  return b + 1;
}

// R = double for per-event parity (GAPS_FP64), float for mixed-precision
// contexts. A block takes chunks of up to 256 consecutive events: its threads
// scan their own events' records for the colourless final state (thread =
// event); its warps cluster the events (lane = pseudo-jet), largest first and
// events of like size and kind together, taking the next ones when they are
// done; its threads form, write and histogram their events' observables
// (thread = event), so the per-event FP64 work (boson kinematics, binning) runs
// once per event.
template <typename R>
__global__ void __launch_bounds__(kObsThreads, sizeof(R) == 4 ? 4 : 2)
    k_observables(DevParams P, DevEvents E, uint64_t first, uint64_t n, int chunk, double* obs, HistSet Hs,
                  double* sumw, double* sumw2) {
  // shared: the warps' events, then per row of the batch sumw and sumw2
  // [GAPS_NHIST][GAPS_HIST_BINS]
  extern __shared__ __align__(16) unsigned char obs_smem[];
  ObsWarp<R>* Wa = reinterpret_cast<ObsWarp<R>*>(obs_smem);
  double* sh = reinterpret_cast<double*>(Wa + kObsWarps);
  __shared__ HistDef sH[kMaxRows];
  __shared__ int s_pp[kMaxRows];
  // the chunk: clustering results, kinds and sizes, events in the order the
  // warps take them, and the next one to be taken
  __shared__ R s_a[kObsThreads], s_b[kObsThreads], s_c[kObsThreads];
  __shared__ int s_jets[kObsThreads];
  __shared__ unsigned char s_np[kObsThreads], s_kind[kObsThreads], s_order[kObsThreads];
  __shared__ int s_bin[kObsSizes], s_alone, s_next;
  static_assert(kMaxFinal <= 255 && kObsThreads <= 256, "bytes");
  constexpr int kSet = GAPS_NHIST * GAPS_HIST_BINS;
  const bool fill = sumw != nullptr;
  if (threadIdx.x < P.n_rows) {
    sH[threadIdx.x] = Hs.h[threadIdx.x];
    s_pp[threadIdx.x] = P.rows[threadIdx.x].process != GAPS_EE_QQ;
  }
  if (fill)
    for (int q = threadIdx.x; q < 2 * kSet * P.n_rows; q += blockDim.x) sh[q] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, me = threadIdx.x;
  ObsWarp<R>& W = Wa[threadIdx.x >> 5];
  for (uint64_t g0 = (uint64_t)blockIdx.x * chunk; g0 < n; g0 += (uint64_t)gridDim.x * chunk) {
    // --- thread = event: the colourless final state (Z, or e- e+) and the
    // number of coloured partons, in a plain scan of the record that stops
    // at the kMaxFinal-th coloured parton
    const int ng = n - g0 < (uint64_t)chunk ? (int)(n - g0) : chunk;
    const uint64_t el = g0 + me;
    const bool live = me < ng;
    int row = 0, np = 0, mc = 0;
    bool pp = false;
    double z0 = 0.0, z1 = 0.0, z2 = 0.0, z3 = 0.0;
    if (me < kObsSizes) s_bin[me] = 0;
    if (live) {
      row = mix_row(P, first + el);
      pp = s_pp[row] != 0;
      np = E.npart[el];
      for (int i = pp ? 2 : 0; i < np && mc < kMaxFinal; ++i) {
        const int fl = E.F(i, el);
        if (fl == 23 || fl == 11 || fl == -11) {
          z0 += E.P(0, i, el); z1 += E.P(1, i, el); z2 += E.P(2, i, el); z3 += E.P(3, i, el);
        } else {
          ++mc;
        }
      }
      s_np[me] = (unsigned char)min(max(np, 0), 255);
      s_kind[me] = pp;
    }
    // their order: the events too large for a quarter of a warp (all, if every
    // warp has one at most), then each kind's by size
    const bool alone = mc > kObsSmall || chunk <= kObsWarps;
    const int size = alone ? 0 : (pp ? 1 : kObsSmall + 2) + kObsSmall - mc;
    __syncthreads();
    if (live) atomicAdd(&s_bin[size], 1);
    __syncthreads();
    if (threadIdx.x < 32) {
      int at = 0;
      for (int q0 = 0; q0 < kObsSizes; q0 += 32) {
        const int c = q0 + lane < kObsSizes ? s_bin[q0 + lane] : 0;
        int to = c;
#pragma unroll
        for (int off = 1; off < 32; off *= 2) {
          const int v = __shfl_up_sync(kFull, to, off);
          if (lane >= off) to += v;
        }
        if (q0 + lane < kObsSizes) s_bin[q0 + lane] = at + to - c;
        if (q0 == 0 && lane == 0) s_alone = c;
        at += __shfl_sync(kFull, to, 31);
      }
      if (lane == 0) s_next = 0;
    }
    __syncthreads();
    if (live) s_order[atomicAdd(&s_bin[size], 1)] = (unsigned char)me;
    __syncthreads();
    // --- lane = pseudo-jet: the clusterings
    const int n_alone = s_alone, takes = n_alone + (ng - n_alone + kObsGroups - 1) / kObsGroups;
    for (;;) {
      int take = 0;
      if (lane == 0) take = atomicAdd(&s_next, 1);
      take = __shfl_sync(kFull, take, 0);
      if (take >= takes) break;
      if (take < n_alone) {
        const ObsTeam<32> T(lane);
        const int k = s_order[take];
        const bool ppk = s_kind[k] != 0;
        const int m = load_event(T, E, g0 + k, s_np[k], ppk, W.one);
        R a = 0, b = 0, c = 0;
        int jets = 0;
        if (!ppk) {
          for (int i = lane; i < m; i += 32) keep_norm(W.one, i);
          __syncwarp();
          a = thrust(T, W.one, m);
        }
        cluster(T, W.one, m, ppk, a, b, c, jets);
        if (lane == 0) { s_a[k] = a; s_b[k] = b; s_c[k] = c; s_jets[k] = jets; }
      } else {
        const ObsTeam<kObsLanes> T(lane);
        const int at = n_alone + kObsGroups * (take - n_alone) + lane / kObsLanes;
        const bool mine = at < ng;
        const int k = mine ? s_order[at] : 0;
        const bool ppk = s_kind[k] != 0;
        ObsEvent<R, kObsSmall>& V = W.four[lane / kObsLanes];
        const int m = load_event(T, E, g0 + k, mine ? s_np[k] : 0, ppk, V);
        R a = ppk ? 0 : 1, b = 0, c = 0;  // (thrust 1: no momenta)
        int jets = 0;
        const int mt = ppk ? 0 : m;
        if (__any_sync(kFull, mt > 0)) {
          for (int i = T.lane; i < mt; i += kObsLanes) keep_norm(V, i);
          __syncwarp();
          // thrust: of small events together; its candidates grow fast with the
          // size, so that the whole warp takes larger ones in turn (up to four
          // subsets a lane against one a lane of each event in turn)
          if (__all_sync(kFull, mt <= 6)) {
            const R t = thrust(T, V, mt);
            if (!ppk) a = t;
          } else {
            for (int g = 0; g < kObsGroups; ++g) {
              const int mg = __shfl_sync(kFull, mt, g * kObsLanes);
              if (mg == 0) continue;
              const R tg = thrust(ObsTeam<32>(lane), W.four[g], mg);
              if (lane / kObsLanes == g) a = tg;
            }
          }
        }
        __syncwarp();
        cluster(T, V, m, ppk, a, b, c, jets);
        if (mine && T.lane == 0) { s_a[k] = a; s_b[k] = b; s_c[k] = c; s_jets[k] = jets; }
      }
      __syncwarp();
    }
    __syncthreads();
    if (!live) continue;
    const R ra = s_a[me], rb = s_b[me], rc = s_c[me];
    const int rn = s_jets[me];
    // --- thread = event: observables, their output and the histograms (the
    // observables stay in named registers: an array picked by H.obs[h] would
    // be placed in local memory)
    const double nem = (double)E.n_emit[el];
    double o0, o1, o2, o3, o4, o5 = 0.0, o6 = 0.0, o7 = 0.0;
    if (!pp) {
      o0 = 1.0 - (double)ra;
      o1 = rb;
      o2 = rc;
      o3 = (double)mc;
      o4 = nem;
    } else {
      double pt = sqrt(z1 * z1 + z2 * z2);
      o0 = pt;
      o1 = 0.5 * log((z0 + z3) / (z0 - z3));
      o2 = pt > 0.0 ? atan2(z2, z1) : 0.0;
      o3 = (double)rn;
      o4 = ra;
      o5 = rb;
      o6 = (double)mc;
      o7 = nem;
    }
    if (obs) {
      double* out = obs + el;
      const uint64_t c = E.cap;
      out[0] = o0; out[c] = o1; out[2 * c] = o2; out[3 * c] = o3;
      out[4 * c] = o4; out[5 * c] = o5; out[6 * c] = o6; out[7 * c] = o7;
    }
    if (fill && E.status[el] == GAPS_STATUS_DONE) {
      const HistDef& H = sH[row];
      double* hw = sh + 2 * kSet * row;
      double* hw2 = hw + kSet;
      const double w = E.weight[el];
#pragma unroll
      for (int h = 0; h < GAPS_NHIST; ++h) {
        const int oi = H.obs[h];
        const double v = oi == 0 ? o0 : oi == 1 ? o1 : oi == 2 ? o2 : oi == 3 ? o3
                       : oi == 4 ? o4 : oi == 5 ? o5 : oi == 6 ? o6 : o7;
        const int bin = bin_of(H, h, v);
        atomicAdd(&hw[h * GAPS_HIST_BINS + bin], w);
        atomicAdd(&hw2[h * GAPS_HIST_BINS + bin], w * w);
      }
    }
  }
  if (fill) {
    __syncthreads();
    for (int q = threadIdx.x; q < kSet * P.n_rows; q += blockDim.x) {
      const int r = q / kSet, k = q % kSet;
      const double a = sh[2 * kSet * r + k], b = sh[2 * kSet * r + kSet + k];
      if (a != 0.0) atomicAdd(&sumw[q], a);
      if (b != 0.0) atomicAdd(&sumw2[q], b);
    }
  }
}

template <typename R>
size_t observables_smem(int n_rows, bool fill) {
  return kObsWarps * sizeof(ObsWarp<R>) +
         (fill ? 2 * (size_t)n_rows * GAPS_NHIST * GAPS_HIST_BINS * sizeof(double) : 0);
}

}  // namespace

// Opt-in for the observables kernels' dynamic shared memory (the warps'
// events and a mixed batch's histograms); called when a context is created.
cudaError_t observables_init() {
  cudaError_t e = cudaFuncSetAttribute(k_observables<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)observables_smem<float>(kMaxRows, true));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_observables<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)observables_smem<double>(kMaxRows, true));
  return e;
}

cudaError_t launch_observables(const DevParams& P, const DevEvents& E, uint64_t first, uint64_t n, double* obs,
                               const HistSet& H, double* sumw, double* sumw2, int fp32, int sm_count,
                               cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  const uint64_t resident = (uint64_t)max(1, sm_count) * (fp32 ? 4 : 2);
  // events of a chunk: a thread each where there are enough, else as few as
  // give every resident block some
  const int chunk = (int)min((uint64_t)kObsThreads, (n + resident - 1) / resident);
  const unsigned grid = (unsigned)min((n + chunk - 1) / chunk, resident);
  const bool fill = sumw != nullptr;
  if (fp32)
    k_observables<float><<<grid, kObsThreads, observables_smem<float>(P.n_rows, fill), stream>>>(
        P, E, first, n, chunk, obs, H, sumw, sumw2);
  else
    k_observables<double><<<grid, kObsThreads, observables_smem<double>(P.n_rows, fill), stream>>>(
        P, E, first, n, chunk, obs, H, sumw, sumw2);
  return cudaGetLastError();
}

}  // namespace gaps
