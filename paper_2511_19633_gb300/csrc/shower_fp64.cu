// FP64 max-veto dipole shower (Section 2, Fig. 1; Appendices A and B of
// arXiv:2511.19633). Compiled without FMA contraction (-fmad=false): every
// event reproduces a plain FP64 evaluation of the same formulas bit for bit.
//
// The algorithm of Fig. 1 draws one trial per channel of every colour end in
// each cycle, takes the largest, and vetoes about fifteen of sixteen winners.
// Three properties let a group of kG lanes run kG cycles of one event at once
// with the same results:
//   - While the event does not change, a cycle uses a fixed number of Philox
//     blocks, so the blocks of the cycles ahead are known.
//   - Which channel wins needs its trial scale only to the accuracy that
//     separates it from the next one. FP32 values with an error bound decide
//     that (screening); a cycle in which the bounds of two channels overlap,
//     or in which a bound straddles a threshold, is decided in FP64.
//   - A winner's exact scale is min(t, t_kin) R^(1/c), with t the exact scale
//     of the cycle before: the powers of the kG cycles are formed side by
//     side, the products one after the other.
// The lanes then evaluate one cycle's acceptance each, assuming that the
// cycles before were vetoed; the first that was not ends the batch and the
// cycles behind it are dropped, their counters with them.
//
// What bounds it: FP64 runs at 1/64 of the FP32 rate here, and an FP64
// instruction costs a warp the same however few lanes are active. One thread
// per event (the earlier form of this file) evaluated every trial in FP64 with
// a partner search and the bound tables again in each cycle; now the end table
// is kept between emissions (only the ends an emission touched are formed
// again), the trials run in FP32 and the FP64 work fills the lanes. The warps
// are in different phases, so the next limit was the instruction cache: with
// every logarithm, division and density inlined the kernel was 376 KB, its
// fetches hit in 48 % and 36 of 55 stall cycles had no instruction; with one
// copy of each it is 154 KB and half the time. An FP64 instruction in the
// screening loop, even a comparison, waits behind the other warps' FP64 work.
// Whole path (hard events, shower, observables), one thread per event and now:
// 30 000 LO pp -> Z events at 13.6 TeV 1138 and 24 ms, 3001 NLO events with
// heavy-quark thresholds 1093 and 16 ms (the longest event's chain of cycles),
// 10 000 e+e- events at 91.2 GeV 34.0 and 1.5 ms, 500 of them 21 and 0.64 ms.
#define GAPS_GM_OUT_OF_LINE
#include "physics_fp64.cuh"

namespace gaps {
namespace {

// One copy of a Philox block outside the screening loop (see
// GAPS_GM_OUT_OF_LINE)
__device__ __noinline__ uint4 block_of(uint64_t event, uint64_t draw, uint32_t k0, uint32_t k1) {
  uint32_t o[4];
  philox((uint32_t)event, (uint32_t)(event >> 32), (uint32_t)draw, (uint32_t)(draw >> 32), k0, k1, o);
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// lanes per event: eight cycles a batch (an acceptance comes every 9 to 16
// cycles), and the about eight ends that an emission touches in one step
constexpr int kG = 8;
// cycles of a batch when a warp has one event left and gives it all its lanes
// (shower of 3001 NLO events with heavy-quark thresholds: 15.6 ms with 8 lanes to
// the end, 13.8 ms with 32; 8, 16 or 32 cycles a batch, 14.3, 13.8 and 13.1 ms, are
// within the spread of single launches, 11 to 19 ms)
constexpr int kWideBatch = 16;
constexpr int kThreads = 128;
constexpr int kGroups = kThreads / kG;  // events a block holds
// 128 registers a thread (5, 6 and 8 blocks, with more spills, were level to
// 10 % slower; so were blocks of 256 and 512 threads that begin a batch together)
constexpr int kMinBlocks = 4;
constexpr int kMaxPerBlock = 128;       // events a block takes before it leaves
constexpr unsigned kAll = 0xffffffffu;

struct Counters {
  unsigned long long finished = 0, steps = 0, trials = 0, isr_trials = 0, vetoes = 0, accepts = 0, violations = 0;
  unsigned long long err_cap = 0, err_iter = 0, err_num = 0;
};

// exact record of a colour end (emitter slot q / 2, side q % 2) in the group's
// scratch: the inputs of its two channels' trials and weights
struct EndX {
  double s, eta, tkin, cc[2], B[2];
  int k, type;  // partner slot (-1: no dipole on this side), dipole type
};
static_assert(sizeof(EndX) == 64, "one end is two sectors");

// a parton's flavour and colour tags
struct Tag { int f, c, a, pad; };

// One event's scratch. `scr` holds the screening values of an end: {1/c of
// channel 0, 1/c of channel 1 (-1: absent, infinity: no trial), ln t_kin,
// number of trial blocks before this end}.
struct Scratch {
  double* p;     // [nmax][4]
  EndX* end;     // [2 nmax]
  float4* scr;   // [2 nmax]
  Tag* tag;      // [nmax]
};
constexpr size_t kSlotBytesPerParton = 4 * sizeof(double) + 2 * sizeof(EndX) + 2 * sizeof(float4) + sizeof(Tag);

__device__ __forceinline__ Scratch scratch_of(unsigned char* base, int nmax) {
  Scratch w;
  w.p = reinterpret_cast<double*>(base);
  w.end = reinterpret_cast<EndX*>(base + (size_t)nmax * 4 * sizeof(double));
  w.scr = reinterpret_cast<float4*>(w.end + 2 * nmax);
  w.tag = reinterpret_cast<Tag*>(w.scr + 2 * nmax);
  return w;
}

// per row of a mixed batch
struct RowShared {
  double t_cut, as_over, as_2pi;  // as_2pi: as_over / 2 pi
  float lnTc;
  int pp;
};

// A group of G consecutive lanes of a warp (G = kG or 32, one copy of the code
// for both): values of lane `src` of the caller's group and reductions over it
// (all 32 lanes of the warp call them).
struct Group {
  int G;
  __device__ __forceinline__ int lane() const { return threadIdx.x & (G - 1); }
  template <class T>
  __device__ __forceinline__ T get(T v, int src) const { return __shfl_sync(kAll, v, src, G); }
  template <class T>
  __device__ __forceinline__ T xchg(T v, int o) const { return __shfl_xor_sync(kAll, v, o); }
  __device__ __forceinline__ float max(float v) const {
#pragma unroll 1
    for (int o = G >> 1; o > 0; o >>= 1) v = fmaxf(v, xchg(v, o));
    return v;
  }
  __device__ __forceinline__ int sum(int v) const {
#pragma unroll 1
    for (int o = G >> 1; o > 0; o >>= 1) v += xchg(v, o);
    return v;
  }
  // bit j: `b` of lane j of the group
  __device__ __forceinline__ unsigned ballot(bool b) const {
    return (__ballot_sync(kAll, b) >> (threadIdx.x & 31 & ~(G - 1))) & (kAll >> (32 - G));
  }
};

// squared mass of the heavy-quark measure of an end's channels (App. A.2: an
// incoming c or b with a threshold draws both its channels in dt/(t - m^2))
__device__ __forceinline__ double heavy_m2(const DevParams& P, int type, int fl) {
  if (type != kIF && type != kII) return 0.0;
  if (fl == 21) return 0.0;
  const int fe = pdf_index(fl);
  return fe >= 0 && P.thr[fe] >= 0 ? P.m2[fe] : 0.0;
}

// channel c of an emitter: 0 q->qg, 1 g->gg, 2 g->qqbar (final); 3 q->qg,
// 4 q->g qbar, 5 g->gg, 6 g->qq (initial)
__device__ __forceinline__ int channel_of(bool ini, int fl, int c) {
  return (ini ? (fl == 21 ? 5 : 3) : (fl == 21 ? 1 : 0)) + c;
}

// The record of end q (one lane): partner, invariant, overestimate
// coefficients and PDF-ratio bounds of its channels.
__device__ __forceinline__ void form_end(const DevParams& P, const Scratch& w, const RowShared& R, int n, int q,
                                      double eta0, double eta1) {
  const int i = q >> 1, side = q & 1;
  const Tag ti = w.tag[i];
  const int tag = side == 0 ? ti.c : ti.a;
  int k = -1;
  if (tag != 0)
    for (int m = 0; m < n; ++m) {
      if (m == i) continue;
      if (side == 0 ? (w.tag[m].a == tag) : (w.tag[m].c == tag)) { k = m; break; }
    }
  EndX x;
  x.k = k;
  x.type = 0;
  float4 sc = make_float4(-1.0f, -1.0f, 0.0f, 0.0f);
  if (k >= 0) {
    const int fi = ti.f;
    const bool ini = R.pp && i < 2, ink = R.pp && k < 2;
    const int type = ini ? (ink ? kII : kIF) : (ink ? kFI : kFF);
    double pi[4], pk[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) { pi[mu] = w.p[4 * i + mu]; pk[mu] = w.p[4 * k + mu]; }
    const double s = 2.0 * dot4(pi, pk);
    double eta = 0.0;
    if (type == kFI) eta = (k == 0) ? eta0 : eta1;
    if (type == kIF || type == kII) eta = (i == 0) ? eta0 : eta1;
    const int nch = (!ini && fi != 21) ? 1 : 2;
    x.type = type;
    x.s = s;
    x.eta = eta;
    x.tkin = t_kin_max(type, s, eta);
    double zm, delta;
    // (every trial starts above the cutoff, so min(t, t_kin) > t_c here is t_kin > t_c)
    const bool ok = !(x.tkin <= R.t_cut) && z_limits(type, R.t_cut, s, eta, zm, delta);
    x.cc[0] = x.cc[1] = 0.0;
    x.B[0] = x.B[1] = 1.0;
    float ic[2] = {-1.0f, -1.0f};
    // the two logarithms of the shapes' integrals, shared by the channels
    double lsoft = 0.0, linv = 0.0;
    if (ok) {
      const double zp = 1.0 - delta;
      int sh0, sh1;
      double unused;
      channel_over(channel_of(ini, fi, 0), type, P.nf, sh0, unused);
      channel_over(channel_of(ini, fi, 1), type, P.nf, sh1, unused);
      if (nch == 1) sh1 = sh0;
      if (sh0 == kSoft || sh0 == kBoth || sh1 == kSoft || sh1 == kBoth) lsoft = gm_log(gm_div(1.0 - zm, delta));
      if (sh0 == kInv || sh0 == kBoth || sh1 == kInv || sh1 == kBoth) linv = gm_log(gm_div(zp, zm));
      // the grid cell of eta, for every channel's bound
      int ix = 0;
      double fx = 0.0;
      const bool on_grid = type != kFF && pdf_locate_x(P, eta, ix, fx);
#pragma unroll 1
      for (int c = 0; c < nch; ++c) {
        const int ch = channel_of(ini, fi, c);
        int shape;
        double coef;
        channel_over(ch, type, P.nf, shape, coef);
        double B = 1.0;
        if (type == kFI) {
          // both channels of a final emitter have the spectator's bound
          if (c == 0) {
            const int f = pdf_index(w.tag[k].f);
            B = on_grid ? pdf_ratio_bound_at(P, f, f, ix, fx) : 0.0;
          } else {
            B = x.B[0];
          }
        } else if (type == kIF || type == kII) {
          int num, den;
          isr_pdf_indices(ch, fi, num, den);
          B = on_grid ? pdf_ratio_bound_at(P, num, den, ix, fx) : 0.0;
        }
        x.B[c] = B;
        if (!(B > 0.0)) continue;
        const double in = shape == kSoft ? lsoft : shape == kFlat ? zp - zm : shape == kBoth ? linv + lsoft : linv;
        const double cc = R.as_2pi * B * coef * in;
        if (cc > 0.0) x.cc[c] = cc;
      }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
      if (c < nch) ic[c] = x.cc[c] > 0.0 ? fminf(1.0f / (float)x.cc[c], 1e30f) : INFINITY;
    sc = make_float4(ic[0], ic[1], __logf((float)x.tkin), 0.0f);
  }
  w.end[q] = x;
  w.scr[q] = sc;
}

// pdf_at of one flavour (0..10; 0 for any other), one copy
__device__ __noinline__ double xf_at(const DevParams& P, int f, const PdfLoc& L) {
  if (f < 0 || f > 10 || !L.ok) return 0.0;
  const float* g = P.grid + ((size_t)f * kNX + L.ix) * kNQ + L.iq;
  const double lo = (1.0 - L.fx) * (double)__ldg(g) + L.fx * (double)__ldg(g + kNQ);
  const double hi = (1.0 - L.fx) * (double)__ldg(g + 1) + L.fx * (double)__ldg(g + kNQ + 1);
  return lo * (1.0 - L.fq) + hi * L.fq;
}

// exact trial scale of channel c of end x below t with the uniform Rt (-1: no
// trial, counted false); the order of Fig. 1's tests
__device__ __noinline__ double exact_trial(const EndX& x, int c, double m2, double t, double t_cut, double Rt, bool& counted) {
  counted = false;
  const double tmax = fmin(t, x.tkin);
  if (!(tmax > t_cut)) return -1.0;
  if (m2 > 0.0 && !(tmax > m2 * (1.0 + kHqFloor))) return -1.0;
  if (!(x.cc[c] > 0.0)) return -1.0;
  counted = true;
  if (m2 > 0.0) {
    const double tt = m2 + (tmax - m2) * gm_exp(gm_div(gm_log(Rt), x.cc[c]));
    return tt > m2 * (1.0 + kHqFloor) ? tt : -1.0;
  }
  return tmax * gm_exp(gm_div(gm_log(Rt), x.cc[c]));
}

// outcome of one cycle
enum Outcome { kVeto = 0, kAccept, kDone, kNumericT, kNumericW, kCapacity };

struct Winner {
  int outcome, type, ch, bi, bk, side, new_fl, fl_j;
  bool violation;
  double t, z, omz, a0, a1, a2, a3, Rphi;  // a0..a3: the map's variables (see emission)
};

// The cycle after its trials for the winner (q, c) at scale tw: Appendix B's
// weight and the accept test. One lane, on its own cycle. Values that every
// dipole type needs (the z sample, alpha_s, the two densities) are formed
// outside the branches on the type, so that the lanes of a warp share them.
__device__ __forceinline__ void weigh(const DevParams& P, const Scratch& w, const RowShared& R, int n, int q, int c,
                                   double tw, double Rz, const uint4& o1, const uint4& o2, Winner& W) {
  W.violation = false;
  W.t = tw;
  if (tw < R.t_cut) { W.outcome = kDone; return; }
  if (!isfinite(tw)) { W.outcome = kNumericT; return; }
  const EndX x = w.end[q];
  const int bi = q >> 1, bk = x.k, type = x.type;
  const int fl_i = w.tag[bi].f;
  const bool ini = type == kIF || type == kII;
  const int ch = channel_of(ini, fl_i, c);
  const double s = x.s, eta = x.eta;
  W.bi = bi; W.bk = bk; W.side = q & 1; W.type = type; W.ch = ch;
  W.new_fl = fl_i; W.fl_j = 21;
  W.outcome = kVeto;
  int shape;
  double coef, zm, delta, z, omz;
  channel_over(ch, type, P.nf, shape, coef);
  z_limits(type, R.t_cut, s, eta, zm, delta);
  shape_sample(shape, zm, delta, Rz, z, omz);
  double zm_t, delta_t;
  if (!z_limits(type, tw, s, eta, zm_t, delta_t) || !(omz > delta_t) || !(z > zm_t)) return;
  const double pover = shape_value(shape, coef, z, omz);
  W.z = z;
  W.omz = omz;
  double xm = 1.0, omx = 0.0, u = 0.0, omu = 1.0, v = 0.0, rho = 0.0, y = 0.0, J = 1.0, den = 1.0, kk;
  double x1 = 0.0;  // the numerator density's momentum fraction
  if (!ini) {
    rho = y = gm_div(tw, z * omz * s);
    double soft = z * y;
    if (type == kFI) {
      xm = gm_div(1.0, 1.0 + rho);
      omx = gm_div(rho, 1.0 + rho);
      soft = omx;
      x1 = eta * (1.0 + rho);
    }
    den = omz + soft;
  } else {
    const double r = gm_div(tw, s);
    if (type == kIF) {
      if (!if_map(r, z, omz, xm, omx, u, omu)) return;
      J = gm_div(1.0, xm * omu + u * omx);
    } else {
      if (!ii_map(r, z, omz, xm, omx, v)) return;
      J = gm_div(1.0, z);
    }
    if (!(xm > eta)) return;
    x1 = gm_div(eta, xm);
    den = (type == kIF) ? (omx + u) : omx;
  }
  // the kernels' soft poles, one division for all channels
  const double pole = gm_div(ch == 5 ? 1.0 : 2.0, den);
  if (ch == 0) kk = kCF * (pole - (1.0 + z));
  else if (ch == 1) kk = kCA / 2.0 * (pole - 2.0 + z * omz);
  else if (ch == 2) kk = P.nf * kTR / 2.0 * (1.0 - 2.0 * z * omz);
  else if (ch == 3) kk = kCF * (pole - (1.0 + xm));
  else if (ch == 4) kk = kTR * (1.0 - 2.0 * xm * omx);
  else if (ch == 5) kk = kCA * (pole + gm_div(omx, xm) - 1.0 + xm * omx);
  else kk = kCF / 2.0 * (xm + gm_div(2.0 * omx, xm));
  const double as_ratio = gm_div(alpha_s(P, tw), R.as_over);
  double wgt, sumF = 0.0;
  PdfLoc l1;
  l1.ok = false;
  if (type == kFF) {
    wgt = gm_div(as_ratio * (1.0 - y) * kk, pover);
  } else {
    // the two points' cells: one Q^2 location for both
    PdfLoc l0;
    l0.ix = l0.iq = 0;
    l0.fx = l0.fq = 0.0;
    l1 = l0;
    const bool okq = pdf_locate_q(P, tw, l0.iq, l0.fq);
    l1.iq = l0.iq;
    l1.fq = l0.fq;
    l0.ok = pdf_locate_x(P, eta, l0.ix, l0.fx) && okq;
    l1.ok = pdf_locate_x(P, x1, l1.ix, l1.fx) && okq;
    int num, den;
    if (type == kFI) num = den = pdf_index(w.tag[bk].f);
    else isr_pdf_indices(ch, fl_i, num, den);
    const double F0 = xf_at(P, den, l0);
    double F1;
    if (ch == 6) {
      F1 = 0.0;
#pragma unroll 1
      for (int f = 1; f <= 10; ++f) F1 += xf_at(P, f, l1);
      sumF = F1;
    } else {
      F1 = xf_at(P, num, l1);
    }
    if (type == kFI) {
      const double ratio = (F0 > 0.0) ? gm_div(xm * F1, F0) : 0.0;
      wgt = gm_div(gm_div(as_ratio * kk, pover) * ratio, x.B[c]);
    } else {
      double Fratio = (F0 > 0.0) ? gm_div(F1, F0) : 0.0;
      const double m2 = heavy_m2(P, type, fl_i);
      if (m2 > 0.0) Fratio = Fratio * gm_div(tw - m2, tw);  // heavy-quark measure correction
      wgt = gm_div(gm_div(as_ratio * kk * J * xm, pover) * Fratio, x.B[c]);
      if (ch == 4) { W.new_fl = 21; W.fl_j = -fl_i; }
      if (ch == 5) { W.new_fl = 21; W.fl_j = 21; }
    }
  }
  if (!isfinite(wgt)) { W.outcome = kNumericW; return; }
  W.violation = wgt > 1.0;
  if (!(u01(o1.x, o1.y) < wgt)) return;

  // accepted: flavours
  const double Rfl = u01(o2.x, o2.y);
  if (ch == 2) {
    int f = 1 + (int)floor(Rfl * P.nf);
    if (f > P.nf) f = P.nf;
    W.new_fl = f; W.fl_j = -f;
  } else if (ch == 6) {
    double target = Rfl * sumF, acc = 0.0;
    int pick = 10;
#pragma unroll 1
    for (int f = 1; f <= 10; ++f) {
      acc += xf_at(P, f, l1);
      if (target < acc) { pick = f; break; }
    }
    const int fl = pick <= 5 ? pick : -(pick - 5);
    W.new_fl = fl; W.fl_j = fl;
  }
  W.outcome = n >= P.nmax ? kCapacity : kAccept;
  W.Rphi = u01(o1.z, o1.w);
  if (type == kFF) { W.a0 = y; W.a1 = W.a2 = W.a3 = 0.0; }
  else if (type == kFI) { W.a0 = rho; W.a1 = W.a2 = W.a3 = 0.0; }
  else if (type == kIF) { W.a0 = xm; W.a1 = omx; W.a2 = u; W.a3 = omu; }
  else { W.a0 = xm; W.a1 = omx; W.a2 = v; W.a3 = 0.0; }
}

// Minkowski product of group-distributed four-vectors (lane mu holds component
// mu, lanes 4.. the same again), summed in dot4's order
__device__ __forceinline__ double gdot(const Group& g, double a, double b) {
  const double m = a * b;
  return g.get(m, 0) - g.get(m, 1) - g.get(m, 2) - g.get(m, 3);
}

// The emission of the group's winner W (lane f's copy, broadcast): kinematics with
// one momentum component per lane (lanes 4.. repeat 0..3), the II kick with
// one parton per lane, colours on lane 0. All lanes of the warp take part;
// groups with on = false compute on slot 0 and write nothing.
__device__ __forceinline__ void emission(const Group& g, const Scratch& w, bool on, int n, const Winner& W, int f, double& eta0,
                                      double& eta1) {
  const int gl = g.lane(), mu = gl & 3;
  const int pack = g.get(W.type | (W.ch << 2) | (W.side << 5) | (W.bi << 6) | (W.bk << 14), f);
  const int type = pack & 3, ch = (pack >> 2) & 7, side = (pack >> 5) & 1;
  const int bi = on ? (pack >> 6) & 0xff : 0, bk = on ? (pack >> 14) & 0xff : 0;
  const int new_fl = g.get(W.new_fl, f), fl_j = g.get(W.fl_j, f);
  const double z = g.get(W.z, f), omz = g.get(W.omz, f), tw = g.get(W.t, f), Rphi = g.get(W.Rphi, f);
  const double a0 = g.get(W.a0, f), a1 = g.get(W.a1, f), a2 = g.get(W.a2, f), a3 = g.get(W.a3, f);
  const double Pm = w.p[4 * bi + mu], K = w.p[4 * bk + mu];
  // transverse basis (physics_fp64.cuh's steps)
  const double PK = gdot(g, Pm, K);
  const double N = 1.0 + gm_div(2.0 * Pm * K, PK);
  const double N1 = g.get(N, 1), N2 = g.get(N, 2), N3 = g.get(N, 3);
  int a = 1;
  double Na = N1;
  if (N2 > Na) { a = 2; Na = N2; }
  if (N3 > Na) { a = 3; Na = N3; }
  int b;
  if (a == 1) b = (N3 > N2) ? 3 : 2;
  else if (a == 2) b = (N3 > N1) ? 3 : 1;
  else b = (N2 > N1) ? 2 : 1;
  const double na = gm_sqrt(Na);
  // K_a / PK, P_a / PK, K_b / PK, P_b / PK: one division, on lanes 0..3
  const double Ka = g.get(K, a), Pa = g.get(Pm, a), Kb = g.get(K, b), Pb = g.get(Pm, b);
  const double dv = gm_div(mu == 0 ? Ka : mu == 1 ? Pa : mu == 2 ? Kb : Pb, PK);
  const double KaP = g.get(dv, 0), PaP = g.get(dv, 1), KbP = g.get(dv, 2), PbP = g.get(dv, 3);
  const double e1 = gm_div(((mu == a) ? 1.0 : 0.0) + KaP * Pm + PaP * K, na);
  const double e1b = g.get(e1, b);
  const double rperp = ((mu == b) ? 1.0 : 0.0) + KbP * Pm + PbP * K;
  const double e2p = rperp - e1b * e1;
  const double n2 = gm_sqrt(-gdot(g, e2p, e2p));
  const double e2 = gm_div(e2p, n2);
  const double st = gm_sqrt(tw);
  double cph, sph;
  gm_sincos2pi(Rphi, cph, sph);  // phi = 2 pi R_phi
  const double kt = st * (cph * e1 + sph * e2);
  double pi, pk, pj;
  if (type == kFF) {
    pi = z * Pm + (a0 * omz) * K + kt;
    pj = omz * Pm + (a0 * z) * K - kt;
    pk = (1.0 - a0) * K;
  } else if (type == kFI) {
    const double xinv = 1.0 + a0;
    pi = z * Pm + (omz * a0) * K + kt;
    pj = omz * Pm + (z * a0) * K - kt;
    pk = xinv * K;
    if (on) { if (bk == 0) eta0 = eta0 * xinv; else eta1 = eta1 * xinv; }
  } else {
    pi = gm_div(Pm, a0);
    if (type == kIF) {
      pj = gm_div(a3 * a1, a0) * Pm + a2 * K - kt;
      pk = gm_div(a2 * a1, a0) * Pm + a3 * K + kt;
    } else {
      pj = gm_div(a1 - a2, a0) * Pm + a2 * K - kt;
      pk = K;
    }
    if (on) { const double en = gm_div(bi == 0 ? eta0 : eta1, a0); if (bi == 0) eta0 = en; else eta1 = en; }
  }
  __syncwarp();  // every lane has read its old momenta
  if (on && gl < 4) {
    w.p[4 * bi + mu] = pi;
    if (type != kII) w.p[4 * bk + mu] = pk;
    w.p[4 * n + mu] = pj;
  }
  if (__any_sync(kAll, on && type == kII)) {
    // Lorentz kick of all other final-state particles (eq. IIkinematics3)
    const double kp = Pm + K, kn = (pi + K) - pj, kq = kp + kn;
    double Kp[4], Kn[4], KK[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) { Kp[m] = g.get(kp, m); Kn[m] = g.get(kn, m); KK[m] = g.get(kq, m); }
    if (on && type == kII) {
      const double KK2 = dot4(KK, KK), Kp2 = dot4(Kp, Kp);
      for (int m = 2 + gl; m < n; m += g.G) {
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = w.p[4 * m + j];
        const double ka = gm_div(2.0 * dot4(KK, v), KK2);
        const double kb = gm_div(2.0 * dot4(Kp, v), Kp2);
#pragma unroll
        for (int j = 0; j < 4; ++j) w.p[4 * m + j] = v[j] - ka * KK[j] + kb * Kn[j];
      }
    }
  }
  if (on && gl == 0) {
    // colours: new tag 100 + slot of the new parton
    const int T = 100 + n;
    Tag t = w.tag[bi];
    int ci = t.c, ai = t.a, cj = 0, aj = 0;
    if (ch == 0 || ch == 1 || ch == 3 || ch == 5) {
      if (side == 0) { cj = ci; aj = T; ci = T; }
      else { aj = ai; cj = T; ai = T; }
    } else if (ch == 2) {
      aj = ai; cj = 0; ai = 0;
    } else if (ch == 4) {
      if (ai != 0) { ci = T; aj = T; cj = 0; }
      else { ai = T; cj = T; aj = 0; }
    } else {
      const int A = ci, Bt = ai;
      if (new_fl > 0) { ci = 0; ai = Bt; cj = A; aj = 0; }
      else { ci = A; ai = 0; cj = 0; aj = Bt; }
    }
    w.tag[bi] = Tag{new_fl, ci, ai, 0};
    w.tag[n] = Tag{fl_j, cj, aj, 0};
  }
  __syncwarp();
}

// The warp-wide sum of every counter, one atomic per warp and counter
__device__ __forceinline__ void flush_counters(const DevParams& P, const Counters& c) {
  __syncwarp();
  const unsigned long long v[10] = {c.finished, c.steps, c.trials, c.isr_trials, c.vetoes,
                                    c.accepts, c.violations, c.err_cap, c.err_iter, c.err_num};
  const int idx[10] = {C_EVENTS, C_STEPS, C_TRIALS, C_ISR_TRIALS, C_VETOES,
                       C_ACCEPTS, C_VIOLATIONS, C_ERR_CAP, C_ERR_ITER, C_ERR_NUM};
#pragma unroll
  for (int q = 0; q < 10; ++q) {
    unsigned long long x = v[q];
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(kAll, x, off);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&P.counters[idx[q]], x);
  }
}

// FP32 bounds of a screened trial: v +- er holds ln t of the exact trial. The
// terms: the uniform's rounding and the fast logarithm (2^-21.41 between 1/2
// and 2, 3 ulp elsewhere) times 1/c, whose own rounding and the product's are
// relative to |lr|; the roundings of ln t_max and of the sum; the bound eT of
// ln t itself. Each is taken at least twice.
__device__ __forceinline__ float screen_error(float ic, float lr, float v, float lnTm, float eT) {
  return ic * (1.2e-6f + 1.2e-6f * fabsf(lr)) + (fabsf(v) + fabsf(lnTm)) * 4e-7f + 2e-6f + eT;
}
// slack of a comparison with a logarithm formed in FP32 (|ln| < 64)
constexpr float kLnSlack = 1e-4f;

// An event in flight, the same in every lane of its group
struct Event {
  bool active = false, table = false;  // table: the end table has to be formed
  uint64_t e = 0, id = 0, draw = 0;
  int n = 0, n_emit = 0, steps = 0, row = 0, status = GAPS_STATUS_ACTIVE;
  int nblk = 0;  // trial blocks of a cycle
  int chg = -1;  // emitter | spectator << 8 of the emission since the last table, -1: all ends
  double t = 0.0, eta0 = 0.0, eta1 = 0.0;
};

// One batch of up to K <= g.G cycles of every group's event, with the end table
// before and the emission after it. All lanes of the warp call it.
__device__ __forceinline__ void batch(const Group g, int K, const DevParams& P, const DevEvents& E, const Scratch& w, const RowShared* rows,
                                      const float* m2f, unsigned char* list, Event& S, Counters& cnt, bool heavy_table) {
  const int G = g.G, gl = g.lane();
  const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
  const RowShared& R = rows[S.row];
  const int ne = S.active ? 2 * S.n : 0;
  __syncwarp();

  // ---- end table: the ends the last emission touched (all: chg < 0) ----
  if (__any_sync(kAll, S.table)) {
    // the ends to form, gathered first so that they fill the group's lanes
    const int ci = S.chg & 0xff, ck = (S.chg >> 8) & 0xff, T = 99 + S.n;
    int todo = 0;
    const int scans = __reduce_max_sync(kAll, S.table ? (ne + G - 1) / G : 0);
    for (int r = 0; r < scans; ++r) {
      const int q = r * G + gl;
      bool form = S.table && q < ne;
      if (form && S.chg >= 0 && q < ne - 2) {
        // an end away from the emitter, the spectator and the new parton
        // whose partner is neither of them keeps its record: its inputs did
        // not change; one without a partner or with the new tag is matched
        // again
        const int i = q >> 1, k = w.end[q].k;
        const Tag ti = w.tag[i];
        const int tag = (q & 1) ? ti.a : ti.c;
        form = !(i != ci && i != ck && k != ci && k != ck && (tag == 0 || (k >= 0 && tag != T)));
      }
      const unsigned m = g.ballot(form);
      if (form) list[todo + __popc(m & ((1u << gl) - 1u))] = (unsigned char)q;
      todo += __popc(m);
    }
    __syncwarp();
    for (int j = gl; j < todo; j += G) form_end(P, w, R, S.n, list[j], S.eta0, S.eta1);
    __syncwarp();
    // trial blocks before each end, and of a cycle
    int run = 0;
    for (int r = 0; r < scans; ++r) {
      const int q = r * G + gl;
      int nd = 0;
      float4 sc = make_float4(-1.0f, -1.0f, 0.0f, 0.0f);
      if (S.table && q < ne) {
        sc = w.scr[q];
        nd = (sc.x >= 0.0f ? 1 : 0) + (sc.y >= 0.0f ? 1 : 0);
      }
      int inc = nd;
#pragma unroll 1
      for (int o = 1; o < G; o <<= 1) {
        const int v = __shfl_up_sync(kAll, inc, o, G);
        if (gl >= o) inc += v;
      }
      if (S.table && q < ne) w.scr[q].w = __int_as_float(run + inc - nd);
      run += g.get(inc, G - 1);
    }
    if (S.table) S.nblk = run;
    S.table = false;
    __syncwarp();
  }

  // ---- screening: the winners of up to K cycles ----------------------
  const uint32_t e0 = (uint32_t)S.id, e1 = (uint32_t)(S.id >> 32);
  const float lnTc = R.lnTc;
  float lnT = S.active ? __logf((float)S.t) : 0.0f, eT = 2e-6f + fabsf(lnT) * 4e-7f;
  int len = 0;                  // cycles with a winner
  bool ends_done = false;       // the cycle after them has no trial above the cutoff
  bool going = S.active;        // the batch can take another cycle
  int my_q = 0, my_c = 0;       // winner of cycle gl
  int my_trials = 0;            // trials of cycle gl: all | initial-state << 16
  const bool live_t = S.t > R.t_cut;
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    if (!__any_sync(kAll, going)) break;
    const uint64_t dk = S.draw + (uint64_t)k * (uint64_t)(S.nblk + 2);
    float u1 = -INFINITY, u2 = -INFINITY, lmax = -INFINITY, v1 = 0.0f, er1 = 0.0f;
    int i1 = 0, nt = 0;
    bool doubt = false;
    if (going && live_t) {
#pragma unroll 1
      for (int q = gl; q < ne; q += G) {
        const float4 sc = w.scr[q];
        // (no FP64 instruction in this loop: it would wait for the other warps')
        float mf = 0.0f;
        if (heavy_table && q < 4 && R.pp && sc.x >= 0.0f) {
          const int fe = pdf_index(w.tag[q >> 1].f);
          mf = fe > 0 ? m2f[fe] : 0.0f;
        }
        // the blocks of both channels side by side (two chains of products)
        uint32_t oc[2][4];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const uint64_t d = dk + (uint64_t)(__float_as_int(sc.w) + c);
          philox(e0, e1, (uint32_t)d, (uint32_t)(d >> 32), k0, k1, oc[c]);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float ic = c == 0 ? sc.x : sc.y;
          if (!(ic >= 0.0f && ic < INFINITY)) continue;  // absent, or no trial
          const uint32_t* o = oc[c];
          const float lnTm = fminf(lnT, sc.z);
          float x = fmaf((float)o[0], 1.0f / 4294967296.0f, (float)o[1]) * (1.0f / 4294967296.0f);
          const bool tiny = o[1] < 16u;  // R below 2^-28: only an upper bound
          if (tiny) x = 3.7252903e-9f;
          const float lr = __logf(x);
          float v = fmaf(lr, ic, lnTm);
          float er = screen_error(ic, lr, v, lnTm, eT);
          bool sure = !tiny && ic < 1e30f;
          if (mf > 0.0f) {
            // the heavy-quark measure: t = m^2 + (t_max - m^2) R^(1/c) is at
            // least t_max R^(1/c), so its relative error is not larger
            const float lnF = __logf(mf * (1.0f + (float)kHqFloor));
            if (lnTm < lnF + kLnSlack) {
              doubt = doubt || lnTm > lnF - kLnSlack;  // whether it draws is close
              if (lnTm <= lnF - kLnSlack) continue;
            }
            v = __logf(mf + (__expf(lnTm) - mf) * __expf(fmaxf(lr * ic, -80.0f)));
            er += kLnSlack;
            if (v < lnF + kLnSlack) sure = false;  // may be below the channel's floor
            if (v + er < lnF - kLnSlack) { ++nt; if (q < 4 && R.pp) nt += 1 << 16; continue; }
          }
          nt += (q < 4 && R.pp) ? 1 + (1 << 16) : 1;
          const float ub = v + er;
          if (sure) lmax = fmaxf(lmax, v - er);
          if (ub > u1) { u2 = u1; u1 = ub; v1 = v; er1 = er; i1 = 2 * q + c; }
          else u2 = fmaxf(u2, ub);
        }
      }
    }
    const float Lm = g.max(lmax);
    const unsigned cand = g.ballot(u1 >= Lm && u1 > -INFINITY);
    const unsigned second = g.ballot((u2 >= Lm && u2 > -INFINITY) || doubt);
    // no trial above the cutoff
    const bool below = !g.ballot(u1 >= lnTc - kLnSlack || doubt);
    if (heavy_table || k == 0) {
      const int s = g.sum(nt);
      if (heavy_table ? gl == k : true) my_trials = s;
    }
    const int wl = __ffs(cand) - 1;
    const float wv = g.get(v1, wl < 0 ? 0 : wl), we = g.get(er1, wl < 0 ? 0 : wl);
    const int wi = g.get(i1, wl < 0 ? 0 : wl);
    // (some channel's lower bound is finite, and it alone reaches it)
    const bool clear = !below && Lm > -INFINITY && __popc(cand) == 1 && !second;
    // a first cycle that the bounds do not decide: exact trials of the
    // channels in question
    const bool decide = going && k == 0 && !below && !clear;
    int xi = -1;
    if (__any_sync(kAll, decide)) {
      double bt = -1.0;
      int bidx = 0x7fffffff, xt = 0;
      if (decide) {
        for (int q = gl; q < ne; q += G) {
          const float4 sc = w.scr[q];
          for (int c = 0; c < 2; ++c) {
            const float ic = c == 0 ? sc.x : sc.y;
            if (!(ic >= 0.0f && ic < INFINITY)) continue;
            const uint64_t d = dk + (uint64_t)(__float_as_int(sc.w) + c);
            const uint4 o = block_of(S.id, d, k0, k1);
            const EndX& x = w.end[q];
            bool counted;
            const double tt = exact_trial(x, c, heavy_m2(P, x.type, w.tag[q >> 1].f), S.t, R.t_cut, u01(o.x, o.y),
                                          counted);
            if (counted) xt += (q < 4 && R.pp) ? 1 + (1 << 16) : 1;
            if (tt > bt) { bt = tt; bidx = 2 * q + c; }
          }
        }
      }
#pragma unroll 1
      for (int o = G / 2; o > 0; o >>= 1) {
        const double ot = g.xchg(bt, o);
        const int oi = g.xchg(bidx, o);
        if (ot > bt || (ot == bt && oi < bidx)) { bt = ot; bidx = oi; }
      }
      const int s = g.sum(xt);
      if (decide) {
        if (!heavy_table || gl == 0) my_trials = s;
        if (bidx != 0x7fffffff) xi = bidx;
      }
    }
    if (going) {
      if (below || (decide && xi < 0)) {
        ends_done = true;
        going = false;
      } else if (clear || decide) {
        const int win = clear ? wi : xi;
        if (gl == k) { my_q = win >> 1; my_c = win & 1; }
        len = k + 1;
        lnT = wv;
        eT = we;
        // near or below the cutoff, or decided exactly: the batch ends here
        if (decide || wv - we < lnTc + kLnSlack) going = false;
      } else {
        going = false;  // not decided in FP32: the next batch begins with it
      }
    }
  }

  // ---- exact scales and weights: lane j evaluates cycle j --------------
  Winner W;
  W.outcome = kVeto;
  W.violation = false;
  W.t = 0.0;
  W.type = W.ch = W.bi = W.bk = W.side = W.new_fl = W.fl_j = 0;
  W.z = W.omz = W.Rphi = W.a0 = W.a1 = W.a2 = W.a3 = 0.0;
  const bool mine = S.active && gl < len;
  const uint64_t dm = S.draw + (uint64_t)gl * (uint64_t)(S.nblk + 2);
  double pw = 1.0, tkin = 0.0, m2 = 0.0, Rz = 0.5;
  if (mine) {
    const EndX& x = w.end[my_q];
    const float4 sc = w.scr[my_q];
    const uint64_t d = dm + (uint64_t)(__float_as_int(sc.w) + my_c);
    const uint4 o = block_of(S.id, d, k0, k1);
    Rz = u01(o.z, o.w);
    pw = gm_exp(gm_div(gm_log(u01(o.x, o.y)), x.cc[my_c]));
    tkin = x.tkin;
    if (heavy_table) m2 = heavy_m2(P, x.type, w.tag[my_q >> 1].f);
  }
  double my_t = 0.0, tc = S.t;
  const int most = __reduce_max_sync(kAll, S.active ? len : 0);
  for (int k = 0; k < most; ++k) {
    const double tmax = fmin(tc, tkin);
    const double tt = m2 > 0.0 ? m2 + (tmax - m2) * pw : tmax * pw;
    if (gl == k) my_t = tt;
    tc = g.get(tt, k);
  }
  if (mine) {
    const uint64_t d1 = dm + (uint64_t)S.nblk;
    const uint4 o1 = block_of(S.id, d1, k0, k1), o2 = block_of(S.id, d1 + 1, k0, k1);
    weigh(P, w, R, S.n, my_q, my_c, my_t, Rz, o1, o2, W);
  }

  // ---- commit: the cycles up to the first that was not vetoed ----------
  const unsigned other = g.ballot(mine && W.outcome != kVeto);
  const int room = P.max_steps - S.steps;  // cycles before the cap
  int f = other ? __ffs(other) - 1 : -1;
  if (f >= room) f = -1;
  int done_cycles = f >= 0 ? f + 1 : min(len, room);  // committed
  const int out = g.get(W.outcome, f < 0 ? 0 : f);
  const bool viol = g.get((int)W.violation, f < 0 ? 0 : f) != 0;
  const bool tail_done = f < 0 && ends_done && done_cycles == len && len < room;
  // scale after the committed cycles (a cycle that ends without a veto test
  // leaves it)
  const int tl = f >= 0 && (out == kDone || out == kNumericT) ? f - 1 : done_cycles - 1;
  const double tn = g.get(my_t, tl < 0 ? 0 : tl);
  bool accepted = false;
  if (S.active) {
    const int counted = done_cycles + (tail_done ? 1 : 0);
    if (!heavy_table ? gl == 0 : gl < counted) {
      const unsigned long long times = heavy_table ? 1 : (unsigned long long)counted;
      cnt.trials += times * (unsigned long long)(my_trials & 0xffff);
      cnt.isr_trials += times * (unsigned long long)(my_trials >> 16);
    }
    if (tl >= 0) S.t = tn;
    S.steps += counted;
    S.draw += (uint64_t)done_cycles * (uint64_t)(S.nblk + 2);
    if (tail_done) S.draw += (uint64_t)S.nblk;
    if (f >= 0 && (out == kDone || out == kNumericT)) S.draw -= 2;
    if (gl == 0) {
      cnt.steps += counted;
      cnt.vetoes += f >= 0 ? f : done_cycles;
      if (f >= 0 && viol) cnt.violations += 1;
    }
    int st = GAPS_STATUS_ACTIVE;
    if (tail_done || (f >= 0 && out == kDone)) st = GAPS_STATUS_DONE;
    else if (f >= 0 && (out == kNumericT || out == kNumericW)) st = GAPS_ERR_NUMERIC;
    else if (f >= 0 && out == kCapacity) st = GAPS_ERR_CAPACITY;
    else if (f >= 0) accepted = true;
    if (st == GAPS_STATUS_ACTIVE && S.steps >= P.max_steps) st = GAPS_ERR_ITER_CAP;
    S.status = st;
  }

  // ---- emission --------------------------------------------------------
  if (__any_sync(kAll, accepted)) {
    emission(g, w, accepted, S.n, W, f < 0 ? 0 : f, S.eta0, S.eta1);
    const int pack = g.get(W.type | (W.bi << 2) | (W.bk << 10), f < 0 ? 0 : f);
    if (accepted) {
      S.chg = (pack & 3) == kII ? -1 : ((pack >> 2) & 0xff) | (((pack >> 10) & 0xff) << 8);
      S.n += 1;
      S.n_emit += 1;
      if (gl == 0) cnt.accepts += 1;
      S.table = true;
    }
  }

  // ---- finished events back into the caller's records ------------------
  if (S.active && S.status != GAPS_STATUS_ACTIVE) {
    for (int s = gl; s < S.n; s += G) {
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) E.P(mu, s, S.e) = w.p[4 * s + mu];
      const Tag tg = w.tag[s];
      E.F(s, S.e) = tg.f;
      E.C(s, S.e) = tg.c;
      E.A(s, S.e) = tg.a;
    }
    if (gl == 0) {
      E.npart[S.e] = S.n;
      if (S.t < INFINITY) E.t[S.e] = S.t;  // (else no cycle had a trial)
      E.eta[S.e] = S.eta0;
      E.eta[E.cap + S.e] = S.eta1;
      E.n_emit[S.e] = S.n_emit;
      E.draw[S.e] = S.draw;
      E.status[S.e] = S.status;
      if (S.status == GAPS_ERR_CAPACITY) cnt.err_cap += 1;
      else if (S.status == GAPS_ERR_ITER_CAP) cnt.err_iter += 1;
      else if (S.status == GAPS_ERR_NUMERIC) cnt.err_num += 1;
    }
    S.active = S.table = false;
  }
  __syncwarp();
}

__global__ void __launch_bounds__(kThreads, kMinBlocks)
    k_shower_fp64(const __grid_constant__ DevParams P, const __grid_constant__ DevEvents E, uint64_t first, uint64_t n_events,
                  unsigned per_block, unsigned char* pool, unsigned* taken, unsigned regions, int heavy_table) {
  __shared__ RowShared rows[kMaxRows];
  __shared__ float m2f[12];
  __shared__ unsigned char s_list[kGroups][256];
  __shared__ int s_region;
  __shared__ unsigned s_next;
  const int tid = threadIdx.x, lane = tid & 31, gl = tid & (kG - 1);
  if (tid < kMaxRows) {
    const RowParams& r = P.rows[tid < P.n_rows ? tid : 0];
    rows[tid] = RowShared{r.t_cut, r.as_over, r.as_over / (2.0 * kPi), (float)gm_log(r.t_cut), r.process != GAPS_EE_QQ};
  }
  if (tid < 12) m2f[tid] = (float)P.m2[tid];
  if (tid == 0) {
    s_next = 0;
    // a free part of the scratch pool: it has one for every block that can be
    // resident on the device at a time, whichever launches they belong to
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    int got = -1;
    for (unsigned k = 0; k < 64 * regions && got < 0; ++k) {
      const unsigned r = (smid * kMinBlocks + k) % regions;
      if (atomicCAS(&taken[r], 0u, 1u) == 0u) got = (int)r;
    }
    s_region = got;
    __threadfence();
  }
  __syncthreads();
  const uint64_t block0 = (uint64_t)blockIdx.x * per_block;
  const unsigned block_n = (unsigned)(n_events - block0 < per_block ? n_events - block0 : per_block);

  Counters cnt;
  if (s_region < 0) {
    // not expected, see above; should it happen, its events end with an error
    for (unsigned j = tid; j < block_n; j += kThreads) {
      cnt.finished += 1;
      if (E.status[block0 + j] != GAPS_STATUS_ACTIVE) continue;
      E.status[block0 + j] = GAPS_ERR_NUMERIC;
      cnt.err_num += 1;
    }
    flush_counters(P, cnt);
    return;
  }
  const size_t slot = (size_t)s_region * kGroups + tid / kG;
  Scratch w = scratch_of(pool + slot * (size_t)P.nmax * kSlotBytesPerParton, P.nmax);
  Event S;
  Group g{kG};
  bool exhausted = false, first_take = true;
  while (true) {
    // ---- a new event for every idle group ------------------------------
    while (__any_sync(kAll, !S.active && !exhausted)) {
      // the block's first events one to a group, spread over the warps first
      unsigned j = (unsigned)(tid >> 5) + (kThreads / 32) * (unsigned)(lane / kG);
      if (!first_take) {
        if (gl == 0 && !S.active && !exhausted) j = kGroups + atomicAdd(&s_next, 1u);
        j = __shfl_sync(kAll, j, 0, kG);
      }
      first_take = false;
      if (S.active || exhausted) continue;
      if (j >= block_n) { exhausted = true; continue; }
      const uint64_t e = block0 + j;
      S.e = e;
      S.id = first + e;
      if (gl == 0) cnt.finished += 1;
      S.status = E.status[e];
      if (S.status != GAPS_STATUS_ACTIVE) continue;
      S.n = E.npart[e];
      S.row = mix_row(P, S.id);
      if (S.n < 2 || S.n > P.nmax) {  // not a record written by the hard-process kernel
        if (gl == 0) { E.status[e] = GAPS_ERR_NUMERIC; cnt.err_num += 1; }
        continue;
      }
      for (int s = gl; s < S.n; s += kG) {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) w.p[4 * s + mu] = E.P(mu, s, e);
        w.tag[s] = Tag{E.F(s, e), E.C(s, e), E.A(s, e), 0};
      }
      // (a record without a scale, NaN, begins at its dipoles' largest ones)
      S.t = isnan(E.t[e]) ? INFINITY : E.t[e];
      S.eta0 = E.eta[e];
      S.eta1 = E.eta[E.cap + e];
      S.n_emit = E.n_emit[e];
      S.draw = E.draw[e];
      S.steps = 0;
      S.active = S.table = true;
      S.chg = -1;
    }
    const unsigned act = __ballot_sync(kAll, S.active);
    if (!act) break;
    if (g.G == kG && __popc(act) == kG && __all_sync(kAll, S.active || exhausted)) {
      // the warp's last event: all 32 lanes take it to its end
      const int src = __ffs(act) - 1;
      S.active = true;
      S.table = __shfl_sync(kAll, (int)S.table, src) != 0;
      S.e = __shfl_sync(kAll, S.e, src);
      S.id = __shfl_sync(kAll, S.id, src);
      S.draw = __shfl_sync(kAll, S.draw, src);
      S.n = __shfl_sync(kAll, S.n, src);
      S.n_emit = __shfl_sync(kAll, S.n_emit, src);
      S.steps = __shfl_sync(kAll, S.steps, src);
      S.row = __shfl_sync(kAll, S.row, src);
      S.status = GAPS_STATUS_ACTIVE;
      S.nblk = __shfl_sync(kAll, S.nblk, src);
      S.chg = __shfl_sync(kAll, S.chg, src);
      S.t = __shfl_sync(kAll, S.t, src);
      S.eta0 = __shfl_sync(kAll, S.eta0, src);
      S.eta1 = __shfl_sync(kAll, S.eta1, src);
      w = scratch_of(reinterpret_cast<unsigned char*>(
                         __shfl_sync(kAll, reinterpret_cast<unsigned long long>(w.p), src)), P.nmax);
      exhausted = true;
      g.G = 32;
    }
    batch(g, g.G == kG ? kG : kWideBatch, P, E, w, rows, m2f, s_list[tid / g.G * (g.G / kG)], S, cnt, heavy_table != 0);
  }
  flush_counters(P, cnt);
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    atomicExch(&taken[s_region], 0u);
  }
}

}  // namespace

// Scratch pool of the FP64 shower: parts for every block that can be resident
// on the device at a time, with a flag each, so that calls on several streams
// share it.
size_t fp64_pool_layout(int n_sm, int nmax, unsigned& regions, size_t& flag_bytes) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_shower_fp64, kThreads, 0) != cudaSuccess || per_sm < 1)
    per_sm = kMinBlocks;
  regions = (unsigned)(n_sm * per_sm);
  flag_bytes = (regions * sizeof(unsigned) + 255) / 256 * 256;
  return flag_bytes + (size_t)regions * kGroups * (size_t)nmax * kSlotBytesPerParton;
}

cudaError_t launch_shower_fp64(const DevParams& P, const DevEvents& E, uint64_t first, uint64_t n, void* pool,
                               unsigned regions, size_t flag_bytes, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  // events a block takes: one round over the resident blocks, up to
  // kMaxPerBlock (its groups refill from the block's share); few events go one
  // to a block, where an event has a warp's FP64 pipe for itself
  uint64_t per = (n + regions - 1) / regions;
  if (per > kMaxPerBlock) per = kMaxPerBlock;
  int heavy = 0;
  for (int f = 0; f < 12; ++f) heavy = heavy || P.thr[f] >= 0;
  const unsigned grid = (unsigned)((n + per - 1) / per);
  k_shower_fp64<<<grid, kThreads, 0, stream>>>(P, E, first, n, (unsigned)per, (unsigned char*)pool + flag_bytes,
                                                (unsigned*)pool, regions, heavy);
  return cudaGetLastError();
}

}  // namespace gaps
