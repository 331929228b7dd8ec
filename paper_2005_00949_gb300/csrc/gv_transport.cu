// gv_transport.cu -- the stepping loop of GeantV (Sec. 2.1.2, Fig.
// "simulation stages") as a persistent, chunk-claiming CUDA kernel driven
// generation by generation from a captured CUDA graph (a device-side while
// loop over bodies of generations), plus the C ABI.
//
// One generation: every live track of the three per-type queues (and the
// primaries injected by the refill plan) is claimed in chunks (a block's
// worth, fewer when few tracks are live; positrons, electrons, photons,
// primaries in that order), stepped K times, and written back -- survivors
// and secondaries appended to the other parity's queues with warp-aggregated
// atomics (the basketizer of scheduler v3, Sec. 2.1.1).  The last block to
// finish writes the plan of the next generation: queue chunk ranges and
// claim size, primaries to inject (the event server refill, bounded by a
// live-track budget) and the steps per claim.
//
// Host side: gv_transport enqueues one transport on the context's stream,
// ordered after the caller's stream (which then waits for it), and returns;
// gv_sync waits for it and fills the caller's result record from the
// control block copied back to pinned memory.  The step kernels read the
// transport's state record from constant memory, one copy per precision and
// GPU; transports of different contexts on one GPU take turns on it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "gv_state.cuh"

namespace gv {

// ------------------------------------------------------------------ sinks
// Scoring (SteppingActions, Sec. 3.8.1).  A lane keeps one pending
// (event, sub-slab) deposit: consecutive deposits of its track to the same sub-slab merge with a
// compensated (Kahan) sum in R; a deposit to another sub-slab flushes the
// pending one with an FP64 atomic; at the end of every round the warp groups
// its pending deposits by key (__match_any_sync), sums each group with a
// compensated shuffle reduction, and one lane per group adds it to the FP64
// tally.  pd == nullptr scores directly.
constexpr unsigned long long kNoKey = ~0ull;

template <typename R> struct Pending {
  unsigned long long key;
  R sum, comp;
};

template <typename R> __device__ __forceinline__ void kahan_add(R &sum, R &comp, R v) {
  const R y = v - comp;
  const R t = sum + y;
  comp = (t - sum) - y;
  sum = t;
}

// A tally's addition, with nothing returned (an atomicAdd here cost a charged
// step 80 cycles, of 1500 at the time and 950 now).
__device__ __forceinline__ void red_add(double *p, double v) {
  asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// row: the event's row of the sub-slab tally.
// EXT: compiled with the cell histogram and the per-event counters; a
// kernel without them serves contexts that have neither.
template <typename R, bool EXT = true>
__device__ __forceinline__ void deposit(const DevState<R> *S, double *row, unsigned ev, int sub, double px, double py,
                                        R dE, Pending<R> *pd = nullptr) {
  if (!(dE != R(0)) || sub < 0) return;
  GV_CHECK(&S->ctl->status, ev < S->n_events && sub < S->view.geo.nsub);
  if (pd) {
    const unsigned long long key = static_cast<unsigned long long>(ev) * S->view.geo.nsub + sub;
    if (pd->key == key) {
      kahan_add(pd->sum, pd->comp, dE);
    } else {
      if (pd->key != kNoKey)
        atomicAdd(&S->edep[pd->key], f2d(pd->sum) - f2d(pd->comp));
      pd->key = key;
      pd->sum = dE;
      pd->comp = R(0);
    }
  } else {
    red_add(&row[sub], f2d(dE));
  }
  if (EXT && S->cell) {
    const GeoConst &g = S->view.geo;
    const int layer = sub / g.nsub_layer;
    // the offset from the wall in FP64, the cell index in FP32 (a cell
    // edge moves by ~1e-7 of the box width; no FP64 division)
    int ix = __float2int_rd(static_cast<float>(px + g.hx) * g.inv_pitch_x);
    int iy = __float2int_rd(static_cast<float>(py + g.hy) * g.inv_pitch_y);
    ix = ix < 0 ? 0 : (ix >= g.nx ? g.nx - 1 : ix);
    iy = iy < 0 ? 0 : (iy >= g.ny ? g.ny - 1 : iy);
    red_add(&S->cell[(static_cast<size_t>(layer) * g.nx + ix) * g.ny + iy], f2d(dE));
  }
}

// Warp flush of the pending deposits (all 32 lanes, converged).
template <typename R> __device__ __forceinline__ void warp_flush(const DevState<R> *S, Pending<R> &p) {
  const unsigned m = __match_any_sync(0xffffffffu, p.key);
  if (p.key != kNoKey) {
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    const R v = p.sum - p.comp;
    R acc = v, comp = R(0);
    unsigned rest = m & ~(1u << leader);
    while (rest) {  // every lane of the group runs the same iterations
      const int src = __ffs(rest) - 1;
      rest &= rest - 1u;
      const R w = __shfl_sync(m, v, src);
      if (lane == leader) kahan_add(acc, comp, w);
    }
    if (lane == leader) atomicAdd(&S->edep[p.key], f2d(acc) - f2d(comp));
  }
  p.key = kNoKey;
}

template <typename R> struct Trk {
  double x, y, z;
  R u, v, w, E, nlam;
  unsigned long long id;
  unsigned ev, step;
  int sub, flags, type;
};

__device__ __forceinline__ void set_status(Ctl *ctl, int code) { atomicCAS(&ctl->status, 0, code); }

// The key of a track's random stream and one counter block of step k.
template <typename R>
__device__ __forceinline__ uint4 track_draw(const DevState<R> *S, unsigned long long id, unsigned ev, uint32_t k,
                                            uint32_t block) {
  return philox4x32_10(make_uint4(static_cast<uint32_t>(id), static_cast<uint32_t>(id >> 32), k, block),
                       S->seed_lo ^ (ev + S->ev_base), S->seed_hi);
}

// Integral approach at the post-step point: the process whose cumulative
// post-step cross section first exceeds `target` (u Sigma_max), or -1 (no
// interaction) above their sum.  Out of line: the option would otherwise
// cost every step kernel registers.
template <typename R> __device__ __noinline__ int integral_choice(const View<R> &V, int mat, int type, R E, R target) {
  int i;
  R f;
  grid_pos(V, E, i, f);
  const V4<R> p4 = lookup_at(V, mat, type, i, f);
  R cum = p4.x;
  if (target < cum) return 0;
  cum += p4.y;
  if (target < cum) return 1;
  if (type == 2) {
    cum += p4.z;
    if (target < cum) return 2;
  }
  return -1;
}

// The interaction due after step k - 1 with the bound Smax, of a track now
// at step k: its process, or -1 and the next n_lambda.  Out of line for the same
// reason: a run that ended at every rejection gave the block a round for each
// (integral approach, FP64, 2360 tracks in 1 cm: 1.82 ms, now 1.23).
template <typename R> struct IntegralStep {
  R nlam;
  int proc;
};
template <typename R>
__device__ __noinline__ IntegralStep<R> integral_step(const View<R> &V, const DevState<R> *S, unsigned long long id,
                                                      unsigned ev, uint32_t k, int mat, int type, R E, R Smax) {
  IntegralStep<R> c;
  c.proc = integral_choice(V, mat, type, E, u24<R>(track_draw(S, id, ev, k - 1u, 0u).y) * Smax);
  c.nlam = R(-1);
  if (c.proc < 0) c.nlam = -m_log(u24<R>(track_draw(S, id, ev, k, 0u).x));
  return c;
}

// ------------------------------------------------------------------ a run of steps
// How a track's run of along-steps ended.
constexpr int kRunOn = 0;    // its budget is used, or a new n_lambda is due: it goes on in the next round
constexpr int kRunPhys = 1;  // a physics-limited step: the process choice is due
constexpr int kRunEnd = 2;   // it ended: below the tracking cut, or out of the box
constexpr int kRunRest = 3;  // a positron stopped: it annihilates at rest
constexpr int kNoteEpEsc = 1, kNoteUnscat = 2;  // an escaped positron, an unscattered primary

// What a run leaves for the process choice and the step counters.
template <typename R> struct Run {
  R sig0, sig1, sig2;  // cross sections of the last step
  unsigned n_st, n_geom, n_iter;
  int note;
  int proc;  // the integral approach's choice after the last step (0 without it)
};

// The tables as the step kernels stage them (stage_tables), addressed from the
// start of shared memory: through the view's pointers every load would be a
// generic one, behind the load of the pointer, which the deposits' atomics
// make the compiler repeat in every step.  What is the same for all tracks
// (planes' count, half widths, cuts) the steps read from the state record in
// constant memory, as operands.
template <typename R> struct Staged {
  const V4<R> *xs;
  const double *zb;
  const float *inv_node;
  const SubRec<R> *rec;
  __device__ __forceinline__ explicit Staged(const DevState<R> *S) {
    extern __shared__ __align__(32) unsigned char smem[];
    xs = reinterpret_cast<const V4<R> *>(smem);
    zb = reinterpret_cast<const double *>(smem + S->xs_bytes);
    inv_node = reinterpret_cast<const float *>(smem + S->xs_bytes + S->zb_bytes);
    rec = reinterpret_cast<const SubRec<R> *>(smem + S->rec_off);
  }
};

// A track left the box (or there is nothing left to stop it).
template <typename R, bool EXT>
__device__ __forceinline__ void escape(const DevState<R> *S, const Trk<R> &t, int plane, Run<R> &r) {
  atomicAdd(&S->escape[t.ev], f2d(t.E));
  if (t.type == 2) r.note |= kNoteEpEsc;
  if ((t.flags & kFlagPrimary) && !(t.flags & kFlagInteracted) && plane == S->view.geo.nsub) r.note |= kNoteUnscat;
}

// Photons: PreStep to the end of a run of at most `budget` steps, every one
// but the last limited by a boundary.  The energy, and with it the grid
// position, and the direction are the same for the whole run; every step
// after the first starts on the plane of its sub-slab, so its FP64 plane
// difference is the tabulated thickness (the same number), and z is needed
// only where the run ends.  A step costs the FP64 pipe its two lateral
// additions instead of three additions, a difference and a conversion, and
// no wall test while the run's lateral bound clears the plane (2000 x 10 GeV:
// 5.39 -> 5.02 ms with the branch-free widening, the shared exponential of
// loss_at and one-branch grid_pos).
//
// A run is one chain of dependent instructions, so the loop has one exit, and
// the next sub-slab's record and cross sections are fetched before the exit is
// decided: 480 -> 176 cycles a step for a warp alone on its SM.
// A run also ends where a wall may limit the next step, by the bound along its
// direction (lateral_way): before the last step of a flight that ends on a wall.
// (That step in the same run, in the loop or after it, cost 2000 x 10 GeV 1 to
// 2 %.)  With a bound that did not know the direction, against the next plane,
// nearly every step ended a run in a box about as wide as its layers are thick:
// 300 x 1 GeV in FP64 in a box of 1 cm took 5.67 ms (now 3.04), 1000 x 1 GeV in
// mixed precision 1.36 (0.70), 1e5 photons of 1 MeV in a box of 1 mm 0.75 (0.33).
template <typename R, bool EXT>
__device__ __forceinline__ int photon_run(const DevState<R> *S, Trk<R> &t, int budget, Run<R> &r) {
  const Staged<R> V(S);
  const GeoConst &geo = S->view.geo;
  int gi;
  R gf;
  const R INF = r_inf<R>();
  const bool up = t.w > R(0);
  int sub = t.sub;
  GV_CHECK(&S->ctl->status, sub >= 0 && sub < geo.nsub);
  SubRec<R> rec = V.rec[sub];
  R h = static_cast<R>(V.zb[plane_ahead(t.w, sub)] - t.z);
  grid_pos_on(V.inv_node, t.E, gi, gf);
  GV_CHECK(&S->ctl->status, gi >= 0 && gi <= kGridN - 2);
  const V4<R> *const tab = V.xs + gi;
  const Divisor<R> by_w(t.w);
  float lat = lateral_way(geo, t.x, t.y, t.u, t.v);
  const int last = geo.nsub - 1, dir = up ? 1 : -1;
  V4<R> sig = lerp4(tab[rec.row], tab[rec.row + 1], gf);  // ComputeIntLen
  R nlam = t.nlam, s;
  // GeomQuery
  R d = way_to_plane(by_w, t.w, h);
  int m = 0, pl = -1;
  if (!walls_clear(lat, d)) walls(geo, t.x, t.y, t.u, t.v, d, d, pl);
  if (d < R(0)) d = R(0);
  int row = rec.row, back_row = -1;  // of this sub-slab and the one before: table row, cross sections, path across
  V4<R> back_sig = sig;
  R back_h = R(0), back_d = R(0);
  h = R(0);  // (the first path starts inside)
  bool finite, geom, out;
  R Sig = sig.x + sig.y + sig.z;
  R s_phys = Sig > R(0) ? q_div(nlam, Sig) : INF;
  s = INF < d ? INF : d;
  s = s_phys < s ? s_phys : s;
  for (;;) {
    const int next = sub + dir;
    const SubRec<R> nrec = V.rec[min(max(next, 0), last)];
    const R nh = up ? nrec.thick : -nrec.thick;  // from the plane it enters through
    V4<R> nsig;
    R nd;
    if (sizeof(R) == 4) {
      nsig = lerp4(tab[nrec.row], tab[nrec.row + 1], gf);
      nd = by_w.div(nh);
    }
    finite = s < INF;
    geom = d == s;
    out = pl < -1 || static_cast<unsigned>(next) > static_cast<unsigned>(last);
    t.x += f2d(s * t.u);
    t.y += f2d(s * t.v);
    lat = lat_after(lat, s);
    ++m;
    if (geom && Sig > R(0)) nlam = nlam - s * Sig;
    if (!finite || !geom || out || !(nlam > R(0)) || m >= budget) break;
    if (sizeof(R) == 8) {
      // FP64 arithmetic is worth waiting for the exit, and in alternating
      // layers the sub-slab before this one has the next one's numbers (300 x
      // 10 GeV: 8.45 -> 8.34 ms)
      if (nrec.row == back_row) {
        nsig = back_sig;
      } else {
        nsig = lerp4(tab[nrec.row], tab[nrec.row + 1], gf);
      }
      if (nh == back_h) {
        nd = back_d;
      } else {
        nd = by_w.div(nh);
      }
      back_row = row;
      back_sig = sig;
      back_h = h;
      back_d = d;
      row = nrec.row;
      h = nh;
    }
    Sig = nsig.x + nsig.y + nsig.z;
    s_phys = Sig > R(0) ? q_div(nlam, Sig) : INF;
    s = INF < nd ? INF : nd;
    s = s_phys < s ? s_phys : s;
    if (!walls_clear(lat, s)) break;
    sub = next;
    d = nd;
    sig = nsig;
  }
  r.sig0 = sig.x;
  r.sig1 = sig.y;
  r.sig2 = sig.z;
  r.n_iter = static_cast<unsigned>(m);
  if (!finite) --m;  // not a step: nothing stops the track
  r.n_st = static_cast<unsigned>(m);
  t.step += static_cast<unsigned>(m);
  r.n_geom = static_cast<unsigned>(finite && !geom ? m - 1 : m);
  int end = kRunOn;
  if (!finite || (geom && out)) {
    end = kRunEnd;
    escape<R, EXT>(S, t, !finite || pl < -1 ? pl : (up ? geo.nsub : 0), r);
  } else {
    if (geom) sub += dir;
    if (r.n_geom) t.z = V.zb[up ? sub : sub + 1];  // the plane it entered through
    if (!geom) {  // physics (a photon has no other limit)
      t.z += f2d(s * t.w);
      nlam = R(0);
      end = kRunPhys;
    }
  }
  t.nlam = nlam;
  t.sub = sub;
  return end;
}

// Electrons and positrons: a run of at most `budget` steps, each limited by
// a boundary, by the continuous loss (or the field) or, the last one, by
// physics.  1600 (step within one node interval) and 2100 cycles (across
// several) a step for a warp alone on its SM became 950 and 1215.
// The walls are looked at where the bound (lateral_free: the direction may
// change) does not clear the step itself: its other limits are known by then, and
// mostly millimetres, where the plane ahead of a slanted track is far.  A run
// that ended wherever the bound did not clear that plane took one step a round
// beside a wall (5000 x 10 MeV e- in FP64 in a box of 0.4 mm 1.15 -> 0.80 ms; in 40 cm
// 2000 x 10 GeV 3.82 -> 3.78).
template <typename R, bool FIELD, bool OPTS, bool EXT>
__device__ __forceinline__ int charged_run(const View<R> &V, const DevState<R> *S, Trk<R> &t, int budget, Run<R> &r,
                                           Pending<R> *pd) {
  const Staged<R> T(S);
  const GeoConst &geo = S->view.geo;
  const R INF = r_inf<R>(), tcut = S->view.rc.tcut;
  const bool pos = t.type == 2, msc = OPTS && (S->view.cut.mask & GV_P_MSC);
  double *const edep = S->edep + static_cast<size_t>(t.ev) * geo.nsub;
  GV_CHECK(&S->ctl->status, t.sub >= 0 && t.sub < geo.nsub);
  float lat = lateral_free(geo, t.x, t.y);
  int plane = plane_ahead(t.w, t.sub);
  R dz = static_cast<R>(T.zb[plane] - t.z);
  int row = T.rec[t.sub].row + (pos ? 2 * kGridN : kGridN);
  Divisor<R> by_w(t.w);
  int lim, wall = -1;
  // the first step's geometry; later ones start the plane's FP64 difference as
  // soon as z is known, and it is done when the loss is
  R s_geom = way_to_plane(by_w, t.w, dz);
  int m = 0, end = kRunOn;
  for (;;) {
    ++r.n_iter;
    const V4<R> *const tab = T.xs + row;
    // the scattering's numbers of this step (counter block 2), early
    uint4 r2 = make_uint4(0u, 0u, 0u, 0u);
    if (msc) r2 = track_draw(S, t.id, t.ev, t.step, 2u);
    // ComputeIntLen; the pre-step energy's grid position serves the lookup and the loss
    int gi;
    R gf;
    grid_pos_on(T.inv_node, t.E, gi, gf);
    const V4<R> n0 = tab[gi], n1 = tab[gi + 1];
    const V4<R> s4 = lerp4(n0, n1, gf);
    r.sig0 = s4.x;
    r.sig1 = s4.y;
    r.sig2 = pos ? s4.z : R(0);
    const R Sig = r.sig0 + r.sig1 + r.sig2;
    // integral approach: the step is drawn with the bound Sigma_max(E) of the
    // cross sections the track can reach; the interaction is accepted at the
    // post-step point
    R Smax = Sig;
    if (OPTS && (S->view.cut.mask & GV_P_INTEGRAL)) {
      const R *mx = V.smax + (V.smat[t.sub] * 2 + t.type - 1) * kGridN;
      Smax = mx[gi] + gf * (mx[gi + 1] - mx[gi]);
    }
    const R s_phys = Smax > R(0) ? q_div(t.nlam, Smax) : INF;
    const R Rr = range_of(s4, t.type);
    const R a = static_cast<R>(kAlphaR) * Rr, b = Rr < static_cast<R>(kRhoF) ? Rr : static_cast<R>(kRhoF);
    R s_cont = a > b ? a : b;
    R curv = R(0);
    if (FIELD && S->view.rc.field_k != R(0)) {  // the field's step limit acts like the continuous one
      curv = field_curv(S->view.rc.field_k, t.type, t.E);
      const R sf = field_limit(geo.field_axis, curv, t.u, t.v, t.w);
      s_cont = sf < s_cont ? sf : s_cont;
    }
    const R ahead = s_geom;
    if (s_geom < R(0)) s_geom = R(0);
    R s = s_cont < s_geom ? s_cont : s_geom;
    s = s_phys < s ? s_phys : s;
    if (!walls_clear(lat, s)) {
      lat = lateral_free(geo, t.x, t.y);
      if (nearer_wall(geo, t.x, t.y, t.u, t.v, s, ahead, s_geom, wall)) {
        s = s_geom < s ? s_geom : s;
        // the wall that the pre-step direction points at (-4, -5: the lower one):
        // a field may turn the track within the step
        if (!((wall == -2 ? t.u : t.v) > R(0))) wall -= 2;
      }
    }
    const int next = slab_behind(t.w, t.sub, geo.nsub, wall);
    lim = (s_geom == s) ? 0 : (s_phys == s ? 1 : 2);
    if (!(s < INF)) {
      escape<R, EXT>(S, t, -1, r);
      end = kRunEnd;
      wall = -1;
      break;
    }
    // Propagation: FP64 positions, advanced by displacements s d formed in R
    // (s and d are R already; an FP32 displacement is widened exactly on the
    // integer ALU, leaving the FP64 pipe one addition per coordinate; in FP64
    // mode this is one fused multiply-add)
    double mx = 0.0, my = 0.0;  // step midpoint: only cell scoring reads it
    if (FIELD && S->view.rc.field_k != R(0)) {  // the helix of the pre-step momentum
      const R d0[3] = {t.u, t.v, t.w};
      R dp[3], nd[3];
      if (EXT && S->cell) {
        helix(geo.field_axis, curv, R(0.5) * s, d0, dp, nd);
        mx = t.x + f2d(dp[0]);
        my = t.y + f2d(dp[1]);
      }
      helix(geo.field_axis, curv, s, d0, dp, nd);
      t.x += f2d(dp[0]);
      t.y += f2d(dp[1]);
      t.z += f2d(dp[2]);
      t.u = nd[0];
      t.v = nd[1];
      t.w = nd[2];
      by_w = Divisor<R>(t.w);
    } else {
      if (EXT && S->cell) {
        mx = t.x + f2d(R(0.5) * s * t.u);
        my = t.y + f2d(R(0.5) * s * t.v);
      }
      t.x += f2d(s * t.u);
      t.y += f2d(s * t.v);
      t.z += f2d(s * t.w);
    }
    const int crossed = plane;  // chosen with the pre-step direction
    if (lim == 0 && wall == -1) t.z = T.zb[crossed];
    const int pre_sub = t.sub, sub = lim == 0 && next >= 0 ? next : t.sub;
    plane = plane_ahead(t.w, sub);
    if (!msc) dz = static_cast<R>(T.zb[plane] - t.z);
    row = T.rec[sub].row + (pos ? 2 * kGridN : kGridN);
    lat = lat_after(lat, s);
    if (Smax > R(0)) t.nlam = (lim == 1) ? R(0) : t.nlam - s * Smax;
    ++t.step;
    ++r.n_st;
    r.n_geom += lim == 0 ? 1u : 0u;
    const R E_pre = t.E;
    // AlongStepAction
    const R Li = pos ? n0.w : n0.z;
    const R dL = (pos ? n1.w : n1.z) - Li;
    const Loss<R> loss = loss_at(tab, t.type, t.E, gi, gf, Li, dL, loss_slope(n0, t.type, dL), s, Rr);
    const R Ep = loss_energy(loss);
    deposit<R, EXT>(S, edep, t.ev, pre_sub, mx, my, t.E - Ep, pd);
    t.E = Ep;
    ++m;
    if (t.E < tcut) {
      if (lim == 0 && wall < -1) {  // it stops on the wall
        const double w = wall == -2 ? geo.wx[1] : (wall == -4 ? geo.wx[0] : (wall == -3 ? geo.wy[1] : geo.wy[0]));
        if (wall & 1) t.y = w;
        else t.x = w;
      }
      deposit<R, EXT>(S, edep, t.ev, pre_sub, t.x, t.y, t.E, pd);
      end = t.type == 2 ? kRunRest : kRunEnd;
      break;
    }
    // multiple scattering of a track that stays in the box (counter block 2)
    if (msc && !(lim == 0 && next < 0)) {
      const R um[4] = {u24<R>(r2.x), u24<R>(r2.y), u24<R>(r2.z), u24<R>(r2.w)};
      R dm[3] = {t.u, t.v, t.w};
      msc_step(geo, T.zb[pre_sub], T.zb[pre_sub + 1], S->view.rc.inv_X0[V.smat[pre_sub]], E_pre, t.E, s, dm, t.x, t.y,
               t.z, um, lat);
      t.u = dm[0];
      t.v = dm[1];
      t.w = dm[2];
      plane = plane_ahead(t.w, sub);
      dz = static_cast<R>(T.zb[plane] - t.z);
      by_w = Divisor<R>(t.w);
    }
    if (lim == 0 && next < 0) {
      escape<R, EXT>(S, t, wall < -1 ? wall : crossed, r);
      end = kRunEnd;
      break;
    }
    t.sub = sub;
    if (lim == 1) {
      if (OPTS && (S->view.cut.mask & GV_P_INTEGRAL)) {
        const IntegralStep<R> c = integral_step(V, S, t.id, t.ev, t.step, V.smat[t.sub], t.type, t.E, Smax);
        if (c.proc < 0) t.nlam = c.nlam;  // nothing happens there: the run goes on
        r.proc = c.proc;
      }
      if (!OPTS || r.proc >= 0) {
        end = kRunPhys;
        break;
      }
    }
    if (m >= budget || !(t.nlam > R(0))) break;
    s_geom = way_to_plane(by_w, t.w, dz);
    wall = -1;
  }
  return end;
}

// One round of a track: PreStep, a new n_lambda where one is due, a run of
// along-steps, and the process choice after a physics-limited one.  Returns
// the request key of the final state now due (type * 3 + process, or
// kKeyRest), or -1; kk is the step whose counter blocks its final state
// draws from, u2 and u3 the words of block 0 it samples with.  `alive` falls
// when the track ended or handed itself to an at-rest annihilation.
//
// The random numbers are drawn here once per round, outside the loop over
// steps: a step that leaves a track without n_lambda (an interaction is the
// rule, a rounding in n_lambda - s Sigma the exception) ends its run, so
// that its warp draws for all of its tracks together; the second block of an
// interaction is drawn by the lane that runs its final state.  Inside the
// loop every draw ran for whichever few lanes of the warp were due it.
template <typename R, bool FIELD, bool OPTS, bool EXT>
__device__ __forceinline__ int run_round(const View<R> &V, const DevState<R> *S, Trk<R> &t, bool &alive, int budget_g,
                                         int budget, uint32_t &kk, R &u2, R &u3, Run<R> &r, Pending<R> *pd) {
  r.n_st = r.n_geom = r.n_iter = 0;
  r.note = 0;
  if (OPTS) r.proc = 0;
  kk = 0;
  if (!alive) return -1;
  int end;
  if (t.E < V.rc.tcut) {  // PreStep: tracking cut
    r.n_iter = 1;
    kk = t.step;
    deposit<R, EXT>(S, S->edep + static_cast<size_t>(t.ev) * S->view.geo.nsub, t.ev, t.sub, t.x, t.y, t.E, pd);
    end = t.type == 2 ? kRunRest : kRunEnd;
  } else {
    if (t.nlam <= R(0)) t.nlam = -m_log(u24<R>(track_draw(S, t.id, t.ev, t.step, 0u).x));
    end = t.type == 0 ? photon_run<R, EXT>(S, t, budget_g, r)
                      : charged_run<R, FIELD, OPTS, EXT>(V, S, t, budget, r, pd);
    kk = t.step - 1u;
  }
  if (EXT && S->evcnt && (r.n_st || r.note)) {  // the optional per-event rows
    unsigned long long *row = &S->evcnt[static_cast<size_t>(t.ev) * GV_NCOUNT];
    atomicAdd(&row[GV_C_STEPS], static_cast<unsigned long long>(r.n_st));
    atomicAdd(&row[GV_C_STEPS_G + t.type], static_cast<unsigned long long>(r.n_st));
    if (r.note & kNoteEpEsc) atomicAdd(&row[GV_C_EP_ESC], 1ull);
    if (r.note & kNoteUnscat) atomicAdd(&row[GV_C_UNSCAT], 1ull);
  }
  // NaN energy, or a non-finite z (tested on its exponent bits: an FP64
  // comparison would take the FP64 pipe)
  if (!(t.E == t.E) || (__double2hiint(t.z) & 0x7ff00000) == 0x7ff00000) {
    set_status(S->ctl, GV_ERR_NUMERIC);
    alive = false;
    return -1;
  }
  if (end == kRunEnd || end == kRunRest) {
    alive = false;
    return end == kRunRest ? kKeyRest : -1;
  }
  if (end == kRunOn) return -1;
  // PostStepActions: process choice
  const uint4 r0 = track_draw(S, t.id, t.ev, kk, 0u);
  int proc = -1;
  if (OPTS && t.type != 0 && (V.cut.mask & GV_P_INTEGRAL)) {  // chosen in the run
    proc = r.proc;
  } else {
    const R target = u24<R>(r0.y) * (r.sig0 + r.sig1 + r.sig2);
    R cum = r.sig0;
    if (target < cum) proc = 0;
    else {
      cum += r.sig1;
      if (target < cum) proc = 1;
      else {
        cum += r.sig2;
        if (target < cum) proc = 2;
      }
    }
    if (proc < 0) proc = r.sig2 > R(0) ? 2 : (r.sig1 > R(0) ? 1 : (r.sig0 > R(0) ? 0 : -1));
  }
  t.nlam = R(-1);
  u2 = u24<R>(r0.z);
  u3 = u24<R>(r0.w);
  return proc < 0 ? -1 : t.type * 3 + proc;
}

// PostStepActions of the request `key`: the final state and its local
// deposit.  Returns 1 if the particle survives, 0 if it ended, -1 if the
// process was kinematically closed at the post-step energy (nothing
// changes).  np, na: pairs and annihilations made.  ids: the words that name
// its first two secondaries (push_kids), drawn with its own numbers: the two
// chains of Philox rounds run side by side.
template <typename R, bool OPTS = true, bool EXT = true, bool ALT = false>
__device__ __forceinline__ int final_state(const View<R> &V, const DevState<R> *S, int key, R &E, R d[3], R u2, R u3,
                                           Kids<R> &kids, unsigned ev, int sub, double x, double y,
                                           unsigned long long id, uint32_t kk, int &np, int &na,
                                           uint4 &ids, Pending<R> *pd = nullptr) {
  const uint4 r1 = track_draw(S, id, ev, kk, 1u);
  ids = track_draw(S, id, ev, kk, kTagId);
  const R u[8] = {R(0), R(0), u2, u3, u24<R>(r1.x), u24<R>(r1.y), u24<R>(r1.z), u24<R>(r1.w)};
  int r = 0;
  bool rest = key == kKeyRest;
  if (!rest) {
    const int type = key / 3;
    R local;
    const RngKey g = {static_cast<uint32_t>(id), static_cast<uint32_t>(id >> 32), kk, S->seed_lo ^ (ev + S->ev_base),
                      S->seed_hi};
    r = interact<R, OPTS, ALT>(V, type, key - 3 * type, E, d, u, g, kids, local, np, na, rest);
    if (r < 0) return -1;
    deposit<R, EXT>(S, S->edep + static_cast<size_t>(ev) * S->view.geo.nsub, ev, sub, x, y, local, pd);
  }
  if (rest) {  // a stopped positron, of this final state or of the run
    at_rest(kids, u[6], u[7]);
    na += 1;
  }
  if (EXT && S->evcnt) {
    unsigned long long *row = &S->evcnt[static_cast<size_t>(ev) * GV_NCOUNT];
    if (np) atomicAdd(&row[GV_C_PAIR], static_cast<unsigned long long>(np));
    if (na) atomicAdd(&row[GV_C_ANNIH], static_cast<unsigned long long>(na));
  }
  return r;
}

// ------------------------------------------------------------------ counters
// Counters of one warp: 16 words of shared memory that only this warp
// writes, lane c to counter c, so that booking takes no atomic (64-bit
// shared-memory atomics are compare-and-swap loops).
using WarpCnt = unsigned long long[16];

__device__ __forceinline__ void wcnt_add(unsigned long long *row, int c, unsigned v) {
  if ((threadIdx.x & 31) == static_cast<unsigned>(c)) row[c] += v;
}

// The step counters of one round.  All 32 lanes of a converged warp.
template <typename R>
__device__ __forceinline__ void count_round(unsigned long long *row, const Run<R> &r, int type, bool chose) {
  // steps, boundary-limited steps (at most 64 per lane) and process choices in one sum
  const unsigned sum = __reduce_add_sync(0xffffffffu, r.n_st | (r.n_geom << 12) | (chose ? 1u << 24 : 0u));
  const unsigned it = __reduce_max_sync(0xffffffffu, r.n_iter);
  const unsigned st = sum & 0xfffu;
  const unsigned by_type = __reduce_add_sync(0xffffffffu, type == 0 ? r.n_st : (type == 1 ? r.n_st << 16 : 0u));
  const unsigned wg = by_type & 0xffffu, we = by_type >> 16;
  const int lane = threadIdx.x & 31;
  unsigned v = 0;
  if (lane == GV_C_STEPS) v = st;
  if (lane == GV_C_STEPS_G) v = wg;
  if (lane == GV_C_STEPS_EM) v = we;
  if (lane == GV_C_STEPS_EP) v = st - wg - we;
  if (lane == GV_C_GEOM) v = (sum >> 12) & 0xfffu;
  if (lane == GV_C_DISCRETE) v = sum >> 24;
  if (lane == GV_C_LANE_SLOTS) v = 32u * it;  // idle-lane fraction
  if (v) row[lane] += v;
  if (__any_sync(0xffffffffu, r.note)) {
    const unsigned esc = __popc(__ballot_sync(0xffffffffu, r.note & kNoteEpEsc));
    const unsigned uns = __popc(__ballot_sync(0xffffffffu, r.note & kNoteUnscat));
    wcnt_add(row, GV_C_EP_ESC, esc);
    wcnt_add(row, GV_C_UNSCAT, uns);
  }
}

// ------------------------------------------------------------------ queues
__device__ __forceinline__ double i2d(unsigned long long v) { return __longlong_as_double(static_cast<long long>(v)); }
__device__ __forceinline__ unsigned long long d2i(double v) {
  return static_cast<unsigned long long>(__double_as_longlong(v));
}

// One track record read from or written to queue (par, type), see
// TrackLayout.
template <typename R>
__device__ __forceinline__ void load_track(const DevState<R> *S, int par, int type, unsigned slot, Trk<R> &t) {
  const unsigned char *b = S->qmem + static_cast<unsigned>(par * 3 + type) * S->q_bytes;
  const unsigned char *p = b + static_cast<unsigned long long>(slot) * 16u;
  const unsigned long long part = S->q_part;
  const double2 a = *reinterpret_cast<const double2 *>(p);
  const double2 c = *reinterpret_cast<const double2 *>(p + part);
  t.x = a.x; t.y = a.y;
  t.z = c.x; t.id = d2i(c.y);
  int sf;
  if constexpr (sizeof(R) == 4) {
    const float4 d = *reinterpret_cast<const float4 *>(p + 2 * part);
    const uint4 e = *reinterpret_cast<const uint4 *>(p + 3 * part);
    t.u = d.x; t.v = d.y; t.w = d.z; t.E = d.w;
    t.nlam = __uint_as_float(e.x); t.ev = e.y; t.step = e.z;
    sf = static_cast<int>(e.w);
  } else {
    const double2 d = *reinterpret_cast<const double2 *>(p + 2 * part);
    const double2 f = *reinterpret_cast<const double2 *>(p + 3 * part);
    const uint4 e = *reinterpret_cast<const uint4 *>(p + 4 * part);
    t.u = d.x; t.v = d.y; t.w = f.x; t.E = f.y;
    t.nlam = __hiloint2double(static_cast<int>(e.y), static_cast<int>(e.x));
    t.ev = e.z; t.step = e.w;
    sf = reinterpret_cast<const int *>(b + 5 * part)[slot];
  }
  t.sub = sf & 0xffff;
  t.flags = sf >> 16;
  t.type = type;
}

template <typename R>
__device__ __forceinline__ void store_track(const DevState<R> *S, int par, int type, unsigned slot, double x, double y,
                                            double z, R u, R v, R w, R E, R nlam, unsigned long long id, unsigned ev,
                                            unsigned step, int sf) {
  unsigned char *b = S->qmem + static_cast<unsigned>(par * 3 + type) * S->q_bytes;
  unsigned char *p = b + static_cast<unsigned long long>(slot) * 16u;
  const unsigned long long part = S->q_part;
  *reinterpret_cast<double2 *>(p) = make_double2(x, y);
  *reinterpret_cast<double2 *>(p + part) = make_double2(z, i2d(id));
  if constexpr (sizeof(R) == 4) {
    *reinterpret_cast<float4 *>(p + 2 * part) = make_float4(u, v, w, E);
    *reinterpret_cast<uint4 *>(p + 3 * part) = make_uint4(__float_as_uint(nlam), ev, step, static_cast<unsigned>(sf));
  } else {
    *reinterpret_cast<double2 *>(p + 2 * part) = make_double2(u, v);
    *reinterpret_cast<double2 *>(p + 3 * part) = make_double2(w, E);
    *reinterpret_cast<uint4 *>(p + 4 * part) =
        make_uint4(static_cast<unsigned>(__double2loint(nlam)), static_cast<unsigned>(__double2hiint(nlam)), ev, step);
    reinterpret_cast<int *>(b + 5 * part)[slot] = sf;
  }
}

// Warp-aggregated append.  A warp adds its lanes' records type by type to
// n[], each lane keeping its record's rank within its type, and then
// reserves the slots of all three types with one atomic instruction (lane q
// for type q): one round trip to L2, where a reservation per type took up to
// three in a row.  All 32 lanes of a converged warp.
struct WarpAppend {
  unsigned n[3] = {0, 0, 0};
  __device__ __forceinline__ unsigned add(bool has, int type) {
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    unsigned rank = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const unsigned m = __ballot_sync(0xffffffffu, has && type == q);
      if (type == q) rank = n[q] + __popc(m & lt);
      n[q] += __popc(m);
    }
    return rank;
  }
  // lane q: the first slot of type q; read with slot()
  __device__ __forceinline__ unsigned reserve(FillSlot *fill) const {
    const int lane = threadIdx.x & 31;
    const unsigned mine = lane == 0 ? n[0] : (lane == 1 ? n[1] : (lane == 2 ? n[2] : 0u));
    return mine ? atomicAdd(&fill[lane].n, mine) : 0u;
  }
  __device__ __forceinline__ static unsigned slot(unsigned base, int type, unsigned rank) {
    return __shfl_sync(0xffffffffu, base, type) + rank;
  }
};

// The parent of a step's secondaries: where they start and whose lineage
// names them.
struct Parent {
  double x, y, z;
  unsigned long long id;
  unsigned ev;
  int sub;
};

// The block's secondary stack in shared memory (the StackBuffer of Sec.
// 2.1.2 for one block): its lanes take the secondaries up in a later round of
// the same claim instead of leaving them to the next generation.  Stored like
// the queues, in 16-byte parts: {x, y} {z, id} {u, v, w, E} {event, sub,
// type, -}.  Photons lie from the bottom up and charged tracks from the top
// down, so that a warp can take one kind: in a mixed warp the two kinds' steps
// run one after the other.  With a key's requests kept to warps of their own
// (step_kernel) this took one 10 GeV shower from 861 to 733 us, 1000 x 1 GeV
// from 1.00 to 0.91 ms and 300 x 10 GeV in FP64 from 10.5 to 9.0 ms.
struct StackCount {
  unsigned used;      // photons | charged tracks << 16; appends reserve here
  unsigned taken[2];  // photons and charged tracks taken since the last appends
  // between the takes of one round and its appends (one thread)
  __device__ __forceinline__ void settle() {
    const unsigned g = used & 0xffffu, q = used >> 16;
    used = (g - min(taken[0], g)) | (q - min(taken[1], q)) << 16;
    taken[0] = taken[1] = 0u;
  }
};
template <typename R> struct LocalStack {
  unsigned char *e;
  StackCount *count;
  int cap;
  static constexpr int kBytes = 48 + 4 * sizeof(R);  // per entry
  __device__ __forceinline__ int place(int charged, unsigned i) const {
    return charged ? cap - 1 - static_cast<int>(i) : static_cast<int>(i);
  }
  // The lanes of `idle` take entries of one kind; true for those that got
  // one.  All 32 lanes of a converged warp.
  __device__ __forceinline__ bool take(unsigned idle, int charged, Trk<R> &t) const {
    const int lane = threadIdx.x & 31;
    const unsigned n = charged ? count->used >> 16 : count->used & 0xffffu;
    if (!idle || !n) return false;
    unsigned k = 0;
    if (lane == 0) k = atomicAdd(&count->taken[charged], static_cast<unsigned>(__popc(idle)));
    k = __shfl_sync(0xffffffffu, k, 0) + __popc(idle & ((1u << lane) - 1u));
    if (!(idle >> lane & 1u) || k >= n) return false;
    get(place(charged, n - 1u - k), t);
    return true;
  }
  __device__ __forceinline__ void put(int i, const Parent &p, unsigned long long id, const R *d, R E, int type) const {
    reinterpret_cast<double2 *>(e)[i] = make_double2(p.x, p.y);
    reinterpret_cast<double2 *>(e + 16 * cap)[i] = make_double2(p.z, i2d(id));
    reinterpret_cast<uint4 *>(e + 32 * cap)[i] = make_uint4(p.ev, static_cast<unsigned>(p.sub), static_cast<unsigned>(type), 0u);
    reinterpret_cast<V4<R> *>(e + 48 * cap)[i] = V4<R>{d[0], d[1], d[2], E};
  }
  __device__ __forceinline__ void get(int i, Trk<R> &t) const {
    const double2 a = reinterpret_cast<const double2 *>(e)[i];
    const double2 c = reinterpret_cast<const double2 *>(e + 16 * cap)[i];
    const uint4 g = reinterpret_cast<const uint4 *>(e + 32 * cap)[i];
    const V4<R> d = reinterpret_cast<const V4<R> *>(e + 48 * cap)[i];
    t.x = a.x; t.y = a.y; t.z = c.x;
    t.id = d2i(c.y);
    t.u = d.x; t.v = d.y; t.w = d.z; t.E = d.w;
    t.nlam = R(-1);
    t.ev = g.x;
    t.step = 0;
    t.sub = static_cast<int>(g.y);
    t.type = static_cast<int>(g.z);
    t.flags = 0;
  }
};

// A lane's running count in a warp: the sum over its own and the lower lanes.
__device__ __forceinline__ unsigned lane_sum(unsigned v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// The ids of a final state's secondaries are words of counter blocks of its
// step (ids: the first two's), so they name each one's index in its parent's
// list, and where it goes changes no result.
template <typename R>
__device__ __forceinline__ unsigned long long kid_id(const DevState<R> *S, const Parent &p, uint32_t kk, const uint4 &ids, int j) {
  uint32_t lo = j ? ids.z : ids.x, hi = j ? ids.w : ids.y;
  if (j == 2) {
    const uint4 b = track_draw(S, p.id, p.ev, kk, kTagId + 1u);
    lo = b.x; hi = b.y;
  }
  return static_cast<unsigned long long>(lo) | (static_cast<unsigned long long>(hi) << 32);
}

// Put the secondaries of a warp's final states on the block's stack while it
// has room.  Returns how many of the lane's the stack took; what it refuses
// leaves it exactly full, so that no later reservation of the round finds
// room.  All 32 lanes of a converged warp.
template <typename R, bool EXT = true>
__device__ __forceinline__ int stack_kids(const DevState<R> *S, const LocalStack<R> &ls, const Parent &p, const Kids<R> &kids,
                                          uint32_t kk, const uint4 &ids, unsigned long long *row) {
  if (!__any_sync(0xffffffffu, kids.n > 0)) return 0;
  const int lane = threadIdx.x & 31;
  // photons | charged tracks << 16: the lane's, up to it, and the warp's
  unsigned mine = 0u;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (j < kids.n) mine += kids.type[j] == 0 ? 1u : 1u << 16;
  const unsigned incl = lane_sum(mine);
  const unsigned all = __shfl_sync(0xffffffffu, incl, 31);
  unsigned used = 0;
  if (lane == 0) used = atomicAdd(&ls.count->used, all);
  used = __shfl_sync(0xffffffffu, used, 0);
  const int free = ls.cap - static_cast<int>((used & 0xffffu) + (used >> 16));
  const unsigned before = incl - mine;
  const int room = max(0, min(free - static_cast<int>((before & 0xffffu) + (before >> 16)), kids.n));
  unsigned at = used + before, made = 0u;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j >= room) break;
    const int charged = kids.type[j] != 0;
    ls.put(ls.place(charged, charged ? at >> 16 : at & 0xffffu), p, kid_id(S, p, kk, ids, j), kids.d[j], kids.E[j],
           kids.type[j]);
    at += charged ? 1u << 16 : 1u;
    made += 1u << 8 * kids.type[j];
    if (EXT && S->evcnt) atomicAdd(&S->evcnt[static_cast<size_t>(p.ev) * GV_NCOUNT + GV_C_TRK_G + kids.type[j]], 1ull);
  }
  if (static_cast<int>((all & 0xffffu) + (all >> 16)) > free) {  // uniform: take back what did not fit
    const unsigned back = __reduce_add_sync(0xffffffffu, used + incl - at);
    if (lane == 0) atomicSub(&ls.count->used, back);
  }
  made = __reduce_add_sync(0xffffffffu, made);
  if (lane >= GV_C_TRK_G && lane < GV_C_TRK_G + 3) row[lane] += made >> 8 * (lane - GV_C_TRK_G) & 0xffu;
  return room;
}

// The end of a claim: the secondaries of the final states the warp ran, from
// `first` on (the block's stack took the others; t's are its own), and its
// lanes' survivors, appended with one reservation: a trip to L2 less per
// claim, and the block does not wait at the results barrier for the warps that
// append secondaries (2000 x 10 GeV: 4.16 -> 3.99 ms).  What bounds it is its
// length: a warp comes here once per claim and fetches most of the
// instructions anew (ballots and ranks record by record took 3500 cycles of a
// claim's 19000, unloaded as well).  So one sum over the lanes, of the records
// of each type a byte each, gives all ranks and counts, and every round's
// appends share this site: the kernel 110 -> 104 KB, 3.99 -> 3.88 ms, 4096
// mixed 10.88 -> 10.62 ms, 1000 x 1 GeV 720 -> 704 us.  All 32 lanes of a
// converged warp.
template <typename R, bool EXT = true>
__device__ __forceinline__ void push_all(const DevState<R> *S, int out, const Parent &p, const Kids<R> &kids, int first,
                                         const uint4 &ids, uint32_t kk, const Trk<R> &t, bool alive,
                                         unsigned long long *row) {
  const int lane = threadIdx.x & 31;
  // the lane's records per type, a byte each (a warp has 128 at most)
  unsigned made = 0u;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (j >= first && j < kids.n) made += 1u << 8 * kids.type[j];
  const unsigned mine = made + (alive ? 1u << 8 * t.type : 0u);
  unsigned at = lane_sum(mine);
  const unsigned all = __shfl_sync(0xffffffffu, at, 31);
  const unsigned n = lane < 3 ? all >> 8 * lane & 0xffu : 0u;
  const unsigned base = n ? atomicAdd(&S->ctl->cnt[out][lane].n, n) : 0u;
  made = __reduce_add_sync(0xffffffffu, made);
  if (lane >= GV_C_TRK_G && lane < GV_C_TRK_G + 3) row[lane] += made >> 8 * (lane - GV_C_TRK_G) & 0xffu;
  if (EXT && S->evcnt) {
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (j >= first && j < kids.n)
        atomicAdd(&S->evcnt[static_cast<size_t>(p.ev) * GV_NCOUNT + GV_C_TRK_G + kids.type[j]], 1ull);
  }
  at -= mine;
  const unsigned b0 = __shfl_sync(0xffffffffu, base, 0), b1 = __shfl_sync(0xffffffffu, base, 1),
                 b2 = __shfl_sync(0xffffffffu, base, 2);
  bool full = false;
  const auto place = [&](int type) {
    const unsigned slot = (type == 0 ? b0 : (type == 1 ? b1 : b2)) + (at >> 8 * type & 0xffu);
    at += 1u << 8 * type;
    return slot;
  };
  if (alive) {
    const unsigned slot = place(t.type);
    if (slot < S->capacity)
      store_track<R>(S, out, t.type, slot, t.x, t.y, t.z, t.u, t.v, t.w, t.E, t.nlam, t.id, t.ev, t.step,
                     t.sub | (t.flags << 16));
    else full = true;
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j < first || j >= kids.n) continue;
    const unsigned slot = place(kids.type[j]);
    if (slot < S->capacity)
      store_track<R>(S, out, kids.type[j], slot, p.x, p.y, p.z, kids.d[j][0], kids.d[j][1], kids.d[j][2], kids.E[j], R(-1),
                     kid_id(S, p, kk, ids, j), p.ev, 0u, p.sub);
    else full = true;
  }
  if (full) set_status(S->ctl, GV_ERR_STACK_FULL);
}

// PostStepActions: append the step's secondaries to the output queues.
// Called by all 32 lanes of a converged warp (lanes without secondaries pass
// kids.n == 0).
template <typename R, bool EXT = true>
__device__ __forceinline__ void push_kids(const DevState<R> *S, int out, const Parent &t, const Kids<R> &kids,
                                          uint32_t kk, const uint4 &ids, unsigned long long *row) {
  if (!__any_sync(0xffffffffu, kids.n > 0)) return;
  Trk<R> none;
  none.type = 0;
  push_all<R, EXT>(S, out, t, kids, 0, ids, kk, none, false, row);
}

// Survivors: one record per lane (has: whether it has one).  All 32 lanes of
// a converged warp.
template <typename R>
__device__ __forceinline__ void push_track(const DevState<R> *S, int out, const Trk<R> &t, bool has) {
  if (!__any_sync(0xffffffffu, has)) return;
  WarpAppend ap;
  const unsigned rank = ap.add(has, t.type);
  const unsigned slot = WarpAppend::slot(ap.reserve(S->ctl->cnt[out]), has ? t.type : 0, rank);
  if (!has) return;
  if (slot >= S->capacity) {
    set_status(S->ctl, GV_ERR_STACK_FULL);
    return;
  }
  store_track<R>(S, out, t.type, slot, t.x, t.y, t.z, t.u, t.v, t.w, t.E, t.nlam, t.id, t.ev, t.step,
                 t.sub | (t.flags << 16));
}

// The automatic events-in-flight cap (the paper keeps a bounded number of
// events in flight, Sec. 2.1.1): a primary of energy E is budgeted 0.15
// live tracks per MeV (about 2.3 times the peak live-track count of a
// shower per MeV) plus 64, and new primaries are admitted while the budgets
// of the events in flight fit the queue capacity.  NaN or negative energies
// get the base budget.
__device__ __forceinline__ unsigned long long prim_cost(double E) {
  const double e = (E > 0.0 && E < 1e12) ? E : 0.0;
  return 64ull + static_cast<unsigned long long>(ceil(0.15 * e));
}

// An event's last track ended: the event leaves the set in flight and
// returns its budget.  Out of line: it runs once per event, and inlined at
// both of its call sites it slowed the step kernel by 0.5 %.
template <typename R> __device__ __noinline__ void event_closed(const DevState<R> *S, unsigned ev) {
  atomicAdd(&S->ctl->ev_done, 1u);
  if (S->evcost) atomicAdd(&S->ctl->cost_done, atomicExch(&S->evcost[ev], 0ull));
}

// A primary was loaded: its budget goes to its event (returned when the
// event closes), or straight back if it never entered the box.
template <typename R>
__device__ __forceinline__ void primary_cost(const DevState<R> *S, unsigned ev, double E, bool entered) {
  if (!S->evcost) return;
  if (entered) atomicAdd(&S->evcost[ev], prim_cost(E));
  else atomicAdd(&S->ctl->cost_done, prim_cost(E));
}

// Live tracks of an event, counted while primaries still wait on the
// in-flight cap (Ctl::book; once the last primary is out nobody asks).  A
// final state books its secondaries and its parent's end as one change, so a
// photoelectric absorption needs no atomic and the event never looks empty
// in between.  Returns the count before a change by -1, which is 1 where
// that closed the event (event_closed); 0 for other changes.
template <typename R> __device__ __forceinline__ unsigned book_live(const DevState<R> *S, unsigned ev, int change) {
  if (change < 0) return atomicSub(&S->evlive[ev], 1u);
  if (change > 0) atomicAdd(&S->evlive[ev], static_cast<unsigned>(change));
  return 0u;
}

// Interaction requests staged in shared memory by the in-block basketizer,
// one slot per thread, in parts like the queues (each access is then free of
// bank conflicts): {x, y} {z, id} {E, direction} {event, step, sub, key}
// {u2, u3} and the final state's return code.
template <typename R> struct ReqStore {
  unsigned char *m;
  int n;  // slots
  static constexpr int kBytes = 48 + 6 * static_cast<int>(sizeof(R)) + 4;  // per slot
  __device__ __forceinline__ double2 &xy(int i) const { return reinterpret_cast<double2 *>(m)[i]; }
  __device__ __forceinline__ double2 &zi(int i) const { return reinterpret_cast<double2 *>(m + 16 * n)[i]; }
  __device__ __forceinline__ uint4 &info(int i) const { return reinterpret_cast<uint4 *>(m + 32 * n)[i]; }
  __device__ __forceinline__ V4<R> &dir(int i) const { return reinterpret_cast<V4<R> *>(m + 48 * n)[i]; }
  __device__ __forceinline__ R &u2(int i) const { return reinterpret_cast<R *>(m + (48 + 4 * sizeof(R)) * n)[i]; }
  __device__ __forceinline__ R &u3(int i) const { return reinterpret_cast<R *>(m + (48 + 5 * sizeof(R)) * n)[i]; }
  __device__ __forceinline__ int &ret(int i) const { return reinterpret_cast<int *>(m + (48 + 6 * sizeof(R)) * n)[i]; }
};
constexpr int kNKey = kNReqKey;

// A primary handed to lane `idx` of the generation: its track, or false if
// it never entered the box.  Counts per event type by type are left to the
// caller's warp.
template <typename R, bool EXT>
__device__ __forceinline__ bool load_primary(const View<R> &V, const DevState<R> *S, unsigned i, bool book, Trk<R> &t,
                                             int &note) {
  Ctl *ctl = S->ctl;
  const unsigned pi = S->order ? S->order[i] : i;
  gv_primary p = S->prim[pi];
  const double e_in = p.E_MeV;  // the budget of the automatic cap is the caller's energy
  p.event -= S->ev_base;        // the tallies' row (events below the range wrap to a large value)
  if (p.type < 0 || p.type > 2 || p.event >= S->n_events) {  // caller's device array: check here
    set_status(ctl, GV_ERR_BAD_ARG);
    p.type = 0;
    p.event = 0;
    p.z = -1.0;
    p.E_MeV = 0.0;
  }
  t.type = p.type;
  t.E = static_cast<R>(p.E_MeV);
  t.x = p.x; t.y = p.y; t.z = p.z;
  t.u = static_cast<R>(p.u); t.v = static_cast<R>(p.v); t.w = static_cast<R>(p.w);
  t.nlam = R(-1);
  t.id = p.id;
  t.ev = p.event;
  t.step = 0;
  t.flags = kFlagPrimary;
  t.sub = locate(V.zb, V.geo.nsub, p.z, p.w);
  const bool in = t.sub >= 0;
  if (EXT && S->evcnt) {
    unsigned long long *row = &S->evcnt[static_cast<size_t>(t.ev) * GV_NCOUNT];
    atomicAdd(&row[GV_C_TRK_G + t.type], 1ull);
    if (!in && t.type == 2) atomicAdd(&row[GV_C_EP_ESC], 1ull);
  }
  if (!in) {
    atomicAdd(&S->escape[t.ev], p.E_MeV);
    if (t.type == 2) note |= kNoteEpEsc;
  }
  if (book) {
    primary_cost(S, t.ev, e_in, in);
    if (in && atomicAdd(&S->evlive[t.ev], 1u) == 0u) atomicAdd(&ctl->ev_started, 1u);
  }
  return in;
}

// Tracks (and escaped positrons) that a warp's primaries add to the counters.
__device__ __forceinline__ void count_primaries(unsigned long long *row, bool has, int type, int note) {
#pragma unroll
  for (int q = 0; q < 3; ++q) wcnt_add(row, GV_C_TRK_G + q, __popc(__ballot_sync(0xffffffffu, has && type == q)));
  wcnt_add(row, GV_C_EP_ESC, __popc(__ballot_sync(0xffffffffu, has && (note & kNoteEpEsc))));
}

// Stage the tables, planes, sub-slab records, 1/E_i and materials into
// shared memory, with a view of them.  Two block barriers inside.
template <typename R> __device__ __forceinline__ void stage_tables(const DevState<R> *S, unsigned char *smem, View<R> &sV) {
  const unsigned tid = threadIdx.x, nt = blockDim.x;
  const uint4 *src = reinterpret_cast<const uint4 *>(S->view.xs);
  uint4 *dst = reinterpret_cast<uint4 *>(smem);
  for (unsigned i = tid; i < S->xs_bytes / 16; i += nt) dst[i] = src[i];
  const double *zsrc = S->view.zb;
  double *zdst = reinterpret_cast<double *>(smem + S->xs_bytes);
  SubRec<R> *rdst = reinterpret_cast<SubRec<R> *>(smem + S->rec_off);
  const unsigned ns = static_cast<unsigned>(S->view.geo.nsub);
  for (unsigned i = tid; i <= ns; i += nt) zdst[i] = zsrc[i];
  for (unsigned i = tid; i < ns; i += nt) {
    rdst[i].thick = static_cast<R>(zsrc[i + 1] - zsrc[i]);
    rdst[i].row = S->view.smat[i] * (3 * kGridN);
  }
  float *idst = reinterpret_cast<float *>(smem + S->xs_bytes + S->zb_bytes);
  for (unsigned i = tid; i < kGridN; i += nt) idst[i] = S->view.inv_node[i];
  unsigned char *mdst = smem + S->xs_bytes + S->zb_bytes + kInvNodeBytes;
  for (unsigned i = tid; i < ns; i += nt) mdst[i] = S->view.smat[i];
  const uint4 *ssrc = reinterpret_cast<const uint4 *>(S->view.smax);
  uint4 *sdst = reinterpret_cast<uint4 *>(smem + S->smax_off);
  for (unsigned i = tid; i < S->smax_bytes / 16; i += nt) sdst[i] = ssrc[i];
  // the view word by word (one thread copying it was a chain of ~200 loads)
  static_assert(sizeof(View<R>) % 4 == 0, "copied in words");
  for (unsigned i = tid; i < sizeof(View<R>) / 4; i += nt)
    reinterpret_cast<unsigned *>(&sV)[i] = reinterpret_cast<const unsigned *>(&S->view)[i];
  __syncthreads();
  if (tid == 0) {
    sV.xs = reinterpret_cast<const V4<R> *>(smem);
    sV.zb = zdst;
    sV.inv_node = idst;
    sV.smat = mdst;
    if (S->smax_bytes) sV.smax = reinterpret_cast<const R *>(smem + S->smax_off);
  }
  __syncthreads();
}

// ------------------------------------------------------------------ planning
// The order in which a generation's chunks are claimed: positrons, electrons,
// photons, then new primaries.  Charged-particle claims take longest (loss,
// more interactions per step), so they go first and the last claims of a
// generation, whose spread leaves blocks idle at its end, are the short
// photon ones (measured: 4 % less transport time than photons first).
__device__ __forceinline__ int claim_queue(int seg) { return seg < 3 ? 2 - seg : 3; }

// The plan of the next generation.  One thread runs it between generations,
// on instructions that no block has fetched before: without 64-bit divisions
// and the counters that this kind of kernel does not use, and with one sum per
// round for the steps by type (count_round), 1000 x 1 GeV took 687 instead of
// 697 us.
template <typename R> __device__ void plan_next(const DevState<R> *S, int pn) {
  Ctl *c = S->ctl;
  // everything the plan depends on, in one round trip
  const unsigned cap = static_cast<unsigned>(S->capacity);
  const unsigned n0 = c->cnt[pn][0].n, n1 = c->cnt[pn][1].n, n2 = c->cnt[pn][2].n;
  const unsigned next = c->prim_next, max_in_flight = c->max_in_flight;
  const unsigned ev_started = c->ev_started, ev_done = c->ev_done;
  unsigned long long cost_started = c->cost_started, cost_done = c->cost_done;
  const unsigned long long live_peak = c->live_peak;
  unsigned long long gen = c->gen;
  int status = c->status;
  const unsigned long long live = static_cast<unsigned long long>(n0) + n1 + n2;
  const unsigned rem = S->n_prim - next;
  unsigned inj = 0;
  if (status == 0 && rem > 0) {
    if (S->mode == GV_ONE_EVENT_PER_LAUNCH) {
      if (live == 0) {
        const unsigned first = S->order ? S->order[next] : next;
        const unsigned ev = S->prim[first].event;
        while (inj < rem) {
          const unsigned i = next + inj;
          const unsigned pi = S->order ? S->order[i] : i;
          if (S->prim[pi].event != ev) break;
          ++inj;
        }
      }
    } else if (live < S->low_water || live == 0) {
      inj = rem < S->batch ? rem : static_cast<unsigned>(S->batch);
      if (max_in_flight) {  // events in flight (Sec. 2.1.1): started and not yet finished
        const unsigned fl = ev_started - ev_done;
        const unsigned room = max_in_flight > fl ? max_in_flight - fl : 0u;
        inj = inj < room ? inj : room;
      }
      if (S->pcost && inj > 0) {  // automatic cap: the budgets of the events in flight fit the capacity
        if (live == 0) c->cost_done = cost_done = cost_started;  // nothing alive: every event has closed
        const unsigned long long held = cost_started > cost_done ? cost_started - cost_done : 0ull;
        const unsigned long long room = S->capacity > held ? S->capacity - held : 0ull;
        const unsigned long long *pc = S->pcost + next;
        const unsigned long long base = pc[0];
        if (pc[inj] - base > room) {  // the longest run of the next primaries that fits
          unsigned lo = 0, hi = inj;  // budget(lo) <= room < budget(hi)
          while (hi - lo > 1) {
            const unsigned mid = lo + (hi - lo) / 2;
            if (pc[mid] - base <= room) lo = mid;
            else hi = mid;
          }
          inj = lo;
        }
        if (inj == 0 && live == 0) inj = 1;  // one primary at least when nothing is alive
        c->cost_started = cost_started + (pc[inj] - base);
      }
    }
  }
  const unsigned long long tot = live + inj;
  const bool last = next + inj == S->n_prim;
  Plan p;
  p.prim_begin = next;
  p.prim_count = inj;
  c->prim_next = next + inj;
  // the events' live tracks are asked for only by the in-flight cap, and that
  // only while primaries wait
  p.book = S->mode == GV_BATCHED && !last && (max_in_flight || S->pcost);
  unsigned B = static_cast<unsigned>(S->chunk);
  // With fewer live tracks than the grid has lanes (the first generations of
  // a shower and its tail), a block claims fewer tracks (a multiple of 32)
  // so that every block gets some: each block's rounds are then short, with
  // fewer warps to wait for at its barriers and its idle lanes left to the
  // secondaries of its block stack.
  if (S->adaptive_chunk) {
    if (tot < static_cast<unsigned long long>(B) * static_cast<unsigned>(S->grid)) {  // (32 bits: a 64-bit division is a call)
      const unsigned g = static_cast<unsigned>(S->grid), per = (static_cast<unsigned>(tot) + g - 1) / g;
      if (per < B) B = per <= 32 ? 32u : (per + 31) / 32 * 32;
    }
  }
  p.B = B;
  p.end[0] = (n2 + B - 1) / B;  // segments in claim_queue order
  p.end[1] = p.end[0] + (n1 + B - 1) / B;
  p.end[2] = p.end[1] + (n0 + B - 1) / B;
  p.end[3] = p.end[2] + (inj + B - 1) / B;
  p.n_in[0] = min(n0, cap);
  p.n_in[1] = min(n1, cap);
  p.n_in[2] = min(n2, cap);
  // long claims (K_tail rounds) once every primary is injected and few
  // tracks are live: in the tail, and at the start of a batch injected at
  // once, where the block stack keeps a claim's secondaries stepping in the
  // block (one-round claims there measured slower on small batches)
  p.K = (last && tot < S->tail_threshold) ? S->K_tail : S->K_bulk;
  for (int q = 0; q < 3; ++q) c->cnt[pn ^ 1][q].n = 0;
  c->claim.n = 0;
  c->blocks_done = 0;
  if (S->chunk == 32) {  // warps claim (blocks have 64 threads or more)
#pragma unroll 1
    for (int r = 0; r < kNClaim; ++r) c->claims[r].n = 0;
  }
  if (S->pipeline) {
    c->req_n = 0;
#pragma unroll 1
    for (int k = 0; k < kNReqKey; ++k) c->key_n[k] = 0;
    c->claim_b = 0;
    c->blocks_done_b = 0;
  }
  if (tot > live_peak) c->live_peak = tot;
  if (tot > 0) c->gen = ++gen;
  if (gen > S->max_gen && status == 0) c->status = status = GV_ERR_TIMEOUT;
  p.done = (status != 0) || (tot == 0 && last);
  if (p.done) p.end[0] = p.end[1] = p.end[2] = p.end[3] = 0;
  p.pad[0] = p.pad[1] = p.pad[2] = 0;
  c->plan = p;
}

// The control block of a transport that starts, and the plan of its first
// generation.
template <typename R> __device__ void start_control(const DevState<R> *S) {
  Ctl *c = S->ctl;
  for (int i = 0; i < 2; ++i)
    for (int q = 0; q < 3; ++q) c->cnt[i][q].n = 0;
  c->prim_next = 0;
  c->status = 0;
  c->plan.done = 0;
  c->gen = 0;
  c->loop_iter = 0;
  c->live_peak = 0;
  c->ev_started = 0;
  c->ev_done = 0;
  c->cost_started = 0;
  c->cost_done = 0;
  if (S->max_in_flight >= 0) {
    c->max_in_flight = static_cast<unsigned>(S->max_in_flight);
  } else if (S->pcost) {  // automatic, per event: the budgets of prim_cost (plan_next)
    c->max_in_flight = 0;
  } else {  // automatic, every event budgeted like the most energetic primary:
            // ~0.065 live tracks per MeV at the peak of a shower, x2.3
    const double emax = static_cast<double>(__uint_as_float(c->emax_bits));
    const double cap = static_cast<double>(S->capacity) / (0.15 * emax + 64.0);
    c->max_in_flight = static_cast<unsigned>(cap < 16.0 ? 16.0 : (cap > 1e9 ? 1e9 : cap));
  }
  for (int i = 0; i < 16; ++i) c->counters[i] = 0;
  plan_next(S, 0);
}

template <typename R> __global__ void init_kernel(const DevState<R> *S) { start_control(S); }

// What a transport needs before its first generation, in two launches: the
// first stores the state record (its argument), clears the tallies and event
// counts and sums the budgets of each scan block's primaries, the second
// turns those into prefix sums (pcost[i] = sum of prim_cost over primaries 0
// .. i-1, for the automatic events-in-flight cap) and starts the control
// block.  One block scanning all primaries after a copy and up to seven
// memsets took 300 us for 1e5 photons, half of a 600 us transport (300 us
// now, of which the step kernels take 230); one shower takes 10 us less.
constexpr int kPrepThreads = 256;
constexpr int kScanBlocks = 304;  // scan blocks at most: two per SM
struct Clear {
  unsigned long long *p[6];  // 8-byte words to zero
  unsigned long long n[6];
  int count;
  void add(void *q, size_t bytes) {
    p[count] = static_cast<unsigned long long *>(q);
    n[count++] = bytes / 8;
  }
};

__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long *s_warp) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();  // s_warp may still be read
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long sum = 0ull;
  for (int w = 0; w < kPrepThreads / 32; ++w) sum += s_warp[w];
  return sum;
}

// the primaries of scan block b
__device__ __forceinline__ void scan_range(unsigned n, unsigned blocks, unsigned b, unsigned &lo, unsigned &hi) {
  const unsigned per = n / blocks + (n % blocks != 0);
  const unsigned long long l = static_cast<unsigned long long>(b) * per;
  lo = l < n ? static_cast<unsigned>(l) : n;
  hi = n - lo < per ? n : lo + per;
}

template <typename R>
__global__ void __launch_bounds__(kPrepThreads)
    prep_kernel(const __grid_constant__ DevState<R> s, DevState<R> *dst, const __grid_constant__ Clear clear,
                unsigned long long *part, unsigned scan_blocks) {
  __shared__ unsigned long long s_warp[kPrepThreads / 32];
  if (blockIdx.x == 0) {
    static_assert(sizeof(DevState<R>) % 4 == 0, "stored in words");
    for (unsigned i = threadIdx.x; i < sizeof(DevState<R>) / 4; i += kPrepThreads)
      reinterpret_cast<unsigned *>(dst)[i] = reinterpret_cast<const unsigned *>(&s)[i];
    if (threadIdx.x == 0) part[kScanBlocks] = 0ull;  // scan blocks done
  }
  const unsigned long long stride = static_cast<unsigned long long>(gridDim.x) * kPrepThreads;
  for (int k = 0; k < clear.count; ++k)
    for (unsigned long long i = static_cast<unsigned long long>(blockIdx.x) * kPrepThreads + threadIdx.x; i < clear.n[k]; i += stride)
      clear.p[k][i] = 0ull;
  if (blockIdx.x >= scan_blocks) return;
  unsigned lo, hi;
  scan_range(s.n_prim, scan_blocks, blockIdx.x, lo, hi);
  unsigned long long sum = 0ull;
  for (unsigned i = lo + threadIdx.x; i < hi; i += kPrepThreads) sum += prim_cost(s.prim[i].E_MeV);
  sum = block_sum(sum, s_warp);
  if (threadIdx.x == 0) part[blockIdx.x] = sum;
}

template <typename R>
__global__ void __launch_bounds__(kPrepThreads)
    start_kernel(const DevState<R> *S, unsigned long long *pcost, unsigned long long *part, unsigned scan_blocks) {
  __shared__ unsigned long long s_warp[kPrepThreads / 32];
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long base = 0ull;
  for (unsigned b = tid; b < blockIdx.x; b += kPrepThreads) base += part[b];
  base = block_sum(base, s_warp);
  unsigned lo, hi;
  scan_range(S->n_prim, scan_blocks, blockIdx.x, lo, hi);
  if (blockIdx.x == 0 && tid == 0) pcost[0] = 0ull;
  for (unsigned t = lo; t < hi; t += min(hi - t, static_cast<unsigned>(kPrepThreads))) {
    const bool has = hi - t > static_cast<unsigned>(tid);
    unsigned long long incl = has ? prim_cost(S->prim[t + tid].E_MeV) : 0ull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    __syncthreads();  // s_warp may still be read
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    unsigned long long before = 0ull, all = 0ull;
    for (int w = 0; w < kPrepThreads / 32; ++w) {
      if (w < warp) before += s_warp[w];
      all += s_warp[w];
    }
    if (has) pcost[static_cast<unsigned long long>(t) + tid + 1u] = base + before + incl;
    base += all;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&part[kScanBlocks], 1ull) == gridDim.x - 1;
  __syncthreads();
  if (s_last && tid == 0) {
    __threadfence();
    start_control(S);
  }
}

// largest primary energy, for the automatic events-in-flight cap of the
// allocation-free entry point
template <typename R> __global__ void prim_emax_kernel(const DevState<R> *S) {
  float m = 0.0f;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < S->n_prim; i += gridDim.x * blockDim.x) {
    const float e = static_cast<float>(S->prim[i].E_MeV);
    m = e > m ? e : m;  // NaN and negative energies leave m unchanged
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.0f) atomicMax(&S->ctl->emax_bits, __float_as_uint(m));
}

// ------------------------------------------------------------------ the transport's state
// The step kernels read the transport's state record (queue and tally
// pointers, seeds, switches) from a constant-memory copy, one per precision
// and GPU: its fields are then instruction operands, which costs no load and
// no register on the step path (2.7 % of the benchmark's kernel time against
// the same record read through a global pointer).  The host fills the copy
// on the transport's stream from the record in device memory; transports of
// different contexts on one GPU take turns on it (StateSlot).  The split
// pipeline's kernels read the device-memory record through their pointer:
// with them on the constant copy as well, the fused step kernel measured
// 1.1 % slower.
__constant__ DevState<float> c_state_f;
__constant__ DevState<double> c_state_d;
template <typename R> __device__ __forceinline__ const DevState<R> *tstate();

// Whether the calling thread's block is the last of the grid to finish; what
// every block wrote before is then visible to it (each block's other threads
// reach the counter through a block barrier).
__device__ __forceinline__ bool block_done(unsigned *counter) {
  unsigned before;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(counter) : "memory");
  return before == gridDim.x - 1;
}
template <> __device__ __forceinline__ const DevState<float> *tstate<float>() { return &c_state_f; }
template <> __device__ __forceinline__ const DevState<double> *tstate<double>() { return &c_state_d; }

// ------------------------------------------------------------------ the kernel
// Register budget: GV_MIN_BLOCKS resident 256-thread blocks per SM in FP32
// (measured: with the along-step loop 2 blocks at up to 128 registers beat
// 3 blocks at 80 registers, which spill 400 bytes: 14.9 ms against 13.3 on
// the mixed-type batch).  FP64 runs one block per SM without a register cap
// (192 to 240 registers, no spills; 4 % faster than two blocks at 128
// registers, which spilled).
// GV_MAX_BLOCK is the largest block the kernels are compiled for.
#ifndef GV_MIN_BLOCKS
#define GV_MIN_BLOCKS 2
#endif
#ifndef GV_MAX_BLOCK
#define GV_MAX_BLOCK 256
#endif

#ifdef GV_MAXNREG
#define GV_STEP_BOUNDS __maxnreg__(GV_MAXNREG)
#else
#define GV_STEP_BOUNDS __launch_bounds__(GV_MAX_BLOCK, sizeof(R) == 4 ? GV_MIN_BLOCKS : 1)
#endif

// What bounds it: the dependent chains of a round at the two blocks per SM
// that its registers allow, and at a block's barriers its slowest warp.  At
// the shower maximum (ncu, 500 x 10 GeV) a scheduler issues in 34 % of its
// cycles; per issue 2.4 warps wait for L2, 2.1 for a fixed-latency result, 1.9
// for shared memory, 1.8 at a barrier and 0.7 for instructions; ALU 26 %, FP64
// pipe 15 %, FMA 13 %, L2 7 %, DRAM 4 % of their peaks.
// FP64 kernels sit on the FP64 pipe (69 % at the maximum).  So the chains are
// short and work is done where many lanes do it: random numbers once per round
// instead of once per step (run_round), one place that makes secondaries (a
// stopped positron is a request like any other), counters booked by ballots
// into words of the warp (a 64-bit shared-memory atomic is a loop), 16-byte
// track parts, one reservation atomic for the three queues, a warp to a model
// (the sort below), a generation's plan in one read; and the code is kept
// small, because a warp fetches what it runs once per claim anew: the same
// kernel with 12 KB more of it lost 5 % on the small transports.  What a caller
// waits for, before these and with them: 2000 x 10 GeV e- in Pb/polystyrene
// 7.69 -> 3.80 ms, 1000 x 1 GeV 1.41 -> 0.70 ms, one 10 GeV shower 1.20 -> 0.59
// ms, 300 x 10 GeV in FP64 13.3 -> 8.5 ms, 2000 x 100 GeV in W/Si with cells
// 95.4 -> 52.3 ms.
template <typename R, bool SORT, bool MERGE, bool FIELD, bool OPTS, bool EXT, bool ALT = !SORT>
__global__ void GV_STEP_BOUNDS
    step_kernel(int parity) {
  const DevState<R> *__restrict__ S = tstate<R>();
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ View<R> sV;
  __shared__ WarpCnt s_wc[GV_MAX_BLOCK / 32];
  __shared__ Plan s_plan;
  __shared__ unsigned s_chunk;
  __shared__ unsigned s_slice[SORT ? 1 : kNClaim + 1];
  __shared__ StackCount s_stack;  // the block's secondary stack (local_stack)
  __shared__ unsigned s_key[2][kNKey];  // requests per key of this round and the next
  Ctl *ctl = S->ctl;
  const int tid = threadIdx.x, lane = tid & 31;
  // Programmatic dependent launch (pdl): the next generation's blocks may
  // start as soon as this one's finish, stage their tables, and wait for
  // this grid (and its plan) to complete before reading the plan.
  asm volatile("griddepcontrol.launch_dependents;");
  // A done flag seen before the wait is final: nothing is planned, and the block
  // leaves.  The previous generation may set it while the block looks, so one
  // verdict holds for the block: what its threads do after the wait (the plan
  // is read by sixteen of them) is done by all of them or by none.
  if (__syncthreads_or(ctl->plan.done)) return;
  unsigned long long *const row = s_wc[tid >> 5];
  if (lane < 16) row[lane] = 0ull;
  if (tid < 2 * kNKey) s_key[tid / kNKey][tid % kNKey] = 0u;
  stage_tables(S, smem, sV);
  if (tid == 0) {
    s_stack.used = s_stack.taken[0] = s_stack.taken[1] = 0u;
    s_chunk = blockIdx.x;  // the first claim is the block's own
  }
  // the previous generation, and its plan, complete before the plan is read
  asm volatile("griddepcontrol.wait;" ::: "memory");
  static_assert(sizeof(Plan) == 64, "read in sixteen words");
  if (tid < 16) reinterpret_cast<unsigned *>(&s_plan)[tid] = reinterpret_cast<const unsigned *>(&ctl->plan)[tid];
  __syncthreads();
  if (s_plan.done) return;  // uniform: nothing planned for this generation
  const unsigned *const s_end = s_plan.end;
  const unsigned s_pb = s_plan.prim_begin;
  const bool block_claims = SORT || S->claim_chunks == 0;
  if (!SORT && tid <= kNClaim)
    s_slice[SORT ? 0 : tid] = static_cast<unsigned>((static_cast<unsigned long long>(s_end[3]) * static_cast<unsigned>(tid)) / kNClaim);
  if (!SORT) __syncthreads();
  const View<R> &V = sV;
  const int in = parity, out = parity ^ 1;
  // With several rounds per claim, the secondaries made in a round stay in
  // the block and fill its idle lanes in the next rounds (local_stack).
  const bool use_local = SORT && S->local_stack && s_plan.K > 1;
  const bool book = s_plan.book != 0;
  LocalStack<R> lstk;
  lstk.e = smem + S->smem_lk_off;
  lstk.count = &s_stack;
  lstk.cap = static_cast<int>(blockDim.x);
  ReqStore<R> req;
  req.m = smem + S->smem_req_off;
  req.n = static_cast<int>(blockDim.x);
  int w_slice = 0, buf = 0;
  if (!block_claims) {
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    w_slice = static_cast<int>((smid * 4u + ((tid >> 5) & 3u)) % kNClaim);
  }
  Pending<R> pend;  // this lane's unflushed deposit (merged scoring)
  pend.key = kNoKey;
  pend.sum = R(0);
  pend.comp = R(0);
  Pending<R> *const pd = MERGE ? &pend : nullptr;
  for (;;) {
    // Work claiming: with the basketizer a chunk is one block (its step loop
    // syncs the block); without it every warp claims its own 32-track chunks
    // and never waits for the rest of the block.
    unsigned chunk, idx;
    if (block_claims) {
      chunk = s_chunk;
      // (the basketizer's own barriers stand between this read and the next write)
      if (!SORT) __syncthreads();
    } else {
      // The chunk range is split into kNClaim slices, each with its own
      // counter in its own cache line: a warp draws from its SM's slice and
      // moves on when that slice is spent, so no single address takes every
      // claim of the generation.
      unsigned c0 = 0;
      if (lane == 0) {
        c0 = 0xffffffffu;
        for (int k = 0; k < kNClaim; ++k) {
          const int r = (w_slice + k) % kNClaim;
          const unsigned lo = s_slice[r], hi = s_slice[r + 1];
          if (lo >= hi) continue;
          const unsigned c = lo + atomicAdd(&ctl->claims[r].n, 1u);
          if (c < hi) {
            c0 = c;
            w_slice = r;
            break;
          }
        }
      }
      chunk = __shfl_sync(0xffffffffu, c0, 0);
      if (chunk == 0xffffffffu) break;
    }
    if (chunk >= s_end[3]) break;
    int qsel = 0;
    while (chunk >= s_end[qsel]) ++qsel;
    {
      const unsigned csize = block_claims ? s_plan.B : 32u;
      idx = (chunk - (qsel ? s_end[qsel - 1] : 0u)) * csize + (block_claims ? tid : lane);
      if (block_claims && static_cast<unsigned>(tid) >= csize) idx = 0xffffffffu;
    }
    qsel = claim_queue(qsel);
    Trk<R> t;
    t.type = 0;
    t.ev = 0;
    bool alive = false;
    if (qsel < 3) {
      if (idx < s_plan.n_in[qsel]) {
        load_track<R>(S, in, qsel, idx, t);
        alive = true;
        GV_CHECK(&ctl->status, t.sub >= 0 && t.sub < V.geo.nsub && t.ev < S->n_events && t.E >= R(0));
      }
    } else {
      const bool has = idx < s_plan.prim_count;
      int note = 0;
      if (has) alive = load_primary<R, EXT>(V, S, s_pb + idx, book, t, note);
      count_primaries(row, has, t.type, note);
    }
    const int K = s_plan.K;
    unsigned ended_own = 0u, ended_req = 0u;  // evlive before this lane's last bookings of an end (1: the event closed)
    unsigned ev_req = 0u, next_chunk = 0u;
    bool claimed = false;
    for (int kk = 0; kk < K; ++kk) {
      // (with the basketizer the block leaves the loop together, after the
      // count barrier below shows that no lane was alive)
      if (!SORT && !__any_sync(0xffffffffu, alive)) break;
      if (use_local && kk > 0) {
        // idle lanes take up secondaries of earlier rounds: of the kind their
        // warp steps already, warps without a track by turns of either kind
        const unsigned live = __ballot_sync(0xffffffffu, alive);
        const int kind = live ? __any_sync(0xffffffffu, alive && t.type != 0) : tid >> 5 & 1;
        if (lstk.take(~live, kind, t)) alive = true;
        if (!__any_sync(0xffffffffu, alive) && lstk.take(~live, kind ^ 1, t)) alive = true;
      }
      const bool was_alive = alive;
      // Along-step part.  With the basketizer a lane keeps stepping (boundary-
      // and continuous-limited steps need no final state) until its track is
      // due a discrete interaction, ends, or has taken its type's budget of
      // steps (photons cross layers in runs of boundary-limited steps; charged
      // tracks are stopped more often by their continuous-loss limit); the
      // block then baskets the interactions.
      uint32_t kstep;
      R u2 = R(0), u3 = R(0);
      Run<R> run;
      const int key = run_round<R, FIELD, OPTS, EXT>(V, S, t, alive, SORT ? S->along_steps_g : 1,
                                                     SORT ? S->along_steps : 1, kstep, u2, u3, run, pd);
      count_round(row, run, t.type, key >= 0 && key != kKeyRest);
      bool own_end = was_alive && !alive && key < 0;  // ended without a final state
      if (!SORT) {  // final state in place (warp-divergent across processes)
        Kids<R> kids;
        kids.n = 0;
        uint4 ids = make_uint4(0u, 0u, 0u, 0u);
        int np = 0, na = 0, change = own_end ? -1 : 0;
        if (key >= 0) {
          R d[3] = {t.u, t.v, t.w};
          const int r = final_state<R, OPTS, EXT, ALT>(V, S, key, t.E, d, u2, u3, kids, t.ev, t.sub, t.x, t.y, t.id, kstep, np,
                                                  na, ids, pd);
          if (r >= 0) {
            t.u = d[0]; t.v = d[1]; t.w = d[2];
            t.flags |= kFlagInteracted;
            alive = r != 0;
          }
          change = kids.n - (r == 0 ? 1 : 0);
        }
        wcnt_add(row, GV_C_PAIR, __popc(__ballot_sync(0xffffffffu, np)));
        wcnt_add(row, GV_C_ANNIH, __popc(__ballot_sync(0xffffffffu, na)));
        if (book && book_live(S, t.ev, change) == 1u) event_closed(S, t.ev);
        push_kids<R, EXT>(S, out, Parent{t.x, t.y, t.z, t.id, t.ev, t.sub}, kids, kstep, ids, row);
        if (MERGE) warp_flush(S, pend);
        continue;
      }
      if (MERGE) warp_flush(S, pend);
      // Basketizer: counting sort of this step's interaction requests by
      // (type, process), so every warp runs a single final-state model.
      // Three block barriers per round: counts, requests, results.  A warp
      // ranks its requests key by key (the keys it has: one to three), and
      // one lane per key adds its count to the block's.
      unsigned rank = 0, base = 0;
      int leader = 0;
      for (unsigned rest = __ballot_sync(0xffffffffu, key >= 0); rest;) {
        const int l = __ffs(rest) - 1;
        const unsigned m = __ballot_sync(0xffffffffu, key == __shfl_sync(0xffffffffu, key, l));
        if (m >> lane & 1u) {
          rank = __popc(m & ((1u << lane) - 1u));
          leader = l;
          if (lane == l) base = __popc(m);
        }
        rest &= ~m;
      }
      if (base) base = atomicAdd(&s_key[buf][key], base);
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!__syncthreads_or(was_alive)) break;  // uniform: no lane of the block was alive this step
      if (use_local && tid == 0) s_stack.settle();
      if (tid < kNKey) s_key[buf ^ 1][tid] = 0u;
      const unsigned ck = lane < kNKey ? s_key[buf][lane] : 0u;
      // each key's slots start at a warp's first thread where the block has
      // the threads for that: no warp then runs two models one after the other
      // (2000 x 10 GeV: 5.11 -> 4.93 ms)
      const unsigned whole = (ck + 31u) & ~31u;
      unsigned incl = ck | whole << 16;
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned total = __shfl_sync(0xffffffffu, incl, kNKey - 1);
      const bool apart = total >> 16 <= blockDim.x;
      const unsigned start = apart ? (incl >> 16) - whole : (incl & 0xffffu) - ck;
      const int slot = static_cast<int>(__shfl_sync(0xffffffffu, start, key >= 0 ? key : 0) + base + rank);
      unsigned nreq = total & 0xffffu;  // requests end here, for this warp
      if (apart) {
        const unsigned wb = tid & ~31u;
        const unsigned mine = __ballot_sync(0xffffffffu, start <= wb && wb < start + ck);
        const unsigned end = __shfl_sync(0xffffffffu, start + ck, mine ? __ffs(mine) - 1 : 0);
        nreq = mine ? end : 0u;
      }
      buf ^= 1;
      if (key >= 0) {
        req.xy(slot) = make_double2(t.x, t.y);
        req.zi(slot) = make_double2(t.z, i2d(t.id));
        req.info(slot) = make_uint4(t.ev, kstep, static_cast<unsigned>(t.sub), static_cast<unsigned>(key));
        req.dir(slot) = V4<R>{t.u, t.v, t.w, t.E};
        req.u2(slot) = u2;
        req.u3(slot) = u3;
      }
      __syncthreads();
      Kids<R> kb;
      kb.n = 0;
      Parent par;
      uint32_t pk = 0;
      uint4 ids = make_uint4(0u, 0u, 0u, 0u);
      int first = 0;  // of the lane's secondaries, the first that is not on the stack
      {
        int np = 0, na = 0;
        if (static_cast<unsigned>(tid) < nreq) {
          const double2 a = req.xy(tid), c = req.zi(tid);
          const uint4 g = req.info(tid);
          const V4<R> dE = req.dir(tid);
          par.x = a.x; par.y = a.y; par.z = c.x;
          par.id = d2i(c.y);
          par.ev = g.x;
          par.sub = static_cast<int>(g.z);
          pk = g.y;
          R d[3] = {dE.x, dE.y, dE.z};
          R e = dE.w;
          const int r = final_state<R, OPTS, EXT, ALT>(V, S, static_cast<int>(g.w), e, d, req.u2(tid), req.u3(tid), kb, par.ev,
                                                  par.sub, par.x, par.y, par.id, pk, np, na, ids);
          req.dir(tid) = V4<R>{d[0], d[1], d[2], e};
          req.ret(tid) = r;
          if (book) {
            ended_req = book_live(S, par.ev, kb.n - (r == 0 ? 1 : 0));
            ev_req = par.ev;
          }
        }
        wcnt_add(row, GV_C_PAIR, __popc(__ballot_sync(0xffffffffu, np)));
        wcnt_add(row, GV_C_ANNIH, __popc(__ballot_sync(0xffffffffu, na)));
        // with more rounds to come the secondaries go on the block's stack
        if (use_local && kk + 1 < K) first = stack_kids<R, EXT>(S, lstk, par, kb, pk, ids, row);
      }
      __syncthreads();
      if (key >= 0 && key != kKeyRest) {
        const int r = req.ret(slot);
        if (r >= 0) {
          const V4<R> dE = req.dir(slot);
          t.E = dE.w; t.u = dE.x; t.v = dE.y; t.w = dE.z;
          t.flags |= kFlagInteracted;
          alive = r != 0;
        }
      }
      if (book && own_end) ended_own = book_live(S, t.ev, -1);
      if (kk + 1 == K) {
        // the next claim's atomic is in flight while the claim's tracks go out
        if (tid == 0) next_chunk = gridDim.x + atomicAdd(&ctl->claim.n, 1u);
        claimed = true;
      }
      if (kk + 1 == K || __any_sync(0xffffffffu, first < kb.n))
        push_all<R, EXT>(S, out, par, kb, first, ids, pk, t, alive && kk + 1 == K, row);
      // (the event counts' atomics were in flight while the tracks went out)
      if (ended_own == 1u) event_closed(S, t.ev);
      if (ended_req == 1u) event_closed(S, ev_req);
      ended_own = ended_req = 0u;
    }
    if (block_claims && !claimed && tid == 0) next_chunk = gridDim.x + atomicAdd(&ctl->claim.n, 1u);
    if (MERGE) warp_flush(S, pend);  // nothing stays pending past a claim
    if (!SORT) push_track(S, out, t, alive);
    if (use_local) {  // what is left on the block's stack goes to the next generation
      __syncthreads();
      const unsigned ng = s_stack.used & 0xffffu, nq = s_stack.used >> 16;
      // (the last round's appends came after its takes were settled)
      Trk<R> k;
      k.type = 0;
      const bool has = static_cast<unsigned>(tid) < ng || static_cast<unsigned>(tid) >= blockDim.x - nq;
      if (has) lstk.get(tid, k);
      push_track(S, out, k, has);
      __syncthreads();
      if (tid == 0) s_stack.used = 0u;
    }
    if (block_claims) {
      if (tid == 0) s_chunk = next_chunk;
      __syncthreads();
    }
  }
  // flush the warps' counters; the last block plans the next generation
  __syncthreads();
  if (tid < 16) {
    unsigned long long v = 0ull;
    for (unsigned w = 0; w < blockDim.x / 32; ++w) v += s_wc[w][tid];
    if (v) atomicAdd(&ctl->counters[tid], v);
  }
  __syncthreads();
  if (tid == 0 && block_done(&ctl->blocks_done)) plan_next(S, out);
}

// ------------------------------------------------------------------ split pipeline
// The same generation in two kernels.  The along-step kernel runs the lanes'
// steps until a track is due a discrete interaction, ends, or has taken its
// along-step budget, without any block barrier after the claim; a track due
// an interaction becomes a request record and its index goes to the list of
// its (type, process) key.  The interaction kernel then gives every warp 32
// requests of one key, so each warp runs one final-state model, and writes
// survivors and secondaries to the output queues; its last block plans the
// next generation.  The price is one request record written and read per
// interaction.

// Hand the tracks due an interaction to the interaction kernel.  All 32
// lanes of a converged warp.
template <typename R>
__device__ void emit_requests(const DevState<R> *S, const Trk<R> &t, int key, uint32_t kstep, R u2, R u3) {
  const bool hand = key >= 0;
  const unsigned mh = __ballot_sync(0xffffffffu, hand);
  if (!mh) return;
  Ctl *ctl = S->ctl;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(&ctl->req_n, __popc(mh));
  const unsigned slot = __shfl_sync(0xffffffffu, base, 0) + __popc(mh & lt);
  const bool ok = hand && slot < S->req_cap;
  if (hand && !ok) set_status(ctl, GV_ERR_STACK_FULL);
  if (ok) {
    GReq<R> &q = S->req[slot];
    q.x = t.x; q.y = t.y; q.z = t.z;
    q.id = t.id;
    q.E = t.E; q.d0 = t.u; q.d1 = t.v; q.d2 = t.w;
    q.u2 = u2;
    q.u3 = u3;
    q.ev = t.ev;
    q.kk = kstep;
    q.sf = t.sub | (t.flags << 16);
    q.key = key;
  }
#pragma unroll
  for (int k = 0; k < kNReqKey; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, ok && key == k);
    if (!m) continue;
    unsigned b = 0;
    if (lane == 0) b = atomicAdd(&ctl->key_n[k], __popc(m));
    b = __shfl_sync(0xffffffffu, b, 0);
    if (m >> lane & 1u) S->keyidx[static_cast<size_t>(k) * S->req_cap + b + __popc(m & lt)] = slot;
  }
}

// FP64: one block per SM without a register cap, as for the step kernel (two
// blocks at 128 registers spilled 144 bytes in the steps' loop: 1000 x 1 GeV
// 12.6 -> 8.25 ms, 1600 tracks between near walls 2.03 -> 1.39 ms).
template <typename R>
#ifndef GV_ALONG_MIN_BLOCKS
#define GV_ALONG_MIN_BLOCKS 2
#endif
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? GV_ALONG_MIN_BLOCKS : 1) along_kernel(const DevState<R> *__restrict__ S, int parity) {
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ View<R> sV;
  __shared__ WarpCnt s_wc[8];
  __shared__ unsigned s_chunk;
  Ctl *ctl = S->ctl;
  const int tid = threadIdx.x, lane = tid & 31;
  if (ctl->plan.done) return;
  unsigned long long *const row = s_wc[tid >> 5];
  if (lane < 16) row[lane] = 0ull;
  stage_tables(S, smem, sV);
  const View<R> &V = sV;
  const int in = parity, out = parity ^ 1;
  const unsigned n_prim_gen = ctl->plan.prim_count, n_chunks = ctl->plan.end[3];
  const bool book = ctl->plan.book != 0;
  for (;;) {
    if (tid == 0) s_chunk = atomicAdd(&ctl->claim.n, 1u);
    __syncthreads();
    const unsigned chunk = s_chunk;
    __syncthreads();
    if (chunk >= n_chunks) break;
    int qsel = 0;
    while (chunk >= ctl->plan.end[qsel]) ++qsel;
    const unsigned idx = (chunk - (qsel ? ctl->plan.end[qsel - 1] : 0u)) * blockDim.x + tid;
    qsel = claim_queue(qsel);
    Trk<R> t;
    t.type = 0;
    t.ev = 0;
    bool alive = false;
    if (qsel < 3) {
      if (idx < ctl->plan.n_in[qsel]) {
        load_track<R>(S, in, qsel, idx, t);
        alive = true;
        GV_CHECK(&ctl->status, t.sub >= 0 && t.sub < V.geo.nsub && t.ev < S->n_events && t.E >= R(0));
      }
    } else {
      const bool has = idx < n_prim_gen;
      int note = 0;
      if (has) alive = load_primary<R, true>(V, S, ctl->plan.prim_begin + idx, book, t, note);
      count_primaries(row, has, t.type, note);
    }
    const int K = ctl->plan.K;
    for (int kk = 0; kk < K; ++kk) {
      if (!__any_sync(0xffffffffu, alive)) break;
      const bool was_alive = alive;
      uint32_t kstep;
      R u2 = R(0), u3 = R(0);
      Run<R> run;
      const int key = run_round<R, true, true, true>(V, S, t, alive, S->along_steps_g, S->along_steps, kstep, u2, u3, run,
                                                     static_cast<Pending<R> *>(nullptr));
      count_round(row, run, t.type, key >= 0 && key != kKeyRest);
      if (book && was_alive && !alive && key < 0 && book_live(S, t.ev, -1) == 1u) event_closed(S, t.ev);
      emit_requests(S, t, key, kstep, u2, u3);
      if (key >= 0) alive = false;  // the interaction kernel owns it now
    }
    push_track(S, out, t, alive);
  }
  __syncthreads();
  if (tid < 16) {
    unsigned long long v = 0ull;
    for (unsigned w = 0; w < blockDim.x / 32; ++w) v += s_wc[w][tid];
    if (v) atomicAdd(&ctl->counters[tid], v);
  }
}

template <typename R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 2 : 1) interact_kernel(const DevState<R> *__restrict__ S, int parity) {
  __shared__ View<R> sV;
  __shared__ WarpCnt s_wc[8];
  __shared__ unsigned s_kend[kNReqKey], s_kn[kNReqKey];
  Ctl *ctl = S->ctl;
  const int tid = threadIdx.x, lane = tid & 31;
  if (ctl->plan.done) return;
  if (tid == 0) {
    sV = S->view;  // tables stay in global memory: the final states read the alias bins only
    unsigned acc = 0;
    for (int k = 0; k < kNReqKey; ++k) {
      const unsigned n = min(ctl->key_n[k], static_cast<unsigned>(S->req_cap));
      s_kn[k] = n;
      acc += (n + 31u) / 32u;
      s_kend[k] = acc;
    }
  }
  unsigned long long *const row = s_wc[tid >> 5];
  if (lane < 16) row[lane] = 0ull;
  __syncthreads();
  const View<R> &V = sV;
  const int out = parity ^ 1;
  const bool book = ctl->plan.book != 0;
  for (;;) {
    unsigned chunk = 0;
    if (lane == 0) chunk = atomicAdd(&ctl->claim_b, 1u);
    chunk = __shfl_sync(0xffffffffu, chunk, 0);
    if (chunk >= s_kend[kNReqKey - 1]) break;
    int k = 0;
    while (chunk >= s_kend[k]) ++k;
    const unsigned pos = (chunk - (k ? s_kend[k - 1] : 0u)) * 32u + lane;
    Trk<R> t;
    t.type = 0;
    Kids<R> kids;
    kids.n = 0;
    Parent par = {0.0, 0.0, 0.0, 0ull, 0u, 0};
    uint32_t kk = 0;
    uint4 ids = make_uint4(0u, 0u, 0u, 0u);
    int np = 0, na = 0;
    unsigned was = 0u;
    bool alive = false;
    if (pos < s_kn[k]) {
      const GReq<R> q = S->req[S->keyidx[static_cast<size_t>(k) * S->req_cap + pos]];
      R d[3] = {q.d0, q.d1, q.d2};
      R e = q.E;
      t.x = q.x; t.y = q.y; t.z = q.z;
      t.id = q.id;
      t.ev = q.ev;
      t.sub = q.sf & 0xffff;
      t.flags = q.sf >> 16;
      t.type = k / 3;
      kk = q.kk;
      t.step = kk + 1;
      t.nlam = R(-1);
      const int r = final_state<R>(V, S, k, e, d, q.u2, q.u3, kids, t.ev, t.sub, t.x, t.y, q.id, q.kk, np, na, ids);
      t.E = e;
      t.u = d[0]; t.v = d[1]; t.w = d[2];
      if (r >= 0) t.flags |= kFlagInteracted;
      alive = r != 0;
      par = Parent{t.x, t.y, t.z, t.id, t.ev, t.sub};
      if (book) was = book_live(S, t.ev, kids.n - (alive ? 0 : 1));
    }
    wcnt_add(row, GV_C_PAIR, __popc(__ballot_sync(0xffffffffu, np)));
    wcnt_add(row, GV_C_ANNIH, __popc(__ballot_sync(0xffffffffu, na)));
    push_kids<R>(S, out, par, kids, kk, ids, row);
    push_track(S, out, t, alive);
    if (was == 1u) event_closed(S, t.ev);
  }
  __syncthreads();
  if (tid < 16) {
    unsigned long long v = 0ull;
    for (unsigned w = 0; w < blockDim.x / 32; ++w) v += s_wc[w][tid];
    if (v) atomicAdd(&ctl->counters[tid], v);
  }
  __syncthreads();
  if (tid == 0 && block_done(&ctl->blocks_done_b)) plan_next(S, out);
}

}  // namespace gv

// ====================================================================== host
using namespace gv;

namespace {

struct Ctx {
  int device = 0, sm_count = 0;
  gv_config cfg;
  std::vector<gv_material> mats;
  gv_layers geo;
  gv_cuts cuts;
  int nsub = 0;
  std::vector<double> zb;
  std::vector<unsigned char> smat;
  bool tables = false;
  HostTables ht;
  // device allocations
  void *d_xs = nullptr, *d_bins = nullptr, *d_smax = nullptr;
  float *d_inv_node = nullptr;
  double *d_zb = nullptr;
  unsigned char *d_smat = nullptr;
  void *d_queues = nullptr;
  Ctl *d_ctl = nullptr;
  void *d_state = nullptr;
  double *d_edep = nullptr, *d_cell = nullptr, *d_escape = nullptr;
  unsigned long long *d_evcnt = nullptr;
  unsigned *d_evlive = nullptr;
  unsigned long long *d_evcost = nullptr;  // budget held per event (automatic in-flight cap)
  size_t ev_cap = 0;
  unsigned long long *d_pcost = nullptr;   // prefix sums of the primaries' budgets
  size_t pcost_cap = 0;
  unsigned long long *d_part = nullptr;    // budgets of each scan block's primaries
  gv_primary *d_prim = nullptr;
  unsigned *d_order = nullptr;
  size_t prim_cap = 0;
  cudaStream_t stream = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr, t0 = nullptr, t1 = nullptr;
  cudaGraphExec_t graph = nullptr;
  int loop_graph = 0;  // graph holds the device-side generation loop
  Ctl *h_ctl = nullptr;  // pinned
  long long launches = 0;
  int last_status = 0;
  // a transport whose completion gv_sync (or the next call) collects
  struct {
    bool active = false;
    gv_result *res = nullptr;
    long long launches = 0;  // launches known before the device-side loop ran
    double kernel_ms = 0.0;  // host-looped transports: measured already
    bool timed_loop = false; // kernel time = t0 .. t1 of the one graph launch
  } pend;
  ModelMeta meta[kNModel];
  size_t xs_bytes = 0, zb_bytes = 0, smem_bytes = 0, req_off = 0, bins_bytes = 0, smax_bytes = 0, smax_off = 0, rec_off = 0;
  size_t lk_off = 0;
  int grid = 0, grid_b = 0;
  // split pipeline: interaction requests and their per-key index lists
  void *d_req = nullptr;
  unsigned *d_keyidx = nullptr;
  // L2 persisting window over the alias bins (config l2_persist)
  size_t l2_window = 0, l2_old_limit = 0;
};

#define CK(x)                                  \
  do {                                         \
    cudaError_t e_ = (x);                      \
    if (e_ != cudaSuccess) return GV_ERR_CUDA; \
  } while (0)

int validate(const gv_material *mats, int n_mats, const gv_layers *geo, const gv_cuts *cuts) {
  if (!mats || !geo || !cuts || n_mats < 1 || n_mats > GV_MAX_MAT) return GV_ERR_BAD_ARG;
  for (int m = 0; m < n_mats; ++m) {
    const gv_material &x = mats[m];
    if (x.n_elem < 1 || x.n_elem > GV_MAX_ELEM || !(x.rho > 0) || !(x.I_eV > 0)) return GV_ERR_BAD_ARG;
    for (int e = 0; e < x.n_elem; ++e)
      if (!(x.Z[e] >= 1) || !(x.A[e] > 0) || !(x.w[e] > 0)) return GV_ERR_BAD_ARG;
  }
  if (geo->n_layers < 1 || geo->n_sub < 1 || geo->n_sub > GV_MAX_SUB ||
      static_cast<long long>(geo->n_layers) * geo->n_sub > GV_MAX_SUBTOTAL)
    return GV_ERR_BAD_ARG;
  for (int j = 0; j < geo->n_sub; ++j)
    if (!(geo->sub_thick_cm[j] > 0) || geo->sub_mat[j] < 0 || geo->sub_mat[j] >= n_mats) return GV_ERR_BAD_ARG;
  if (geo->nx_cells < 0 || geo->ny_cells < 0) return GV_ERR_BAD_ARG;
  if (!(std::fabs(geo->field_T) < 1e4) || geo->field_axis < 0 || geo->field_axis > 2) return GV_ERR_BAD_ARG;
  if ((geo->nx_cells > 0 || geo->ny_cells > 0) &&
      !(geo->nx_cells > 0 && geo->ny_cells > 0 && geo->half_x_cm > 0 && geo->half_y_cm > 0))
    return GV_ERR_BAD_ARG;
  if (!(cuts->track_cut_MeV >= kGridEmin) || !(cuts->gamma_cut_MeV >= cuts->track_cut_MeV) ||
      !(cuts->e_cut_MeV >= cuts->track_cut_MeV))
    return GV_ERR_BAD_ARG;
  return GV_OK;
}

int validate_cfg(const gv_config &c) {
  if (c.precision != GV_MIXED && c.precision != GV_FP64) return GV_ERR_BAD_ARG;
  if (c.mode != GV_BATCHED && c.mode != GV_ONE_EVENT_PER_LAUNCH) return GV_ERR_BAD_ARG;
  if (c.block_size < 64 || c.block_size > GV_MAX_BLOCK || c.block_size % 32) return GV_ERR_BAD_ARG;
  if (c.blocks_per_sm < 1 || c.blocks_per_sm > 32) return GV_ERR_BAD_ARG;
  if (c.steps_per_claim < 1 || c.tail_steps_per_claim < 1 || c.steps_per_claim > 4096 ||
      c.tail_steps_per_claim > 4096)
    return GV_ERR_BAD_ARG;
  if (c.stack_capacity < 1024 || c.stack_capacity > (1ll << 31)) return GV_ERR_BAD_ARG;
  if (c.refill_batch < 1 || c.refill_low_water < 0) return GV_ERR_BAD_ARG;
  if (c.generations_per_graph < 2 || c.generations_per_graph % 2 || c.generations_per_graph > 1024)
    return GV_ERR_BAD_ARG;
  if (c.max_generations < 1 || c.max_events_in_flight < -1) return GV_ERR_BAD_ARG;
  if (c.claim_chunks < 0 || c.claim_chunks > 1) return GV_ERR_BAD_ARG;
  if (c.along_steps < 1 || c.along_steps > 64) return GV_ERR_BAD_ARG;
  if (c.along_steps_photon < 0 || c.along_steps_photon > 64) return GV_ERR_BAD_ARG;
  if (c.scoring < 0 || c.scoring > 1) return GV_ERR_BAD_ARG;
  if (c.l2_persist < 0 || c.l2_persist > 1) return GV_ERR_BAD_ARG;
  if (c.local_stack < 0 || c.local_stack > 1) return GV_ERR_BAD_ARG;
  if (c.pdl < 0 || c.pdl > 1) return GV_ERR_BAD_ARG;
  if (c.device_loop < 0 || c.device_loop > 1) return GV_ERR_BAD_ARG;
  if (c.blocking < 0 || c.blocking > 1) return GV_ERR_BAD_ARG;
  if (c.pipeline < 0 || c.pipeline > 1 || (c.pipeline == 1 && c.scoring != 0)) return GV_ERR_BAD_ARG;
  return GV_OK;
}

template <typename R> int upload_tables(Ctx *c) {
  const HostTables &h = c->ht;
  // cross sections as V4<R>
  const size_t nv = static_cast<size_t>(h.n_mat) * 3 * kGridN;
  std::vector<V4<R>> xs(nv);
  for (size_t i = 0; i < nv; ++i) {
    // the range (e- component z, e+ component w) is stored as ln R
    const int type = static_cast<int>((i / kGridN) % 3);
    xs[i].x = static_cast<R>(h.xs[4 * i + 0]);
    xs[i].y = static_cast<R>(h.xs[4 * i + 1]);
    xs[i].z = static_cast<R>(type == 1 ? std::log(h.xs[4 * i + 2]) : h.xs[4 * i + 2]);
    xs[i].w = static_cast<R>(type == 2 ? std::log(h.xs[4 * i + 3]) : h.xs[4 * i + 3]);
  }
  if (sizeof(R) == 8)  // an electron's free component: the slope of its ln R (loss_slope)
    for (size_t i = 0; i + 1 < nv; ++i)
      if ((i / kGridN) % 3 == 1 && i % kGridN + 1 < kGridN) xs[i].w = static_cast<R>(kLnNode / (xs[i + 1].z - xs[i].z));
  c->xs_bytes = nv * sizeof(V4<R>);
  CK(cudaMalloc(&c->d_xs, c->xs_bytes));
  CK(cudaMemcpy(c->d_xs, xs.data(), c->xs_bytes, cudaMemcpyHostToDevice));
  // reciprocal node energies for the FP32 interval fraction
  std::vector<float> inv(kGridN);
  for (int i = 0; i < kGridN; ++i)
    inv[i] = static_cast<float>(std::exp(-(std::log(kGridEmin) + i * std::log(10.0) / kGridPerDecade)));
  CK(cudaMalloc(&c->d_inv_node, sizeof(float) * kGridN));
  CK(cudaMemcpy(c->d_inv_node, inv.data(), sizeof(float) * kGridN, cudaMemcpyHostToDevice));
  // alias bins
  std::vector<AliasBin<R>> bins;
  for (int m = 0; m < kNModel; ++m) {
    c->meta[m].ln_Elo = std::log(h.a_Elo[m]);
    c->meta[m].inv_dl = kAliasPerDecade / std::log(10.0);
    c->meta[m].cut = h.a_cut[m];
    c->meta[m].nE = h.a_nE[m];
    c->meta[m].off = static_cast<int>(bins.size());
    for (int ie = 0; ie < h.a_nE[m]; ++ie)
      for (int j = 0; j < kNB; ++j) {
        AliasBin<R> b;
        b.q = h.a_q[m][static_cast<size_t>(ie) * kNB + j];
        b.a = h.a_alias[m][static_cast<size_t>(ie) * kNB + j];
        b.p0 = static_cast<R>(h.a_pdf[m][static_cast<size_t>(ie) * (kNB + 1) + j]);
        b.p1 = static_cast<R>(h.a_pdf[m][static_cast<size_t>(ie) * (kNB + 1) + j + 1]);
        bins.push_back(b);
      }
  }
  {  // the integral approach's bound
    std::vector<R> sm(h.smax.size());
    for (size_t i = 0; i < sm.size(); ++i) sm[i] = static_cast<R>(h.smax[i]);
    c->smax_bytes = (sm.size() * sizeof(R) + 15) / 16 * 16;
    CK(cudaMalloc(&c->d_smax, c->smax_bytes));
    CK(cudaMemcpy(c->d_smax, sm.data(), sm.size() * sizeof(R), cudaMemcpyHostToDevice));
  }
  c->bins_bytes = bins.size() * sizeof(AliasBin<R>);
  CK(cudaMalloc(&c->d_bins, c->bins_bytes));
  CK(cudaMemcpy(c->d_bins, bins.data(), c->bins_bytes, cudaMemcpyHostToDevice));
  return GV_OK;
}

// Alias bins are read at random by every interaction; a persisting L2
// window keeps them resident while the queues stream through L2.  The
// context's persisting set-aside is raised to the window (if smaller) and put
// back by gv_destroy.
int setup_l2_window(Ctx *c) {
  if (!c->cfg.l2_persist || !c->bins_bytes) return GV_OK;
  int max_persist = 0, max_window = 0;
  CK(cudaDeviceGetAttribute(&max_persist, cudaDevAttrMaxPersistingL2CacheSize, c->device));
  CK(cudaDeviceGetAttribute(&max_window, cudaDevAttrMaxAccessPolicyWindowSize, c->device));
  const size_t w = std::min(c->bins_bytes, static_cast<size_t>(std::min(max_persist, max_window)));
  if (w == 0) return GV_OK;  // no persisting L2 on this device: nothing to do
  CK(cudaDeviceGetLimit(&c->l2_old_limit, cudaLimitPersistingL2CacheSize));
  if (c->l2_old_limit < w) CK(cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, w));
  c->l2_window = w;
  return GV_OK;
}

template <typename R> View<R> make_view(const Ctx *c) {
  View<R> v;
  v.xs = reinterpret_cast<const V4<R> *>(c->d_xs);
  v.inv_node = c->d_inv_node;
  v.zb = c->d_zb;
  v.smat = c->d_smat;
  v.bins = reinterpret_cast<const AliasBin<R> *>(c->d_bins);
  v.smax = reinterpret_cast<const R *>(c->d_smax);
  v.status = nullptr;  // unit kernels: no status word
  for (int m = 0; m < kNModel; ++m) v.meta[m] = c->meta[m];
  v.geo.nsub = c->nsub;
  v.geo.nsub_layer = c->geo.n_sub;
  v.geo.n_layers = c->geo.n_layers;
  v.geo.nx = c->geo.nx_cells;
  v.geo.ny = c->geo.ny_cells;
  v.geo.hx = c->geo.half_x_cm;
  v.geo.hy = c->geo.half_y_cm;
  v.geo.wx[0] = -c->geo.half_x_cm;
  v.geo.wx[1] = c->geo.half_x_cm;
  v.geo.wy[0] = -c->geo.half_y_cm;
  v.geo.wy[1] = c->geo.half_y_cm;
  {  // the half widths rounded down to FP32
    float fx = static_cast<float>(c->geo.half_x_cm), fy = static_cast<float>(c->geo.half_y_cm);
    if (static_cast<double>(fx) > c->geo.half_x_cm) fx = std::nextafter(fx, 0.0f);
    if (static_cast<double>(fy) > c->geo.half_y_cm) fy = std::nextafter(fy, 0.0f);
    v.geo.hx_lo = fx;
    v.geo.hy_lo = fy;
  }
  v.geo.walls_x = c->geo.half_x_cm > 0.0;
  v.geo.walls_y = c->geo.half_y_cm > 0.0;
  v.geo.field_axis = c->geo.field_axis;
  v.rc.field_k = static_cast<R>(2.99792458 * c->geo.field_T);
  v.geo.pitch_x = c->geo.nx_cells > 0 ? 2.0 * c->geo.half_x_cm / c->geo.nx_cells : 1.0;
  v.geo.pitch_y = c->geo.ny_cells > 0 ? 2.0 * c->geo.half_y_cm / c->geo.ny_cells : 1.0;
  v.geo.inv_pitch_x = static_cast<float>(1.0 / v.geo.pitch_x);
  v.geo.inv_pitch_y = static_cast<float>(1.0 / v.geo.pitch_y);
  v.cut.gcut = c->cuts.gamma_cut_MeV;
  v.cut.ecut = c->cuts.e_cut_MeV;
  v.cut.tcut = c->cuts.track_cut_MeV;
  v.rc.tcut = static_cast<R>(c->cuts.track_cut_MeV);
  v.rc.gcut = static_cast<R>(c->cuts.gamma_cut_MeV);
  v.rc.ecut = static_cast<R>(c->cuts.e_cut_MeV);
  v.rc.ecut_push = static_cast<R>(std::max(c->cuts.e_cut_MeV, c->cuts.track_cut_MeV));
  for (int m = 0; m < kNModel; ++m) {
    v.rc.ln_Elo[m] = static_cast<R>(c->meta[m].ln_Elo);
    v.rc.inv_dl[m] = static_cast<R>(c->meta[m].inv_dl);
    v.rc.cut[m] = static_cast<R>(c->meta[m].cut);
  }
  for (int m = 0; m < GV_MAX_MAT; ++m) v.rc.inv_X0[m] = static_cast<R>(c->ht.inv_X0_cm[m]);
  for (int m = 0; m < kNModel; ++m) {  // a threshold beyond R's range means "never"
    const double r = c->cuts.reject_min_MeV[m];
    v.rc.rej_min[m] = r < 1e30 ? static_cast<R>(r) : r_inf_host<R>();
  }
  v.cut.mask = c->cuts.process_mask;
  return v;
}

template <typename R> using StepFn = void (*)(int);

// The step kernel compiled for this configuration: basketizer or not, merged
// or direct scoring, with or without the field propagation.  The basketizing
// kernel also comes without the code of the optional processes (multiple
// scattering, the integral approach, rejection sampling), and without the
// cell histogram and per-event counters, for contexts that use none of
// them: each cut measured about 3 % on the benchmark against carrying the
// code behind run-time switches.
template <typename R> StepFn<R> pick_step_kernel(const Ctx *x) {
  const gv_config &c = x->cfg;
  const bool field = x->geo.field_T != 0.0;
  bool opts = (x->cuts.process_mask & (GV_P_MSC | GV_P_INTEGRAL)) != 0;
  for (int m = 0; m < kNModel; ++m) opts = opts || x->cuts.reject_min_MeV[m] < 1e30;
  // a transport scores cells or per-event counts only if the context has
  // cells or keeps per-event counts: otherwise both pointers stay null
  const bool ext = c.per_event_counts != 0 || static_cast<size_t>(x->geo.n_layers) * x->geo.nx_cells * x->geo.ny_cells != 0;
  if (field)
    return c.process_sort ? step_kernel<R, true, false, true, true, true> : step_kernel<R, false, false, true, true, true>;
  if (c.process_sort) {
    if (c.scoring) return step_kernel<R, true, true, false, true, true>;
    if (opts) return step_kernel<R, true, false, false, true, true>;
    return ext ? step_kernel<R, true, false, false, false, true> : step_kernel<R, true, false, false, false, false>;
  }
  return c.scoring ? step_kernel<R, false, true, false, true, true> : step_kernel<R, false, false, false, true, true>;
}

// The constant-memory state record of each precision and GPU (c_state_f,
// c_state_d) is shared by every context on that GPU.  A transport takes it
// on its stream once the previous transport of any context has released it
// (an event), fills it from its record in device memory, and releases it
// when everything it queued is on the stream.  The host lock orders the
// takes; the events order the uses on the GPU, so transports of different
// contexts on one GPU run one after another.
constexpr int kMaxDevices = 64;
std::mutex &slot_mutex() {
  static std::mutex m;
  return m;
}
cudaEvent_t g_slot_free[2][kMaxDevices];  // [FP64][device]

// Made with a context (gv_setup allocates anyway), so that the
// allocation-free entry point never creates one.
cudaError_t slot_event_create(int device, bool fp64) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(slot_mutex());
  cudaEvent_t &e = g_slot_free[fp64 ? 1 : 0][device];
  if (e) return cudaSuccess;
  return cudaEventCreateWithFlags(&e, cudaEventDisableTiming);
}

template <typename R> class StateSlot {
 public:
  StateSlot(int device, cudaStream_t st)
      : lk_(slot_mutex()), st_(st),
        ev_(device >= 0 && device < kMaxDevices ? g_slot_free[sizeof(R) == 8 ? 1 : 0][device] : nullptr) {}
  StateSlot(const StateSlot &) = delete;
  StateSlot &operator=(const StateSlot &) = delete;
  // wait for the previous user
  cudaError_t wait() { return ev_ ? cudaStreamWaitEvent(st_, ev_, 0) : cudaErrorInvalidResourceHandle; }
  // wait for the previous user, then copy the record into the slot
  cudaError_t take(const DevState<R> *record) {
    const cudaError_t e = wait();
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(R) == 8)
      return cudaMemcpyToSymbolAsync(c_state_d, record, sizeof(DevState<R>), 0, cudaMemcpyDeviceToDevice, st_);
    else
      return cudaMemcpyToSymbolAsync(c_state_f, record, sizeof(DevState<R>), 0, cudaMemcpyDeviceToDevice, st_);
  }
  ~StateSlot() {
    if (ev_) cudaEventRecord(ev_, st_);  // also after an error: what was queued is covered
  }

 private:
  std::unique_lock<std::mutex> lk_;
  cudaStream_t st_;
  cudaEvent_t ev_;
};

// Lets launches of `kern` on the current device have `bytes` of dynamic shared
// memory.  The limit is a property of the function, which contexts of other
// sizes and other threads launch too (or have captured and launch later), so
// it is always raised to the same value, the most a block of this kernel can
// have, and never lowered to what one of them needs.
cudaError_t allow_shared(const void *kern, int device, size_t bytes) {
  cudaFuncAttributes a;
  int most = 0;
  cudaError_t e = cudaFuncGetAttributes(&a, kern);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return e;
  most -= static_cast<int>(a.sharedSizeBytes);
  if (most < 0 || bytes > static_cast<size_t>(most)) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

template <typename R> int prepare_device(Ctx *c) {
  CK(cudaSetDevice(c->device));
  CK(slot_event_create(c->device, sizeof(R) == 8));
  int rc = upload_tables<R>(c);
  if (rc) return rc;
  rc = setup_l2_window(c);
  if (rc) return rc;
  const long long cap = c->cfg.stack_capacity;
  const size_t per = TrackLayout<R>::queue_bytes(cap);
  if (cudaMalloc(&c->d_queues, per * 6) != cudaSuccess) return GV_ERR_OOM;
  CK(cudaMalloc(&c->d_ctl, sizeof(Ctl)));
  CK(cudaMemset(c->d_ctl, 0, sizeof(Ctl)));
  CK(cudaMalloc(&c->d_state, sizeof(DevState<R>)));
  CK(cudaMalloc(&c->d_part, sizeof(unsigned long long) * (kScanBlocks + 1)));
  CK(cudaMallocHost(&c->h_ctl, sizeof(Ctl)));
  // the integral approach's bound is staged where that approach is on
  const size_t smax_bytes = (c->cuts.process_mask & GV_P_INTEGRAL) ? c->smax_bytes : 0;
  const auto layout = [c](size_t smax) {
    c->smax_bytes = smax;
    c->zb_bytes = ((c->nsub + 1) * sizeof(double) + 15) / 16 * 16;
    c->smax_off = c->xs_bytes + c->zb_bytes + kInvNodeBytes + (c->nsub + 15) / 16 * 16;
    c->rec_off = c->smax_off + smax;
    c->req_off = (c->rec_off + c->nsub * sizeof(SubRec<R>) + 31) / 32 * 32;
    c->smem_bytes = c->req_off;
    if (!c->cfg.pipeline && c->cfg.process_sort)
      c->smem_bytes += static_cast<size_t>(ReqStore<R>::kBytes) * c->cfg.block_size;
    c->lk_off = (c->smem_bytes + 31) / 32 * 32;
    if (!c->cfg.pipeline && c->cfg.process_sort && c->cfg.local_stack)
      c->smem_bytes = c->lk_off + static_cast<size_t>(LocalStack<R>::kBytes) * c->cfg.block_size;
  };
  layout(smax_bytes);
  if (c->cfg.pipeline) {
    const size_t rc_ = static_cast<size_t>(cap);
    if (cudaMalloc(&c->d_req, rc_ * sizeof(GReq<R>)) != cudaSuccess ||
        cudaMalloc(&c->d_keyidx, rc_ * kNReqKey * sizeof(unsigned)) != cudaSuccess)
      return GV_ERR_OOM;
    const void *ka = reinterpret_cast<const void *>(along_kernel<R>);
    const void *kb = reinterpret_cast<const void *>(interact_kernel<R>);
    CK(allow_shared(ka, c->device, c->smem_bytes));
    int occ = 0, occ_b = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ka, c->cfg.block_size, c->smem_bytes));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_b, kb, 256, 0));
    if (occ < 1 || occ_b < 1) return GV_ERR_BAD_ARG;
    c->grid = c->sm_count * std::min(occ, c->cfg.blocks_per_sm);
    c->grid_b = c->sm_count * occ_b;
    return GV_OK;
  }
  const void *kern = reinterpret_cast<const void *>(pick_step_kernel<R>(c));
  int occ = 0;
  const auto blocks = [&] {
    CK(allow_shared(kern, c->device, c->smem_bytes));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, c->cfg.block_size, c->smem_bytes));
    return static_cast<int>(GV_OK);
  };
  if (const int e = blocks()) return e;
  if (smax_bytes && occ < 2) {
    // four materials with many sub-slabs: the bound is read from L2 where its
    // place in shared memory would cost a block
    const int staged = occ;
    layout(0);
    if (const int e = blocks()) return e;
    if (occ == staged) {
      layout(smax_bytes);
      if (const int e = blocks()) return e;
    }
  }
  if (occ < 1) return GV_ERR_BAD_ARG;
  c->grid = c->sm_count * std::min(occ, c->cfg.blocks_per_sm);
  return GV_OK;
}

template <typename R> DevState<R> make_state(Ctx *c) {
  DevState<R> s;
  std::memset(&s, 0, sizeof(s));
  s.view = make_view<R>(c);
  s.qmem = static_cast<unsigned char *>(c->d_queues);
  s.q_bytes = TrackLayout<R>::queue_bytes(c->cfg.stack_capacity);
  s.q_part = TrackLayout<R>::part_bytes(c->cfg.stack_capacity);
  s.capacity = static_cast<unsigned long long>(c->cfg.stack_capacity);
  s.ctl = c->d_ctl;
  s.view.status = &c->d_ctl->status;  // device address; checks of the checking build
  s.block_size = c->cfg.block_size;
  s.chunk = (c->cfg.pipeline || c->cfg.process_sort || c->cfg.claim_chunks == 0) ? c->cfg.block_size : 32;
  s.grid = c->grid;
  s.adaptive_chunk = (c->cfg.process_sort && !c->cfg.pipeline) ? 1 : 0;
  s.claim_chunks = c->cfg.claim_chunks;
  s.along_steps = c->cfg.along_steps;
  s.along_steps_g = c->cfg.along_steps_photon > 0 ? c->cfg.along_steps_photon : c->cfg.along_steps;
  s.scoring = c->cfg.scoring;
  s.pipeline = c->cfg.pipeline;
  s.req = reinterpret_cast<GReq<R> *>(c->d_req);
  s.keyidx = c->d_keyidx;
  s.req_cap = c->d_req ? static_cast<unsigned long long>(c->cfg.stack_capacity) : 0ull;
  s.mode = c->cfg.mode;
  s.K_bulk = c->cfg.steps_per_claim;
  s.K_tail = c->cfg.tail_steps_per_claim;
  s.tail_threshold = static_cast<unsigned long long>(c->cfg.tail_threshold);
  s.low_water = static_cast<unsigned long long>(c->cfg.mode == GV_ONE_EVENT_PER_LAUNCH ? 1 : c->cfg.refill_low_water);
  s.batch = static_cast<unsigned long long>(c->cfg.refill_batch);
  s.max_gen = static_cast<unsigned long long>(c->cfg.max_generations);
  s.n_mat = static_cast<int>(c->mats.size());
  s.xs_bytes = static_cast<unsigned>(c->xs_bytes);
  s.zb_bytes = static_cast<unsigned>(c->zb_bytes);
  s.smem_req_off = static_cast<unsigned>(c->req_off);
  s.smax_off = static_cast<unsigned>(c->smax_off);
  s.rec_off = static_cast<unsigned>(c->rec_off);
  s.smem_lk_off = static_cast<unsigned>(c->lk_off);
  s.local_stack = c->cfg.local_stack;
  s.smax_bytes = static_cast<unsigned>(c->smax_bytes);
  return s;
}

// The gate at the end of every body of the device-side generation loop: it
// keeps the loop running while the transport is not done.  The loop cannot
// outrun its budget: after max_iter bodies the gate records GV_ERR_TIMEOUT,
// marks the transport done and ends the loop (the generation budget itself
// ends it earlier through plan_next).
__global__ void loop_gate_kernel(Ctl *ctl, cudaGraphConditionalHandle h, unsigned long long max_iter) {
  const unsigned long long it = ++ctl->loop_iter;
  int stop = ctl->plan.done;
  if (!stop && it >= max_iter) {
    if (ctl->status == 0) ctl->status = GV_ERR_TIMEOUT;
    ctl->plan.done = 1;
    stop = 1;
  }
  cudaGraphSetConditional(h, stop ? 0u : 1u);
}

// Puts the persisting-L2 window on every kernel node of g.
cudaError_t set_l2_window(const Ctx *c, cudaGraph_t g) {
  size_t nn = 0;
  cudaError_t e = cudaGraphGetNodes(g, nullptr, &nn);
  std::vector<cudaGraphNode_t> nodes(nn);
  if (e == cudaSuccess && nn) e = cudaGraphGetNodes(g, nodes.data(), &nn);
  cudaKernelNodeAttrValue v{};
  v.accessPolicyWindow.base_ptr = c->d_bins;
  v.accessPolicyWindow.num_bytes = c->l2_window;
  v.accessPolicyWindow.hitRatio = 1.0f;
  v.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
  v.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
  for (size_t i = 0; e == cudaSuccess && i < nn; ++i) {
    cudaGraphNodeType ty;
    e = cudaGraphNodeGetType(nodes[i], &ty);
    if (e == cudaSuccess && ty == cudaGraphNodeTypeKernel)
      e = cudaGraphKernelNodeSetAttribute(nodes[i], cudaKernelNodeAttributeAccessPolicyWindow, &v);
  }
  return e;
}

// The generations of one graph body, recorded on the (capturing) stream.
template <typename R> cudaError_t record_generations(Ctx *c) {
  const DevState<R> *S = reinterpret_cast<const DevState<R> *>(c->d_state);
  if (c->cfg.pipeline) {
    for (int i = 0; i < c->cfg.generations_per_graph; ++i) {
      along_kernel<R><<<c->grid, c->cfg.block_size, c->smem_bytes, c->stream>>>(S, i & 1);
      interact_kernel<R><<<c->grid_b, 256, 0, c->stream>>>(S, i & 1);
    }
    return cudaGetLastError();
  }
  const StepFn<R> step = pick_step_kernel<R>(c);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  for (int i = 0; i < c->cfg.generations_per_graph; ++i) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(c->grid);
    lc.blockDim = dim3(c->cfg.block_size);
    lc.dynamicSmemBytes = c->smem_bytes;
    lc.stream = c->stream;
    lc.attrs = attr;
    lc.numAttrs = (c->cfg.pdl && i > 0) ? 1 : 0;  // overlap with the previous generation's tail
    const int parity = i & 1;
    const cudaError_t e = cudaLaunchKernelEx(&lc, step, parity);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The transport as one graph: a device-side while loop whose body runs
// generations_per_graph generations and then the gate, so the host launches
// once and waits once, and no body starts after the plan that ends the
// transport (the rest of its own body returns at once).
template <typename R> int capture_loop_graph(Ctx *c) {
  cudaGraph_t outer = nullptr;
  if (cudaGraphCreate(&outer, 0) != cudaSuccess) return GV_ERR_CUDA;
  cudaGraphConditionalHandle h;
  cudaGraphNodeParams np = {};
  cudaGraphNode_t node;
  if (cudaGraphConditionalHandleCreate(&h, outer, 1u, cudaGraphCondAssignDefault) != cudaSuccess) {
    cudaGraphDestroy(outer);
    return GV_ERR_CUDA;
  }
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = h;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  if (cudaGraphAddNode(&node, outer, nullptr, nullptr, 0, &np) != cudaSuccess) {
    cudaGraphDestroy(outer);
    return GV_ERR_CUDA;
  }
  cudaGraph_t body = np.conditional.phGraph_out[0];
  if (cudaStreamBeginCaptureToGraph(c->stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) !=
      cudaSuccess) {
    cudaGraphDestroy(outer);
    return GV_ERR_CUDA;
  }
  cudaError_t e = record_generations<R>(c);
  const unsigned long long max_iter =
      static_cast<unsigned long long>(c->cfg.max_generations) / c->cfg.generations_per_graph + 2;
  if (e == cudaSuccess) {
    loop_gate_kernel<<<1, 1, 0, c->stream>>>(c->d_ctl, h, max_iter);
    e = cudaGetLastError();
  }
  cudaGraph_t captured = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(c->stream, &captured);
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess && c->l2_window) e = set_l2_window(c, body);
  if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph, outer, 0);
  cudaGraphDestroy(outer);
  if (e != cudaSuccess) {
    c->graph = nullptr;
    return GV_ERR_CUDA;
  }
  c->loop_graph = 1;
  return GV_OK;
}

template <typename R> int capture_graph(Ctx *c) {
  if (c->graph) return GV_OK;
  c->loop_graph = 0;
  if (c->cfg.device_loop && capture_loop_graph<R>(c) == GV_OK) return GV_OK;
  cudaGetLastError();  // no conditional nodes in this runtime: generations looped by the host
  cudaGraph_t g = nullptr;
  CK(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
  cudaError_t e = record_generations<R>(c);
  const cudaError_t e2 = cudaStreamEndCapture(c->stream, &g);
  if (e == cudaSuccess) e = e2;
  if (e == cudaSuccess && c->l2_window) e = set_l2_window(c, g);  // the window rides on every step launch
  if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph, g, 0);
  if (g) cudaGraphDestroy(g);
  if (e != cudaSuccess) c->graph = nullptr;
  return e == cudaSuccess ? GV_OK : GV_ERR_CUDA;
}

// Whether the kernels may accumulate into the caller's buffer in place: this
// GPU's own memory, and aligned for the atomics.
bool is_own_device_ptr(const void *p, int device) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice && a.device == device && reinterpret_cast<uintptr_t>(p) % 8 == 0;
}

bool is_device_ptr(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// Completes the transport in flight (if any): waits for its last copy, then
// fills the caller's result record from the pinned control block.
int finish_pending(Ctx *c) {
  if (!c->pend.active) return c->last_status;
  c->pend.active = false;
  CK(cudaEventSynchronize(c->ev_out));
  const Ctl &h = *c->h_ctl;
  double kernel_ms = c->pend.kernel_ms;
  long long launches = c->pend.launches;
  if (c->pend.timed_loop) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, c->t0, c->t1));
    kernel_ms = ms;
    launches += static_cast<long long>(h.loop_iter) * (c->cfg.generations_per_graph * (c->cfg.pipeline ? 2 : 1) + 1);
  }
  c->launches = launches;
  const int status = h.status;
  gv_result *res = c->pend.res;
  if (res) {
    for (int i = 0; i < 16; ++i) res->counters[i] = h.counters[i];
    res->counters[GV_C_GENERATIONS] = h.gen;
    res->counters[15] = h.live_peak;
    res->status = status;
    res->kernel_ms = kernel_ms;
  }
  c->last_status = status;
  return status;
}

template <typename R>
int run_transport(Ctx *c, const gv_primary *p, long long n, long long first_event, long long n_events,
                  unsigned long long seed, cudaStream_t user, gv_result *res) {
  CK(cudaSetDevice(c->device));
  const int nsub = c->nsub;
  const size_t ncell = static_cast<size_t>(c->geo.n_layers) * c->geo.nx_cells * c->geo.ny_cells;
  const size_t evlive_bytes = (sizeof(unsigned) * n_events + 7) / 8 * 8;  // cleared in 8-byte words
  if (static_cast<size_t>(n_events) > c->ev_cap) {
    cudaFree(c->d_edep);
    cudaFree(c->d_escape);
    cudaFree(c->d_evcnt);
    cudaFree(c->d_evlive);
    cudaFree(c->d_evcost);
    c->d_edep = nullptr;
    c->d_escape = nullptr;
    c->d_evcnt = nullptr;
    c->d_evlive = nullptr;
    c->d_evcost = nullptr;
    c->ev_cap = 0;
    if (cudaMalloc(&c->d_edep, sizeof(double) * n_events * nsub) != cudaSuccess ||
        cudaMalloc(&c->d_escape, sizeof(double) * n_events) != cudaSuccess ||
        cudaMalloc(&c->d_evcnt, sizeof(unsigned long long) * n_events * GV_NCOUNT) != cudaSuccess ||
        cudaMalloc(&c->d_evlive, evlive_bytes) != cudaSuccess ||
        cudaMalloc(&c->d_evcost, sizeof(unsigned long long) * n_events) != cudaSuccess)
      return GV_ERR_OOM;
    c->ev_cap = n_events;
  }
  // the automatic events-in-flight cap of a batched transport budgets every
  // event by its own primaries (start_kernel, plan_next)
  const bool cost_cap = c->cfg.max_events_in_flight < 0 && c->cfg.mode == GV_BATCHED && n > 0;
  if (cost_cap && static_cast<size_t>(n) + 1 > c->pcost_cap) {
    cudaFree(c->d_pcost);
    c->d_pcost = nullptr;
    c->pcost_cap = 0;
    if (cudaMalloc(&c->d_pcost, sizeof(unsigned long long) * (n + 1)) != cudaSuccess) return GV_ERR_OOM;
    c->pcost_cap = static_cast<size_t>(n) + 1;
  }
  if (ncell && !c->d_cell) {
    if (cudaMalloc(&c->d_cell, sizeof(double) * ncell) != cudaSuccess) return GV_ERR_OOM;
  }
  const bool dev_prim = is_device_ptr(p);
  std::vector<unsigned> order;
  if (c->cfg.mode == GV_ONE_EVENT_PER_LAUNCH || !dev_prim) {
    if (static_cast<size_t>(n) > c->prim_cap) {
      cudaFree(c->d_prim);
      cudaFree(c->d_order);
      c->d_prim = nullptr;
      c->d_order = nullptr;
      if (cudaMalloc(&c->d_prim, sizeof(gv_primary) * n) != cudaSuccess ||
          cudaMalloc(&c->d_order, sizeof(unsigned) * n) != cudaSuccess)
        return GV_ERR_OOM;
      c->prim_cap = n;
    }
  }
  // the work stream waits for whatever the caller queued before
  CK(cudaEventRecord(c->ev_in, user));
  CK(cudaStreamWaitEvent(c->stream, c->ev_in, 0));
  const gv_primary *dp = p;
  std::vector<gv_primary> hp;
  if (!dev_prim) {
    CK(cudaMemcpyAsync(c->d_prim, p, sizeof(gv_primary) * n, cudaMemcpyHostToDevice, c->stream));
    dp = c->d_prim;
  }
  if (c->cfg.mode == GV_ONE_EVENT_PER_LAUNCH) {
    if (dev_prim) {
      hp.resize(n);
      CK(cudaMemcpyAsync(hp.data(), p, sizeof(gv_primary) * n, cudaMemcpyDeviceToHost, c->stream));
      CK(cudaStreamSynchronize(c->stream));
    }
    const gv_primary *src = dev_prim ? hp.data() : p;
    order.resize(n);
    for (long long i = 0; i < n; ++i) order[i] = static_cast<unsigned>(i);
    std::stable_sort(order.begin(), order.end(), [src](unsigned a, unsigned b) { return src[a].event < src[b].event; });
    CK(cudaMemcpyAsync(c->d_order, order.data(), sizeof(unsigned) * n, cudaMemcpyHostToDevice, c->stream));
  }
  // tallies in this GPU's memory are accumulated in place
  double *const edep = is_own_device_ptr(res->edep, c->device) ? res->edep : c->d_edep;
  double *const escape = res->escape_E && is_own_device_ptr(res->escape_E, c->device) ? res->escape_E : c->d_escape;
  double *const cell = ncell && res->cell_edep && is_own_device_ptr(res->cell_edep, c->device) ? res->cell_edep : c->d_cell;
  const bool evc = c->cfg.per_event_counts != 0 && res->event_counts;
  unsigned long long *const evcnt = evc && is_own_device_ptr(res->event_counts, c->device)
                                        ? reinterpret_cast<unsigned long long *>(res->event_counts)
                                        : c->d_evcnt;
  Clear clear = {};
  clear.add(edep, sizeof(double) * n_events * nsub);
  clear.add(escape, sizeof(double) * n_events);
  clear.add(c->d_evlive, evlive_bytes);
  if (ncell && res->cell_edep) clear.add(cell, sizeof(double) * ncell);
  if (evc) clear.add(evcnt, sizeof(unsigned long long) * n_events * GV_NCOUNT);
  if (cost_cap) clear.add(c->d_evcost, sizeof(unsigned long long) * n_events);
  DevState<R> s = make_state<R>(c);
  s.prim = dp;
  s.order = c->cfg.mode == GV_ONE_EVENT_PER_LAUNCH ? c->d_order : nullptr;
  s.n_prim = static_cast<unsigned>(n);
  s.n_events = static_cast<unsigned>(n_events);
  s.ev_base = static_cast<unsigned>(first_event);
  s.edep = edep;
  s.cell = (ncell && res->cell_edep) ? cell : nullptr;
  s.escape = escape;
  s.evcnt = evc ? evcnt : nullptr;
  s.evlive = c->d_evlive;
  s.max_in_flight = static_cast<int>(std::min<long long>(c->cfg.max_events_in_flight, 0x7fffffffll));
  s.pcost = cost_cap ? c->d_pcost : nullptr;
  s.evcost = cost_cap ? c->d_evcost : nullptr;
  s.seed_lo = static_cast<unsigned>(seed);
  s.seed_hi = static_cast<unsigned>(seed >> 32);
  DevState<R> *const S = reinterpret_cast<DevState<R> *>(c->d_state);
  // the graph first: what follows is then enqueued without a gap
  int rc = capture_graph<R>(c);
  if (rc) return rc;
  StateSlot<R> slot(c->device, c->stream);  // held until every launch below is queued
  const unsigned scan = cost_cap ? static_cast<unsigned>(std::min<long long>((n + kPrepThreads - 1) / kPrepThreads, kScanBlocks)) : 0u;
  unsigned long long words = 0;
  for (int k = 0; k < clear.count; ++k) words += clear.n[k];
  const unsigned grid = std::max(scan, static_cast<unsigned>(std::min<unsigned long long>(words / (4 * kPrepThreads) + 1, 4 * c->sm_count)));
  prep_kernel<R><<<grid, kPrepThreads, 0, c->stream>>>(s, S, clear, c->d_part, scan);
  CK(slot.take(S));
  if (cost_cap) {
    start_kernel<R><<<scan, kPrepThreads, 0, c->stream>>>(S, c->d_pcost, c->d_part, scan);
  } else {
    if (s.max_in_flight < 0) {
      CK(cudaMemsetAsync(&c->d_ctl->emax_bits, 0, sizeof(unsigned), c->stream));
      if (n > 0) prim_emax_kernel<R><<<static_cast<int>(std::min<long long>((n + 255) / 256, 4 * c->sm_count)), 256, 0,
                                       c->stream>>>(S);
    }
    init_kernel<R><<<1, 1, 0, c->stream>>>(S);
  }
  CK(cudaGetLastError());
  long long launches = cost_cap ? 2 : (s.max_in_flight < 0 && n > 0) ? 3 : 2;
  double kernel_ms = 0.0;
  if (c->loop_graph) {  // one launch: the device-side loop runs until the transport is done
    CK(cudaEventRecord(c->t0, c->stream));
    CK(cudaGraphLaunch(c->graph, c->stream));
    CK(cudaEventRecord(c->t1, c->stream));
  } else {  // the host relaunches the generation graph until the plan says done
    int between = 1;
    for (;;) {
      CK(cudaEventRecord(c->t0, c->stream));
      for (int i = 0; i < between; ++i) CK(cudaGraphLaunch(c->graph, c->stream));
      CK(cudaEventRecord(c->t1, c->stream));
      launches += static_cast<long long>(between) * c->cfg.generations_per_graph * (c->cfg.pipeline ? 2 : 1);
      CK(cudaMemcpyAsync(c->h_ctl, c->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
      CK(cudaStreamSynchronize(c->stream));
      float ms = 0.f;
      CK(cudaEventElapsedTime(&ms, c->t0, c->t1));
      kernel_ms += ms;
      if (c->h_ctl->plan.done) break;
      between = std::min(between * 2, 64);
    }
  }
  // the control block and the tallies follow on the work stream; the
  // caller's stream waits for them
  CK(cudaMemcpyAsync(c->h_ctl, c->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
  if (res->edep != edep)
    CK(cudaMemcpyAsync(res->edep, c->d_edep, sizeof(double) * n_events * nsub, cudaMemcpyDefault, c->stream));
  if (res->escape_E && res->escape_E != escape)
    CK(cudaMemcpyAsync(res->escape_E, c->d_escape, sizeof(double) * n_events, cudaMemcpyDefault, c->stream));
  if (res->cell_edep && ncell && res->cell_edep != cell)
    CK(cudaMemcpyAsync(res->cell_edep, c->d_cell, sizeof(double) * ncell, cudaMemcpyDefault, c->stream));
  if (evc && evcnt == c->d_evcnt)
    CK(cudaMemcpyAsync(res->event_counts, c->d_evcnt, sizeof(long long) * n_events * GV_NCOUNT, cudaMemcpyDefault,
                       c->stream));
  CK(cudaEventRecord(c->ev_out, c->stream));
  CK(cudaStreamWaitEvent(user, c->ev_out, 0));
  c->pend.active = true;
  c->pend.res = res;
  c->pend.launches = launches;
  c->pend.kernel_ms = kernel_ms;
  c->pend.timed_loop = c->loop_graph != 0;
  if (c->cfg.blocking || !c->loop_graph) return finish_pending(c);
  return GV_OK;
}

}  // namespace

// ====================================================================== C ABI
extern "C" {

int gv_default_config(gv_config *cfg) {
  if (!cfg) return GV_ERR_BAD_ARG;
  cfg->precision = GV_MIXED;
  cfg->mode = GV_BATCHED;
  // measured on 2000 x 10 GeV e- in Pb/polystyrene (GB300), the budgets on an
  // earlier form of the kernels: the basketizing kernel with block claims, 2
  // blocks of 256 per SM, up to 3 along-steps per basket round for electrons
  // and positrons and 5 for photons (8 would take 3 % less time in mixed
  // precision now, one 10 GeV shower 8 %, and 1.4 % more in FP64), one round
  // per claim
  cfg->block_size = 256;
  cfg->blocks_per_sm = 2;
  cfg->steps_per_claim = 1;
  cfg->tail_steps_per_claim = 4;
  cfg->tail_threshold = 1ll << 15;
  cfg->stack_capacity = 1ll << 23;
  cfg->refill_low_water = 1ll << 21;
  cfg->refill_batch = 1ll << 14;
  cfg->generations_per_graph = 16;
  cfg->max_generations = 1ll << 20;
  cfg->per_event_counts = 0;
  cfg->process_sort = 1;
  cfg->max_events_in_flight = -1;
  cfg->claim_chunks = 0;
  cfg->along_steps = 3;
  cfg->along_steps_photon = 5;
  cfg->scoring = 0;
  cfg->l2_persist = 0;
  cfg->pipeline = 0;
  cfg->local_stack = 1;
  cfg->pdl = 1;
  cfg->device_loop = 1;
  cfg->blocking = 0;
  return GV_OK;
}

int gv_setup(void **ctx_out, const gv_material *mats, int n_mats, const gv_layers *geo, const gv_cuts *cuts,
             const gv_config *cfg) {
  if (!ctx_out) return GV_ERR_BAD_ARG;
  *ctx_out = nullptr;
  int rc = validate(mats, n_mats, geo, cuts);
  if (rc) return rc;
  gv_config c;
  gv_default_config(&c);
  if (cfg) c = *cfg;
  rc = validate_cfg(c);
  if (rc) return rc;
  if (geo->field_T != 0.0 && c.scoring != 0) return GV_ERR_BAD_ARG;  // no merged-scoring field kernel
  Ctx *x = new Ctx();
  x->cfg = c;
  x->mats.assign(mats, mats + n_mats);
  x->geo = *geo;
  x->cuts = *cuts;
  x->nsub = geo->n_layers * geo->n_sub;
  x->zb.resize(x->nsub + 1);
  x->smat.resize(x->nsub);
  double z = 0.0;
  x->zb[0] = 0.0;
  for (int l = 0; l < geo->n_layers; ++l)
    for (int j = 0; j < geo->n_sub; ++j) {
      const int k = l * geo->n_sub + j;
      z += geo->sub_thick_cm[j];
      x->zb[k + 1] = z;
      x->smat[k] = static_cast<unsigned char>(geo->sub_mat[j]);
    }
  if (cudaGetDevice(&x->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&x->sm_count, cudaDevAttrMultiProcessorCount, x->device) != cudaSuccess) {
    delete x;
    return GV_ERR_CUDA;
  }
  if (cudaMalloc(&x->d_zb, sizeof(double) * (x->nsub + 1)) != cudaSuccess ||
      cudaMalloc(&x->d_smat, x->nsub) != cudaSuccess ||
      cudaMemcpy(x->d_zb, x->zb.data(), sizeof(double) * (x->nsub + 1), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(x->d_smat, x->smat.data(), x->nsub, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaStreamCreateWithFlags(&x->stream, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&x->ev_in, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&x->ev_out, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreate(&x->t0) != cudaSuccess || cudaEventCreate(&x->t1) != cudaSuccess) {
    gv_destroy(x);
    return GV_ERR_CUDA;
  }
  *ctx_out = x;
  return GV_OK;
}

int gv_build_tables(void *ctx) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c) return GV_ERR_BAD_ARG;
  if (c->tables) return GV_OK;
  std::string err;
  int rc = build_host_tables(c->mats.data(), static_cast<int>(c->mats.size()), c->cuts, &c->ht, &err);
  if (rc) return rc;
  rc = c->cfg.precision == GV_FP64 ? prepare_device<double>(c) : prepare_device<float>(c);
  if (rc) return rc;
  c->tables = true;
  return GV_OK;
}

int gv_transport_events(void *ctx, const gv_primary *p, long long n, long long first_event, long long n_events,
                        unsigned long long seed, void *stream, gv_result *res) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c || (!p && n > 0) || n < 0 || n_events < 1 || n > 0xffffffffll || first_event < 0 ||
      first_event + n_events > 0xffffffffll)
    return GV_ERR_BAD_ARG;
  if (!c->tables) return GV_ERR_NO_TABLES;
  if (!res || !res->edep) return GV_ERR_BAD_ARG;
  if (res->event_counts && !c->cfg.per_event_counts) return GV_ERR_BAD_ARG;
  if (!is_device_ptr(p)) {
    for (long long i = 0; i < n; ++i)
      if (p[i].type < 0 || p[i].type > 2 || p[i].event < static_cast<unsigned long long>(first_event) ||
          p[i].event - static_cast<unsigned long long>(first_event) >= static_cast<unsigned long long>(n_events) ||
          !(p[i].E_MeV >= 0))
        return GV_ERR_BAD_ARG;
  }
  finish_pending(c);  // the previous transport of this context completes first
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return c->cfg.precision == GV_FP64 ? run_transport<double>(c, p, n, first_event, n_events, seed, s, res)
                                     : run_transport<float>(c, p, n, first_event, n_events, seed, s, res);
}

int gv_transport(void *ctx, const gv_primary *p, long long n, long long n_events, unsigned long long seed,
                 void *stream, gv_result *res) {
  return gv_transport_events(ctx, p, n, 0, n_events, seed, stream, res);
}

int gv_sync(void *ctx, void *stream) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c) return GV_ERR_BAD_ARG;
  const int rc = finish_pending(c);
  if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return GV_ERR_CUDA;
  return rc;
}

long long gv_last_launches(void *ctx) {
  Ctx *c = static_cast<Ctx *>(ctx);
  return c ? c->launches : -1;
}

void gv_destroy(void *ctx) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c) return;
  if (c->stream) cudaStreamSynchronize(c->stream);
  c->pend.active = false;  // a result not collected by gv_sync stays unfilled
  if (c->graph) cudaGraphExecDestroy(c->graph);
  if (c->l2_window) {  // release the persisting lines and the set-aside taken at setup
    cudaCtxResetPersistingL2Cache();
    cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, c->l2_old_limit);
  }
  cudaFree(c->d_xs);
  cudaFree(c->d_inv_node);
  cudaFree(c->d_bins);
  cudaFree(c->d_smax);
  cudaFree(c->d_zb);
  cudaFree(c->d_smat);
  cudaFree(c->d_queues);
  cudaFree(c->d_ctl);
  cudaFree(c->d_state);
  cudaFree(c->d_edep);
  cudaFree(c->d_cell);
  cudaFree(c->d_escape);
  cudaFree(c->d_evcnt);
  cudaFree(c->d_evlive);
  cudaFree(c->d_evcost);
  cudaFree(c->d_pcost);
  cudaFree(c->d_part);
  cudaFree(c->d_prim);
  cudaFree(c->d_order);
  cudaFree(c->d_req);
  cudaFree(c->d_keyidx);
  if (c->h_ctl) cudaFreeHost(c->h_ctl);
  if (c->ev_in) cudaEventDestroy(c->ev_in);
  if (c->ev_out) cudaEventDestroy(c->ev_out);
  if (c->t0) cudaEventDestroy(c->t0);
  if (c->t1) cudaEventDestroy(c->t1);
  if (c->stream) cudaStreamDestroy(c->stream);
  delete c;
}

const char *gv_strerror(int code) {
  switch (code) {
    case GV_OK: return "ok";
    case GV_ERR_BAD_ARG: return "bad argument";
    case GV_ERR_NO_TABLES: return "tables not built";
    case GV_ERR_OOM: return "device allocation failed";
    case GV_ERR_STACK_FULL: return "track queue overflow";
    case GV_ERR_TIMEOUT: return "generation budget exhausted";
    case GV_ERR_NUMERIC: return "non-finite track state";
    case GV_ERR_CUDA: return "CUDA runtime error";
    case GV_ERR_INTERNAL: return "internal check failed";
    default: return "unknown error";
  }
}

}  // extern "C"

// exported for the element-wise entry points (gv_unit.cu)
namespace gv {
int ctx_views(void *ctx, int *precision, View<float> *vf, View<double> *vd) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c) return GV_ERR_BAD_ARG;
  if (!c->tables) return GV_ERR_NO_TABLES;
  *precision = c->cfg.precision;
  if (c->cfg.precision == GV_FP64) *vd = make_view<double>(c);
  else *vf = make_view<float>(c);
  return GV_OK;
}
int ctx_nmat(void *ctx) { return static_cast<int>(static_cast<Ctx *>(ctx)->mats.size()); }
}  // namespace gv

// ====================================================================== transport without allocation
// Some callers must not have this library allocate device memory while they
// run: a host framework that hands out all of a GPU's memory from its own
// pools under a fixed budget (as large event-processing frameworks do) cannot
// let a library call cudaMalloc behind its back, and cudaMalloc/cudaFree also
// synchronise the whole device and may fail or stall under memory pressure.
// gv_transport_static runs the same step kernel as gv_transport, but keeps
// every piece of scratch memory it needs -- the double-buffered track queues,
// the generation control block, the kernel's state record and the per-event
// live-track counts -- in the file-scope array below, sized once for a modest
// maximum.  The array is part of the module image: every GPU that loads
// libgv holds it until the process exits.
namespace {
constexpr long long kStaticCap = 1 << 16;         // tracks per particle type and buffer
constexpr long long kStaticMaxEvents = 1 << 16;   // events per call
constexpr size_t kStaticCtlOff = 0;
constexpr size_t kStaticStateOff = 4096;
constexpr size_t kStaticEvliveOff = 12288;
constexpr size_t kStaticQueueOff = kStaticEvliveOff + sizeof(unsigned) * kStaticMaxEvents;
constexpr size_t kStaticQueueBytes = 6 * static_cast<size_t>(kStaticCap) * track_bytes<float>();
constexpr size_t kStaticBytes = kStaticQueueOff + kStaticQueueBytes;  // 25,440,256 bytes
static_assert(sizeof(Ctl) <= kStaticStateOff - kStaticCtlOff, "control block does not fit");
static_assert(sizeof(DevState<float>) <= kStaticEvliveOff - kStaticStateOff, "state does not fit");
static_assert(kStaticCap % 16 == 0, "queue parts must stay 256-byte aligned");
}  // namespace

static __device__ __align__(256) unsigned char g_gv_static_scratch[kStaticBytes];

namespace {

// Device address of the scratch array on the current device.  Host code only
// sees a host-side stand-in under the array's name, so the address is asked
// of the runtime, with the device current, on every call: a cached address
// would outlive a device reset or a new primary context.
int static_scratch(unsigned char **base) {
  void *p = nullptr;
  if (cudaGetSymbolAddress(&p, g_gv_static_scratch) != cudaSuccess || !p) {
    cudaGetLastError();
    return GV_ERR_CUDA;
  }
  *base = static_cast<unsigned char *>(p);
  return GV_OK;
}

// the state record travels as a kernel argument, so no staging copy is needed
__global__ void static_state_kernel(DevState<float> s, DevState<float> *dst) {
  *dst = s;
  s.ctl->emax_bits = 0u;
}

}  // namespace

extern "C" int gv_transport_static(void *ctx, const gv_primary *prim, long long n, long long n_events,
                                   unsigned long long seed, void *stream, double *edep, double *escape_E,
                                   unsigned long long *counters) {
  Ctx *c = static_cast<Ctx *>(ctx);
  if (!c || n < 0 || (n > 0 && !prim) || n_events < 1 || !edep || !escape_E || !counters) return GV_ERR_BAD_ARG;
  if (!c->tables) return GV_ERR_NO_TABLES;
  if (c->cfg.precision != GV_MIXED) return GV_ERR_BAD_ARG;  // the array is sized for the mixed layout
  if (c->geo.field_T != 0.0) return GV_ERR_BAD_ARG;          // its kernel is the field-free one
  if (n_events > kStaticMaxEvents || n > 0xffffffffll) return GV_ERR_BAD_ARG;
  if (cudaSetDevice(c->device) != cudaSuccess) return GV_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  {  // the call waits on the host between launches: a capturing stream cannot take it
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
      cudaGetLastError();
      return GV_ERR_CUDA;
    }
    if (cs != cudaStreamCaptureStatusNone) return GV_ERR_BAD_ARG;
  }
  if ((n > 0 && !is_device_ptr(prim)) || !is_device_ptr(edep) || !is_device_ptr(escape_E)) return GV_ERR_BAD_ARG;
  finish_pending(c);  // a gv_transport of this context still in flight completes first
  unsigned char *base = nullptr;
  int rc = static_scratch(&base);
  if (rc) return rc;
  // the basketizing kernel (with the arithmetic of the one without, which this
  // call ran before: the same showers at half the time)
  bool opts = (c->cuts.process_mask & (GV_P_MSC | GV_P_INTEGRAL)) != 0;
  for (int m = 0; m < kNModel; ++m) opts = opts || c->cuts.reject_min_MeV[m] < 1e30;
  const StepFn<float> step = opts ? step_kernel<float, true, false, false, true, false, true>
                                  : step_kernel<float, true, false, false, false, false, true>;
  const int block = c->cfg.block_size;
  const size_t lk_off = (c->req_off + static_cast<size_t>(ReqStore<float>::kBytes) * block + 31) / 32 * 32;
  const size_t smem = lk_off + static_cast<size_t>(LocalStack<float>::kBytes) * block;
  if (allow_shared(reinterpret_cast<const void *>(step), c->device, smem) != cudaSuccess) return GV_ERR_CUDA;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, reinterpret_cast<const void *>(step), block, smem) != cudaSuccess ||
      occ < 1)
    return GV_ERR_CUDA;
  const int grid = c->sm_count * std::min(occ, c->cfg.blocks_per_sm);
  DevState<float> s = make_state<float>(c);
  s.qmem = base + kStaticQueueOff;
  s.q_bytes = TrackLayout<float>::queue_bytes(kStaticCap);
  s.q_part = TrackLayout<float>::part_bytes(kStaticCap);
  s.capacity = static_cast<unsigned long long>(kStaticCap);
  s.ctl = reinterpret_cast<Ctl *>(base + kStaticCtlOff);
  s.view.status = &s.ctl->status;
  s.mode = GV_BATCHED;
  s.chunk = block;
  s.adaptive_chunk = 1;
  s.grid = grid;
  s.pipeline = 0;
  s.smem_lk_off = static_cast<unsigned>(lk_off);
  s.low_water = static_cast<unsigned long long>(kStaticCap / 4);
  s.batch = std::min<unsigned long long>(s.batch, 64);
  s.max_in_flight = -1;  // automatic: capacity / (0.15 per MeV of the most energetic primary + 64)
  s.prim = prim;
  s.order = nullptr;
  s.n_prim = static_cast<unsigned>(n);
  s.n_events = static_cast<unsigned>(n_events);
  s.edep = edep;
  s.cell = nullptr;
  s.escape = escape_E;
  s.evcnt = nullptr;
  s.evlive = reinterpret_cast<unsigned *>(base + kStaticEvliveOff);
  s.ev_base = 0;
  s.seed_lo = static_cast<unsigned>(seed);
  s.seed_hi = static_cast<unsigned>(seed >> 32);
  DevState<float> *S = reinterpret_cast<DevState<float> *>(base + kStaticStateOff);
  // Held until the call returns.  The scratch array is touched only from here
  // on: a call of another thread may use it until then, and clearing its event
  // counts would keep its in-flight cap from ever admitting the next event.
  StateSlot<float> slot(c->device, st);
  // the tallies and the event counts start from zero on every call
  if (slot.wait() != cudaSuccess || cudaMemsetAsync(edep, 0, sizeof(double) * n_events * c->nsub, st) != cudaSuccess ||
      cudaMemsetAsync(escape_E, 0, sizeof(double) * n_events, st) != cudaSuccess ||
      cudaMemsetAsync(base + kStaticEvliveOff, 0, sizeof(unsigned) * n_events, st) != cudaSuccess)
    return GV_ERR_CUDA;
  static_state_kernel<<<1, 1, 0, st>>>(s, S);
  if (slot.take(S) != cudaSuccess) return GV_ERR_CUDA;
  if (n > 0)
    prim_emax_kernel<float><<<static_cast<int>(std::min<long long>((n + 255) / 256, 4 * c->sm_count)), 256, 0, st>>>(S);
  init_kernel<float><<<1, 1, 0, st>>>(S);
  if (cudaGetLastError() != cudaSuccess) return GV_ERR_CUDA;
  // Generations go out in batches, and the next batch before the host has seen
  // whether the last one ended the transport: the GPU does not wait for the
  // host, and at most two batches of generations return at once.
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(block);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  lc.attrs = attr;
  constexpr int kBatch = 12;  // even: a batch starts at parity 0
  const cudaEvent_t seen[2] = {c->ev_in, c->ev_out};
  for (int batch = 0;; ++batch) {
    for (int i = 0; i < kBatch; ++i) {
      lc.numAttrs = (c->cfg.pdl && i > 0) ? 1 : 0;
      const int parity = i & 1;
      if (cudaLaunchKernelEx(&lc, step, parity) != cudaSuccess) return GV_ERR_CUDA;
    }
    if (cudaMemcpyAsync(c->h_ctl, s.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaEventRecord(seen[batch & 1], st) != cudaSuccess)
      return GV_ERR_CUDA;
    if (batch == 0) continue;
    if (cudaEventSynchronize(seen[(batch - 1) & 1]) != cudaSuccess) return GV_ERR_CUDA;
    if (*const_cast<volatile int *>(&c->h_ctl->plan.done)) break;  // final once set, whichever batch it came with
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return GV_ERR_CUDA;
  for (int i = 0; i < 16; ++i) counters[i] = c->h_ctl->counters[i];
  counters[GV_C_GENERATIONS] = c->h_ctl->gen;
  counters[15] = c->h_ctl->live_peak;
  c->last_status = c->h_ctl->status;  // what a later gv_sync on this context reports
  return c->last_status;
}
