// Kernels of one simulation step (see moss_device.cuh for the layout).
#pragma once

#include <type_traits>

#include "moss_device.cuh"

namespace moss {

// Programmatic dependent launch: a kernel of a step may start while the one
// before it drains.  grid_wait returns once that kernel has finished and its
// writes are visible (at once for an ordinary launch); grid_release lets the
// next kernel start when every block of this one has called it or ended.  It
// is called after grid_wait, so a kernel that runs early knows that all but
// the kernel directly before it have finished.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// entrant list of a lane for this step's tag (-1 if empty or stale)
__device__ __forceinline__ int list_head(const unsigned long long* head, int lane, int tag) {
    const unsigned long long h = head[lane];
    return (int)(h >> 32) == tag ? (int)(unsigned)(h & 0xffffffffull) : -1;
}

// append entrant q to the list of `lane`
__device__ __forceinline__ void list_push(unsigned long long* head, int32_t* enext, int lane, int q, int tag) {
    const unsigned long long prev =
        atomicExch(&head[lane], ((unsigned long long)(unsigned)tag << 32) | (unsigned)q);
    enext[q] = (int)(prev >> 32) == tag ? (int)(unsigned)(prev & 0xffffffffull) : -1;
}

// ---------------------------------------------------------------------------
// the tile (k_place's or k_lanescan's) that holds lane l, whose segment starts
// at off
template <typename Real>
__device__ __forceinline__ int tile_key(const Ctx<Real>& c, int off, int l) {
    return (int)(((long long)off * c.slot_w + (long long)c.lane_w * l) >> c.tile_shift);
}

// a vehicle leaves / enters lane l: counted for the lane and for its tile
template <typename Real>
__device__ __forceinline__ void count_leave(const Ctx<Real>& c, int l) {
    atomicAdd(&c.leave[l], 1);
    atomicAdd(&c.tile_delta[tile_key(c, c.slot_w ? c.cur.off[l] : 0, l)], -1);
}
template <typename Real>
__device__ __forceinline__ void count_enter(const Ctx<Real>& c, int l) {
    atomicAdd(&c.enter[l], 1);
    atomicAdd(&c.tile_delta[tile_key(c, c.slot_w ? c.cur.off[l] : 0, l)], 1);
}

// a vehicle goes from lane l to lane m.  Within a scan tile nothing grows:
// nearly all lane changes, whose atomics on a few words would otherwise queue
// up when many vehicles change at once (18,098 of 67,769 in a step, 7 scan
// tiles: k_decide 49.4 -> 32.6 us).  The tiles of k_place are many, and the
// comparison would wait there for both lanes' offsets.
template <typename Real>
__device__ __forceinline__ void count_move(const Ctx<Real>& c, int l, int m) {
    if (c.slot_w) {
        count_leave(c, l);
        count_enter(c, m);
        return;
    }
    atomicAdd(&c.leave[l], 1);
    atomicAdd(&c.enter[m], 1);
    const int from = l >> c.tile_shift, to = m >> c.tile_shift;
    if (from != to) {
        atomicAdd(&c.tile_delta[from], -1);
        atomicAdd(&c.tile_delta[to], 1);
    }
}

// A k_decide block's lane-change candidates: their indices in the candidate
// list, resolved by the block once its run is done.  The first cand_cap of
// them (a schedule value, at most CAND_LOCAL) are listed in shared memory,
// the rest in the run's own part of cand_late, which starts at the run's
// first slot (a run has at most one candidate per slot).
constexpr int CAND_LOCAL = 256;
struct CandLocal {
    int n;
    int run[2];  // slots of the run
    int idx[CAND_LOCAL];
};

template <typename Real>
__device__ __forceinline__ void note_candidate(const Ctx<Real>& c, CandLocal& cl, int k) {
    const int j = atomicAdd(&cl.n, 1);
    if (j < c.cand_cap) cl.idx[j] = k;
    else c.cand_late[cl.run[0] + j - c.cand_cap] = k;
}

// ---------------------------------------------------------------------------
// Departure insertion (R18) for start lane l: the head of its FIFO enters at
// s = 0, v = 0 when due and the snapshot's rearmost vehicle on the lane has
// s - len >= s0 (or the lane is empty).
template <typename Real>
__device__ void insert_departure(const Ctx<Real>& c, int l, int tag) {
    const int h = c.q_head[l];
    if (h >= c.q_off[l + 1]) return;
    const int vid = c.q_ids[h];
    const LaneInfo ls = c.lane[l];
    if (ls.flags & LF_RESTRICTED) return;  // no departure onto a restricted lane (R25)
    const int sc = ls.scen;
    if (c.scen_ctl[sc]) return;  // a frozen or retiring slot
    const long long t = c.scen_step[sc];
    if ((long long)c.dep[vid] > t) return;
    const int b = c.cur.off[l], e = c.cur.off[l + 1];
    int fl = F_INSERTED;
    if (e > b) {
        const Real sr = c.cur.a[e - 1].s;
        const Real g = sr - c.len - c.s0;
        const Real scl = sr > Real(1) ? sr : Real(1);
        if (rabs(g) < c.band * scl) fl |= F_FLAGGED;
        if (!(g >= Real(0))) return;
    }
    const int q = warp_claim(&c.cnt->n_ent);
    const int2 rs = c.route_span[vid];
    const int r0 = rs.x, r1 = rs.y - 1;
    int nl = -1;
    if (r0 < r1) nl = jl_toward(c, c.lane[l], c.routes[r0 + 1]);  // -1: no access from this lane (R27)
    RecA<Real> A;
    A.s = Real(0); A.v = Real(0); A.id = vid; A.lane = l;
    RecB B;
    B.v0f = c.v0f[vid]; B.rptr = r0; B.rlast = r1; B.nl = nl;
    c.ea[q] = A;
    c.eb[q] = B;
    count_enter(c, l);
    list_push(c.head, c.enext, l, q, tag);
    c.q_head[l] = h + 1;
    c.vstatus[vid] = 1;
    c.vflags[vid] = int((t & 0xFFFFFF) << 8) | fl;
    long long* M = c.metrics + (long long)sc * M_NFIELDS;
    atomicAdd((unsigned long long*)&M[M_INSERTED], 1ull);
    atomicAdd((unsigned long long*)&M[M_CUR_ACTIVE], 1ull);
    if (fl & F_FLAGGED) atomicAdd((unsigned long long*)&M[M_FLAGGED], 1ull);
}

// ---------------------------------------------------------------------------
// Ballistic update with clamps (R12, R13), transfer and arrival (R17), and the
// outputs of one vehicle (slot i) driving on lane `nlane` (record ni) with
// lane kinematics la.  Returns 1 if the vehicle leaves its lane's segment.
template <typename Real>
__device__ __forceinline__ int integrate_emit(const Ctx<Real>& c, MetricAcc& acc, int i, const RecA<Real>& E,
                                              const RecB& EB, const LaneAcc<Real>& la, int nlane, int fl,
                                              bool own_overlap, long long t, int sc, int tag) {
    const int lane = E.lane;
    const Real s = E.s, v = E.v, a = la.a, dt = c.dt;
    Real vn = v + a * dt, disp;
    if (vn >= Real(0)) {
        disp = v * dt + Real(0.5) * a * dt * dt;
    } else {
        disp = -v * v / (Real(2) * a);
        vn = Real(0);
    }
    if (la.has_leader) { const Real cl = gt(la.gap, Real(0)) ? la.gap : Real(0); if (gt(disp, cl)) disp = cl; }
    if (la.stop) { const Real cl = gt(la.stop_gap, Real(0)) ? la.stop_gap : Real(0); if (gt(disp, cl)) disp = cl; }
    LaneInfo ni = c.lane[nlane];
    Real sn = s + disp;
    if (la.stop && sn > Real(ni.L)) sn = Real(ni.L);
    // The overshoot past the lane end is taken as disp - (L - s): L - s is
    // exact for s >= L/2 (Sterbenz), so the position on the next lane does
    // not lose the bits of L.
    int rptr = EB.rptr;
    const int rlast = EB.rlast;
    int nl = la.nl;
    bool arrived = false;
    Real ex = disp - (Real(ni.L) - s);  // distance beyond the end of nlane
    if (!la.stop) {
        for (int iter = 0;;) {
            const Real Ll = Real(ni.L);
            const bool road = ni.lo >= 0;
            if (within(ex, c.band, at_least_1(Ll))) fl |= F_FLAGGED;
            if (road && rptr == rlast) {
                if (ex >= Real(0)) arrived = true;
                break;
            }
            if (!(ex > Real(0))) break;
            if (++iter > 4 || nl < 0) { atomicOr(c.err, ERR_TRANSFER); sn = Ll; break; }
            sn = ex;
            fl |= F_TRANSFER;
            nlane = nl;
            ni = c.lane[nlane];
            if (road) {
                nl = ni.hi;  // entered a junction lane: next is its target road lane
            } else {
                rptr += 1;  // entered the next road
                // -1 on the last road, or without access from this lane (R27)
                nl = (rptr < rlast) ? jl_toward(c, ni, c.routes[rptr + 1]) : -1;
            }
            ex = sn - Real(ni.L);
        }
    }
    if (arrived) fl |= F_ARRIVED;
    acc.upd += 1;
    acc.spd += speed_fixed(vn);
    if (fl & F_FLAGGED) acc.flg += 1;
    if (fl & F_CHANGED) acc.lc += 1;
    if (own_overlap) acc.ovl += 1;
    if (fl) c.vflags[E.id] = int((t & 0xFFFFFF) << 8) | fl;
    if (arrived) {
        c.code[i] = C_ARRIVE;
        c.vstatus[E.id] = 2;
        acc.arr += 1;
        acc.tt += (t + 1) - (long long)c.dep[E.id];
        count_leave(c, lane);
        long long* M = c.metrics + (long long)sc * M_NFIELDS;
        atomicAdd((unsigned long long*)&M[M_CUR_ACTIVE], (unsigned long long)(-1ll));
        atomicAdd((unsigned long long*)&M[M_CUR_ARRIVED], 1ull);
        return 1;
    }
    if (nlane == lane) {
        c.code[i] = C_STAY;
        SV<Real> w;
        w.s = sn; w.v = vn;
        c.stay[i] = w;
        return 0;
    }
    c.code[i] = C_MOVE;
    count_move(c, lane, nlane);
    const int q = warp_claim(&c.cnt->n_ent);
    RecA<Real> A;
    A.s = sn; A.v = vn; A.id = E.id; A.lane = nlane;
    RecB B;
    B.v0f = EB.v0f; B.rptr = rptr; B.rlast = rlast; B.nl = nl;
    c.ea[q] = A;
    c.eb[q] = B;
    list_push(c.head, c.enext, nlane, q, tag);
    return 1;
}

// a candidate's kinematics on its target lane
template <typename Real>
__device__ __forceinline__ LaneAcc<Real> target_acc(const Ctx<Real>& c, const RecA<Real>& E, const RecB& EB,
                                                    const Decision<Real>& D) {
    const LaneInfo ti = c.lane[D.tl];
    RecA<Real> TLr;
    TLr.s = Real(0); TLr.v = Real(0);
    const bool lead = D.gp > c.cur.off[D.tl];
    if (lead) TLr = c.cur.a[D.gp - 1];
    return accel_on_lane<Real, true>(c, ti, E.s, E.v, free_term(E.v, Real(EB.v0f) * Real(ti.vmax)), lead,
                                               TLr.s, TLr.v, D.nlt, EB.rptr, EB.rlast);
}

// ---------------------------------------------------------------------------
// A lane-change candidate leaves its decision for the end of the run: a record in the
// candidate list, linked into the list of its target gap.
template <typename Real>
__device__ __forceinline__ void list_candidate(const Ctx<Real>& c, int i, const RecA<Real>& E, const RecB& EB,
                                               int sc, const Decision<Real>& D, int tag, CandLocal& cl) {
    const LaneAcc<Real> T = target_acc(c, E, EB, D);
    Cand<Real> C;
    C.E = E; C.EB = EB;
    C.slot = i; C.gap = D.gp + D.tl;
    C.bits = (D.dir > 0 ? CB_RIGHT : 0) | (D.flag ? CB_FLAG : 0) | (D.own.has_leader ? CB_LEADER : 0) |
             (D.own.stop ? CB_STOP : 0) | (D.own.overlap ? CB_OVERLAP : 0) | (T.has_leader ? CB_TLEADER : 0) |
             (T.stop ? CB_TSTOP : 0) | (T.overlap ? CB_TOVERLAP : 0);
    C.nl = D.own.nl; C.tnl = T.nl; C.scen = sc; C.pad = 0;
    C.u = D.u; C.scale = D.scale;
    C.a = D.own.a; C.lgap = D.own.gap; C.sgap = D.own.stop_gap;
    C.ta = T.a; C.tlgap = T.gap; C.tsgap = T.stop_gap;
    const int k = warp_claim(&c.cnt->n_cand);
    const unsigned long long prev =
        atomicExch(&c.gap_head[C.gap], ((unsigned long long)(unsigned)tag << 32) | (unsigned)k);
    C.next = (int)(prev >> 32) == tag ? (int)(unsigned)(prev & 0xffffffffull) : -1;
    c.cands[k] = C;
    note_candidate(c, cl, k);
}

// ---------------------------------------------------------------------------
// Resolution of lane-change candidate k.  Conflict rule R9: a candidate
// conflicts with the candidates that enter the same lane from the other side
// into the same gap
// (the other members of its gap list with the opposite direction); the
// larger utility wins, ties to the smaller id.  Both sides compare the same
// stored utilities, so the outcome is consistent.  Then the update on the
// target lane (granted) or with the stored own-lane kinematics (lost).
template <typename Real>
__device__ __forceinline__ void resolve_one(const Ctx<Real>& c, MetricAcc& acc, int k, int nc, int tag) {
    {
        const Cand<Real> C = c.cands[k];
        const int i = C.slot;
        const RecA<Real> E = C.E;
        const RecB EB = C.EB;
        const int lane = E.lane;
        const int dir = (C.bits & CB_RIGHT) ? 1 : -1;
        const int sc = C.scen;
        if (sc != acc.scen) {
            macc_flush_thread(acc, c.metrics);
            macc_reset(acc, sc);
        }
        const long long t = c.scen_step[sc];
        int fl = F_CANDIDATE | ((C.bits & CB_FLAG) ? F_FLAGGED : 0);
        bool granted = true;
        const unsigned long long h = c.gap_head[C.gap];
        int q = (int)(h >> 32) == tag ? (int)(unsigned)(h & 0xffffffffull) : -1;
        for (int guard = 0; q >= 0; q = c.cands[q].next) {
            if (++guard > nc) { atomicOr(c.err, ERR_RANGE); break; }
            if (q == k) continue;
            const int rbits = c.cands[q].bits;
            if (((rbits & CB_RIGHT) ? 1 : -1) == dir) continue;  // same side: no conflict
            const Real ru = c.cands[q].u, rs = c.cands[q].scale;
            const Real sc2 = C.scale > rs ? C.scale : rs;
            if (rabs(C.u - ru) < c.band * sc2) fl |= F_FLAGGED;
            if (!(C.u > ru || (C.u == ru && E.id < c.cands[q].E.id))) granted = false;
        }
        LaneAcc<Real> la;
        int nlane = lane;
        if (granted) {
            fl |= F_CHANGED;
            nlane = lane + dir;
            la.a = C.ta; la.gap = C.tlgap; la.stop_gap = C.tsgap; la.nl = C.tnl;
            la.has_leader = (C.bits & CB_TLEADER) != 0;
            la.stop = (C.bits & CB_TSTOP) != 0;
            la.overlap = (C.bits & CB_TOVERLAP) != 0;
        } else {
            fl |= F_CONFLICT_LOST;
            la.a = C.a; la.gap = C.lgap; la.stop_gap = C.sgap; la.nl = C.nl;
            la.has_leader = (C.bits & CB_LEADER) != 0;
            la.stop = (C.bits & CB_STOP) != 0;
            la.overlap = (C.bits & CB_OVERLAP) != 0;
        }
        integrate_emit(c, acc, i, E, EB, la, nlane, fl, (C.bits & CB_OVERLAP) != 0, t, sc, tag);
    }
}

// ---------------------------------------------------------------------------
// The vehicles whose attempt draw passed are queued in shared memory, one
// queue of 64 entries per warp, and MOBIL runs over a warp's queue 32 at a
// time: a warp otherwise carries the whole MOBIL evaluation of any one of
// its lanes while the others idle.
template <typename Real>
struct MobilQueue {
    Real a[2 * TILE], gap[2 * TILE], sgap[2 * TILE];  // own-lane kinematics (LaneAcc)
    int i[2 * TILE], lane[2 * TILE], bits[2 * TILE], nl[2 * TILE];
    float u_lc[2 * TILE], u_dir[2 * TILE];
    int n[TILE / 32];
};

// MOBIL and the update of queued vehicle k (the snapshot and lane records
// are read again; the own-lane part comes from the queue)
template <typename Real, bool Groups>
__device__ __forceinline__ void mobil_finish(const Ctx<Real>& c, const MobilQueue<Real>& q, int k, int n,
                                             MetricAcc& acc, int tag, CandLocal& cl) {
    const int i = q.i[k], lane = q.lane[k];
    const RecA<Real> E = c.cur.a[i];
    const RecB EB = c.cur.b[i];
    const LaneInfo li = c.lane[lane];
    RecA<Real> OLr = no_rec<Real>(), OFr = no_rec<Real>();
    float of_v0f = 0.0f;
    if (i > 0) OLr = c.cur.a[i - 1];
    if (i + 1 < n) {
        OFr = c.cur.a[i + 1];
        of_v0f = c.cur.b[i + 1].v0f;
    }
    LaneAcc<Real> own;
    own.a = q.a[k]; own.gap = q.gap[k]; own.stop_gap = q.sgap[k];
    const int bits = q.bits[k];
    own.has_leader = bits & 1; own.stop = (bits >> 1) & 1; own.overlap = (bits >> 2) & 1;
    own.nl = q.nl[k];
    const int sc = li.scen;
    if (sc != acc.scen) {
        macc_flush_thread(acc, c.metrics);
        macc_reset(acc, sc);
    }
    const Decision<Real> D = decide_mobil<Real, Groups>(c, E, EB, li, OLr, OFr, of_v0f, own, q.u_lc[k], q.u_dir[k]);
    if (D.cand) {
        list_candidate(c, i, E, EB, sc, D, tag, cl);
        return;
    }
    const long long t = c.scen_step[sc];
    integrate_emit(c, acc, i, E, EB, own, lane, D.flag ? F_FLAGGED : 0, own.overlap != 0, t, sc, tag);
}

// ---------------------------------------------------------------------------
// The wide form of the decision, taken in FP64: a pass over up to TILE slots
// in three phases of the whole block.  (1) Each vehicle: own lane and attempt
// draw; those that go on enter one queue of the block.  (2) A thread for each
// side of each queued vehicle and one for its old follower.  (3) A thread per
// queued vehicle: the choice, the conflicts and the update.  A run whose
// vehicles pass through the queue in one round settles its conflicts here, in
// shared memory; longer runs leave their candidates for the end of the run.
//
// An FP64 instruction occupies an SM for 16 cycles whether one thread of the
// warp is active or all are, so what counts is the number of warps that run
// each part: against a queue per warp and one thread for the whole of a
// vehicle's MOBIL, the vehicles of all warps are packed and the second side
// costs only those that have one.  30x30 grid of 100,000 trips in FP64:
// k_decide 157 -> 61 us a step between its events.  In FP32, where latency
// bounds the kernel, the exchange and the three barriers cost more than that
// saves (4x4 to 30x30 grids 0 to 8% slower, 350,000 trips in 12 slots 46 -> 54
// us a step): the form above.
template <typename Real>
struct WideQueue {
    Real a[TILE], gap[TILE], sgap[TILE];          // own-lane kinematics (LaneAcc)
    Real f[TILE];                                 // the ego's free term on its lane
    Real a_old[TILE], at_old[TILE];               // mobil_old
    Real t_ego[2 * TILE], t_new[2 * TILE], t_anew[2 * TILE];  // mobil_side of the left (2k) and right (2k + 1) side
    Real cu[TILE], cscale[TILE];                  // candidates: utility, flag scale
    int gp[2 * TILE], tnl[2 * TILE], tbits[2 * TILE];  // tbits: 1 valid, 2 feasible, 4 flag
    int i[TILE], lane[TILE], bits[TILE], nl[TILE];     // bits: 1 leader, 2 stop, 4 overlap, 8 mandatory change
    int ckey[TILE], cid[TILE];                    // candidates: gap key, id (right: ~id)
    float u_lc[TILE], u_dir[TILE];
    short item[2 * TILE];                         // sides to evaluate
    int n, n_items;
};

// phase 1: vehicle i enters the queue
template <typename Real>
__device__ __forceinline__ void wide_push(WideQueue<Real>& q, int i, int lane, const LaneInfo& li,
                                          const OwnPart<Real>& P) {
    const int k = warp_claim(&q.n);
    q.i[k] = i; q.lane[k] = lane;
    q.a[k] = P.own.a; q.gap[k] = P.own.gap; q.sgap[k] = P.own.stop_gap;
    q.bits[k] = (P.own.has_leader ? 1 : 0) | (P.own.stop ? 2 : 0) | (P.own.overlap ? 4 : 0) | (P.mand ? 8 : 0);
    q.f[k] = P.f;
    q.nl[k] = P.own.nl;
    q.u_lc[k] = P.u_lc; q.u_dir[k] = P.u_dir;
    q.tbits[2 * k] = 0; q.tbits[2 * k + 1] = 0;
    if (P.mand) return;
    if (lane - 1 >= li.lo) q.item[warp_claim(&q.n_items)] = (short)(2 * k);
    if (lane + 1 < li.hi) q.item[warp_claim(&q.n_items)] = (short)(2 * k + 1);
}

// phase 2: side x & 1 of queued vehicle x >> 1
template <typename Real, bool Groups>
__device__ __forceinline__ void wide_side(const Ctx<Real>& c, WideQueue<Real>& q, int x) {
    const int k = x >> 1, i = q.i[k], lane = q.lane[k], tl = lane + ((x & 1) ? 1 : -1);
    const RecA<Real> E = c.cur.a[i];
    const RecB EB = c.cur.b[i];
    const LaneInfo ti = c.lane[tl];
    // a side is a lane of the road that is not restricted from passing (R25)
    if (ti.flags & LF_RESTRICTED) return;
    const int next_road = EB.nl >= 0 ? c.lane[EB.nl].road : -1;
    const LaneInfo li = c.lane[lane];
    const SideTerms<Real> S = mobil_side<Real, Groups, true>(c, E, EB, li.jb, ti, tl, next_road, q.f[k], li.vmax);
    q.t_ego[x] = S.at_ego; q.t_new[x] = S.at_new; q.t_anew[x] = S.a_new;
    q.gp[x] = S.gp; q.tnl[x] = S.nlt;
    q.tbits[x] = (S.valid ? 1 : 0) | (S.feas ? 2 : 0) | (S.flag ? 4 : 0);
}

// phase 2: the old follower of queued vehicle k
template <typename Real>
__device__ __forceinline__ void wide_old(const Ctx<Real>& c, WideQueue<Real>& q, int k, int n) {
    if (q.bits[k] & 8) return;
    const int i = q.i[k];
    const RecA<Real> E = c.cur.a[i];
    RecA<Real> OLr = no_rec<Real>(), OFr = no_rec<Real>();
    float of_v0f = 0.0f;
    if (i > 0) OLr = c.cur.a[i - 1];
    if (i + 1 < n) {
        OFr = c.cur.a[i + 1];
        of_v0f = c.cur.b[i + 1].v0f;
    }
    Real a_old, at_old;
    mobil_old(c, E, c.lane[q.lane[k]].vmax, OLr, OFr, of_v0f, &a_old, &at_old);
    q.a_old[k] = a_old; q.at_old[k] = at_old;
}

// phase 3: queued vehicle k (k < 0: none; every thread of the block calls it)
template <typename Real, bool Groups>
__device__ __forceinline__ void wide_finish(const Ctx<Real>& c, WideQueue<Real>& q, int k, bool local, MetricAcc& acc,
                                            int tag, CandLocal& cl) {
    Decision<Real> D;
    D.cand = 0; D.flag = 0;
    RecA<Real> E;
    RecB EB;
    LaneAcc<Real> T;
    int sc = 0, i = 0, lane = 0;
    if (k >= 0) {
        i = q.i[k]; lane = q.lane[k];
        E = c.cur.a[i];
        EB = c.cur.b[i];
        const LaneInfo li = c.lane[lane];
        sc = li.scen;
        LaneAcc<Real> own;
        const int bits = q.bits[k];
        own.a = q.a[k]; own.gap = q.gap[k]; own.stop_gap = q.sgap[k]; own.nl = q.nl[k];
        own.has_leader = bits & 1; own.stop = (bits >> 1) & 1; own.overlap = (bits >> 2) & 1;
        if (sc != acc.scen) {
            macc_flush_thread(acc, c.metrics);
            macc_reset(acc, sc);
        }
        if (Groups && (bits & 8)) {
            D = decide_mandatory(c, i, E, EB, li, own);
        } else {
            D = no_decision(own);
            Real u[2] = {Real(0), Real(0)}, scl[2] = {Real(0), Real(0)};
            int feas[2] = {0, 0};
#pragma unroll
            for (int sd = 0; sd < 2; ++sd) {
                const int x = 2 * k + sd, tb = q.tbits[x];
                if (!(tb & 1)) continue;
                if (tb & 4) D.flag = 1;
                feas[sd] = (tb >> 1) & 1;
                side_utility(c, q.t_ego[x], q.t_new[x], q.t_anew[x], own.a, q.a_old[k], q.at_old[k], &u[sd], &scl[sd]);
            }
            const int sd = mobil_choose(c, u, scl, feas, q.u_lc[k], q.u_dir[k], D);
            if (sd >= 0) {
                D.tl = lane + (sd ? 1 : -1);
                D.gp = q.gp[2 * k + sd];
                D.nlt = q.tnl[2 * k + sd];
            }
        }
        if (D.cand) {
            if (local) {
                cl.idx[atomicAdd(&cl.n, 1)] = k;
                q.ckey[k] = D.gp + D.tl;
                q.cid[k] = D.dir > 0 ? ~E.id : E.id;
                q.cu[k] = D.u; q.cscale[k] = D.scale;
                T = target_acc(c, E, EB, D);
            } else {
                list_candidate(c, i, E, EB, sc, D, tag, cl);
            }
        } else {
            integrate_emit(c, acc, i, E, EB, own, lane, D.flag ? F_FLAGGED : 0, own.overlap != 0, c.scen_step[sc], sc,
                           tag);
        }
    }
    if (!local) return;
    __syncthreads();
    if (k < 0 || !D.cand) return;
    // the conflict rule R9, as in resolve_one
    int fl = F_CANDIDATE | (D.flag ? F_FLAGGED : 0);
    bool granted = true;
    const int key = D.gp + D.tl;
    for (int j = 0; j < cl.n; ++j) {
        const int r = cl.idx[j];
        if (r == k || q.ckey[r] != key) continue;
        const int rid = q.cid[r];
        if ((rid < 0) == (D.dir > 0)) continue;  // same side: no conflict
        const Real ru = q.cu[r], rs = q.cscale[r];
        const Real sc2 = D.scale > rs ? D.scale : rs;
        if (rabs(D.u - ru) < c.band * sc2) fl |= F_FLAGGED;
        if (!(D.u > ru || (D.u == ru && E.id < (rid < 0 ? ~rid : rid)))) granted = false;
    }
    fl |= granted ? F_CHANGED : F_CONFLICT_LOST;
    integrate_emit(c, acc, i, E, EB, granted ? T : D.own, granted ? D.tl : lane, fl, D.own.overlap != 0, c.scen_step[sc],
                   sc, tag);
}

// ---------------------------------------------------------------------------
// k_decide: blocks [0, n_work) take runs of slots of the current snapshot, 256
// at a time (one vehicle per thread); blocks [n_work, gridDim) run the
// insertion and add up the phase pressures of the max-pressure junctions.
// Per vehicle: the own-lane acceleration and the attempt draw, MOBIL if the
// draw passed (from the warp's queue in FP32, the block's in FP64), then the
// update; lane-change candidates are finished at the end of the block's run,
// or with the queue where one round of it holds the run (FP64).
// Groups: the network has lane groups (some road has a turn that not all of
// its lanes serve), so the mandatory changes of R27 can occur; without them
// that path is not compiled in.
// MOSS_DECIDE_MIN_BLOCKS: resident blocks per SM the register budget targets.
#ifndef MOSS_DECIDE_MIN_BLOCKS
#define MOSS_DECIDE_MIN_BLOCKS 5
#endif
#ifndef MOSS_DECIDE_MIN_BLOCKS_FP64
#define MOSS_DECIDE_MIN_BLOCKS_FP64 3
#endif
template <typename Real>
__host__ __device__ constexpr bool wide_form() { return sizeof(Real) == 8; }
template <typename Real>
__host__ __device__ constexpr int decide_min_blocks() {
    return sizeof(Real) == 8 ? MOSS_DECIDE_MIN_BLOCKS_FP64 : MOSS_DECIDE_MIN_BLOCKS;
}
// The run of slots [*sb, *se) of work block vb of n_work.  A vehicle on a
// road lane costs about twice one on a junction lane (MOBIL, longer
// neighbour searches), so the runs split the snapshot by weight: run_w (a
// schedule choice, fitted by default) per road-lane slot, 1 per junction-lane
// slot, from the current lane offsets at the lane ranges of each scenario
// (road lanes first, then junction lanes), when blocks take four tiles or
// more each; then each end moves back to the start of its road.  The runs
// are contiguous and cover every slot.  s_run: shared, the run on return.
__device__ __forceinline__ long long run_weight(int a, int b, int e, int wq) {
    return (long long)wq * (b - a) + 256ll * (e - b);
}
// road-lane slot weight x256 of this step's runs: the schedule's fixed value,
// else the fit of the previous step's block times (1 before any)
template <typename Real>
__device__ __forceinline__ int run_wq(const Ctx<Real>& c) {
    if (c.run_w > 0) return 256 * c.run_w;
    const int f = c.cnt->run_wq;
    return f > 0 ? f : 256;
}

// First slot of the road whose lane holds `slot` (a junction-lane slot
// stays where it is): the block runs begin and end there, so the vehicles of
// a road, and with them every rival of a lane-change candidate, lie in one run.
template <typename Real>
__device__ __forceinline__ int road_start(const Ctx<Real>& c, int slot, int n) {
    if (slot <= 0) return 0;
    if (slot >= n) return n;
    const int lane = c.cur.a[slot].lane;
    if ((unsigned)lane >= (unsigned)c.n_lanes) return slot;  // reported by the decision
    const int lo = c.lane[lane].lo;
    return lo >= 0 ? c.cur.off[lo] : slot;
}

template <typename Real>
__device__ __forceinline__ void decide_run(const Ctx<Real>& c, int n, int n_work, int vb, int* s_run, int* sb,
                                           int* se) {
    const int n_tiles = (n + TILE - 1) / TILE;
    if (n_tiles < 4 * n_work) {
        // a few tiles per block: equal slot counts (weights would leave
        // blocks idle at this granularity)
        if (threadIdx.x < 2) s_run[threadIdx.x] = road_start(c, (int)((long long)(vb + (int)threadIdx.x) * n / n_work), n);
    } else if (threadIdx.x < 32) {
        const int wl = threadIdx.x;
        const int wq = run_wq(c);
        long long tot = 0;
        for (int k0 = 0; k0 < c.n_scen; k0 += 32) {
            long long w = 0;
            if (k0 + wl < c.n_scen) {
                const int4 L = c.scen_lanes[k0 + wl];
                w = run_weight(c.cur.off[L.x], c.cur.off[L.y], c.cur.off[L.z], wq);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            tot += w;
        }
        // weights T0, T1 -> slots (scan of the scenarios' weights)
        const long long T[2] = {tot * vb / n_work, tot * (vb + 1) / n_work};
        int slot[2] = {-1, -1};
        long long carry = 0;
        for (int k0 = 0; k0 < c.n_scen && (slot[0] < 0 || slot[1] < 0); k0 += 32) {
            const int k = k0 + wl;
            int a = 0, b = 0, e = 0;
            long long w = 0;
            if (k < c.n_scen) {
                const int4 L = c.scen_lanes[k];
                a = c.cur.off[L.x]; b = c.cur.off[L.y]; e = c.cur.off[L.z];
                w = run_weight(a, b, e, wq);
            }
            long long P = w;  // inclusive prefix over the chunk
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, P, o);
                if (wl >= o) P += y;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                // the first scenario whose weight reaches past T (m and
                // slot[q] are the same on every lane: the branch is uniform)
                const unsigned m = __ballot_sync(0xffffffffu, k < c.n_scen && carry + P > T[q]);
                if (slot[q] < 0 && m) {
                    const int src = __ffs(m) - 1;
                    const long long local = T[q] - (carry + __shfl_sync(0xffffffffu, P - w, src));
                    const int sa = __shfl_sync(0xffffffffu, a, src), sb = __shfl_sync(0xffffffffu, b, src);
                    const long long wr = (long long)wq * (sb - sa);
                    slot[q] = local < wr ? sa + (int)(local / wq) : sb + (int)((local - wr) / 256);
                }
            }
            carry += __shfl_sync(0xffffffffu, P, 31);
        }
        if (wl == 0) {
            const int s0 = slot[0] < 0 ? n : slot[0], s1 = slot[1] < 0 ? n : slot[1];
            s_run[0] = road_start(c, s0, n);
            s_run[1] = vb == n_work - 1 ? n : road_start(c, s1, n);
        }
    }
    __syncthreads();
    *sb = s_run[0];
    *se = s_run[1];
}

// The work of block vb of nvb (k_decide's grid, or a virtual block of the
// single-launch step): vb < n_work takes a run of slot tiles, the others run
// the insertion and add up the phase pressures of the max-pressure junctions
// (the kernel after it advances those).
template <typename Real, bool Groups>
__device__ __forceinline__ void decide_block(const Ctx<Real>& c, int n_work, int vb, int nvb) {
    constexpr bool Wide = wide_form<Real>();
    const int tag = c.cnt->tag;
    if (vb >= n_work) {
        const int stride = (nvb - n_work) * TILE;
        for (int k = (vb - n_work) * TILE + threadIdx.x; k < c.n_start; k += stride)
            insert_departure(c, c.start_lanes[k], tag);
        if (*c.n_mp > 0)
            for (int k = (vb - n_work) * TILE + threadIdx.x; k < c.n_jj; k += stride) mp_accumulate(c, k);
        return;
    }
    const int n = c.cnt->n_cur;
    // each block takes a contiguous run of slots: a thread's scenario (and so
    // its metric partials) changes rarely, neighbouring lanes stay close, and
    // the run holds whole roads, so the block resolves its own lane-change
    // candidates once its run is done (rule R9: rivals share the road)
    __shared__ CandLocal cl;
    __shared__ typename std::conditional<Wide, WideQueue<Real>, MobilQueue<Real>>::type q;
    __shared__ int s_road;  // road-lane vehicles of the run (for the run-weight fit)
    unsigned long long t_start = 0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_start));
    if (threadIdx.x == 0) { cl.n = 0; s_road = 0; }
    if (vb == 0 && threadIdx.x == 0) c.cnt->n_runs = n_work;
    int n_road = 0;
    int s_beg, s_end;
    decide_run(c, n, n_work, vb, cl.run, &s_beg, &s_end);
    // passes of TILE slots: from a multiple of TILE on, but a run that fits
    // one pass takes one (its first slot rounded down to a line of records)
    const int base = s_end - (s_beg & ~7) <= TILE ? s_beg & ~7 : s_beg / TILE * TILE;
    const int n_pass = s_beg < s_end ? (s_end - base + TILE - 1) / TILE : 0;
    MetricAcc acc;
    macc_reset(acc, -1);
    const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31, qb = warp * 64;
    if constexpr (Wide) {
        if (threadIdx.x == 0) q.n = q.n_items = 0;
        __syncthreads();
    } else {
        if (wl == 0) q.n[warp] = 0;
        __syncwarp();
    }
    bool local = false;  // (wide) the run's conflicts were settled in its only round of the queue
    int rounds = 0;
    for (int pass = 0;; ++pass) {
        const bool last = pass >= n_pass;
        const int i = base + pass * TILE + threadIdx.x;
        if (!last && i >= s_beg && i < s_end) {
            const RecA<Real> E = c.cur.a[i];
            const RecB EB = c.cur.b[i];
            const RecA<Real> OLr = i > 0 ? c.cur.a[i - 1] : no_rec<Real>();
            const int lane = E.lane;
            if ((unsigned)lane >= (unsigned)c.n_lanes) {
                atomicOr(c.err, ERR_RANGE);
            } else {
                const LaneInfo li = c.lane[lane];
                n_road += li.lo >= 0;
                const int sc = li.scen;
                if (sc != acc.scen) {
                    macc_flush_thread(acc, c.metrics);
                    macc_reset(acc, sc);
                }
                const int ctl = c.scen_ctl[sc];
                if (ctl) {
                    // a slot that does not advance: a frozen one keeps its
                    // vehicles as they are, a retiring one removes them
                    if (ctl & SC_RETIRE) {
                        c.code[i] = C_ARRIVE;
                        c.vstatus[E.id] = 2;
                        count_leave(c, lane);
                    } else {
                        c.code[i] = C_STAY;
                        SV<Real> w;
                        w.s = E.s; w.v = E.v;
                        c.stay[i] = w;
                    }
                } else {
                    const long long t = c.scen_step[sc];
                    const OwnPart<Real> P =
                        decide_own<Real, Groups>(c, E, EB, li, OLr, t, c.key0[sc], c.key1[sc], c.veh_base[sc]);
                    int fl = 0;
                    bool cand = false;
                    if constexpr (Wide) {
                        if (P.att) acc.mob += 1;
                        if (P.att || (Groups && P.mand)) {
                            wide_push(q, i, lane, li, P);
                            cand = true;  // finished from the queue
                        }
                    } else if (P.att) {
                        acc.mob += 1;
                        const int k = qb + warp_claim(&q.n[warp]);
                        q.i[k] = i; q.lane[k] = lane;
                        q.a[k] = P.own.a; q.gap[k] = P.own.gap; q.sgap[k] = P.own.stop_gap;
                        q.bits[k] = (P.own.has_leader ? 1 : 0) | (P.own.stop ? 2 : 0) | (P.own.overlap ? 4 : 0);
                        q.nl[k] = P.own.nl;
                        q.u_lc[k] = P.u_lc; q.u_dir[k] = P.u_dir;
                        cand = true;  // finished from the queue
                    } else if (Groups && P.mand) {
                        const Decision<Real> D = decide_mandatory(c, i, E, EB, li, P.own);
                        if (D.cand) {
                            list_candidate(c, i, E, EB, sc, D, tag, cl);
                            cand = true;
                        }
                        fl = D.flag ? F_FLAGGED : 0;
                    }
                    if (!cand) integrate_emit(c, acc, i, E, EB, P.own, lane, fl, P.own.overlap != 0, t, sc, tag);
                }
            }
        }
        if constexpr (Wide) {
            if (last) break;
            __syncthreads();
            // phases 2 and 3 once the queue might not hold the next pass
            const int nq = q.n, ni = q.n_items, ni32 = (ni + 31) & ~31;
            const bool end = pass + 1 == n_pass;
            if (!end && nq + min(TILE, s_end - (base + (pass + 1) * TILE)) <= TILE) {
                __syncthreads();
                continue;
            }
            local = end && rounds == 0;
            ++rounds;
            for (int x = threadIdx.x; x < ni32 + nq; x += TILE) {
                if (x < ni) wide_side<Real, Groups>(c, q, q.item[x]);
                else if (x >= ni32) wide_old(c, q, x - ni32, n);
            }
            __syncthreads();
            wide_finish<Real, Groups>(c, q, (int)threadIdx.x < nq ? (int)threadIdx.x : -1, local, acc, tag, cl);
            __syncthreads();
            if (threadIdx.x == 0) q.n = q.n_items = 0;
            __syncthreads();
            continue;
        } else {
        // MOBIL over the last 32 entries of the warp's queue once it holds
        // 32, and over what is left after the last pass
        __syncwarp();
        const int nq = q.n[warp];
        const int take = last ? nq : (nq >= 32 ? 32 : 0);
        if (take > 0) {
            if (wl < take) mobil_finish<Real, Groups>(c, q, qb + nq - take + wl, n, acc, tag, cl);
            __syncwarp();
            if (wl == 0) q.n[warp] = nq - take;
            __syncwarp();
        }
        if (last) break;
        }
    }
    // the run's lane-change candidates (their rivals are all in this run)
    __syncthreads();
    const int ncl = local ? 0 : cl.n;
    for (int j = threadIdx.x; j < ncl; j += TILE)
        resolve_one(c, acc, j < c.cand_cap ? cl.idx[j] : c.cand_late[s_beg + j - c.cand_cap], c.n_veh, tag);
    if (n_road) atomicAdd(&s_road, n_road);
    macc_flush_block<TILE>(acc, c.metrics);  // (its barriers also complete s_road)
    // the run's statistics for the next step's weight fit (run_fit)
    if (threadIdx.x == 0 && vb < RUNSTAT_MAX) {
        unsigned long long t_end = 0;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_end));
        const long long dt = (long long)(t_end - t_start);
        const int ns = s_end - s_beg;
        c.runstat[vb] = make_int4((int)min(dt, (long long)INT_MAX), s_road, ns - s_road, 1);
    }
}

template <typename Real, bool Groups>
__global__ void __launch_bounds__(TILE, decide_min_blocks<Real>()) k_decide(Ctx<Real> c, int n_work) {
    grid_wait();
    grid_release();
    if (__syncthreads_or(threadIdx.x == 0 ? *c.err & ERR_POISON : 0)) return;
    decide_block<Real, Groups>(c, n_work, blockIdx.x, gridDim.x);
}

// Fit of the cost of a road-lane and a junction-lane vehicle in k_decide
// from this step's work blocks: least squares of run time ~ c_road x (road
// slots) + c_junction x (junction slots) over the runs; the next step splits
// its runs with the weight c_road / c_junction (clamped to [0.5, 4]; the
// previous weight when the fit is degenerate, e.g. no junction vehicles).
// One block (a ticket of k_place); every work run rewrites its entry each
// step.
template <typename Real>
__device__ void run_fit(const Ctx<Real>& c) {
    // FP32 sums of normalised values (slots in thousands, times in units of
    // 100 us): the five sums stay within a few thousand for any run count
    __shared__ float s_sum[5][TILE / 32];
    float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // RR, RJ, JJ, dR, dJ
    const int nr = min(c.cnt->n_runs, RUNSTAT_MAX);
    for (int k = threadIdx.x; k < nr; k += TILE) {
        const int4 r = c.runstat[k];
        if (!r.w) continue;
        const float d = 1e-5f * (float)r.x, R = 1e-3f * (float)r.y, J = 1e-3f * (float)r.z;
        v[0] += R * R; v[1] += R * J; v[2] += J * J; v[3] += d * R; v[4] += d * J;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        float x = v[q];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) s_sum[q][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float t[5];
        for (int q = 0; q < 5; ++q) {
            t[q] = 0.f;
            for (int w = 0; w < TILE / 32; ++w) t[q] += s_sum[q][w];
        }
        int wq = c.cnt->run_wq;
        const float det = t[0] * t[2] - t[1] * t[1];
        if (det > 1e-4f * t[0] * t[2] && t[2] > 0.f) {
            const float cr = (t[3] * t[2] - t[4] * t[1]) / det, cj = (t[0] * t[4] - t[1] * t[3]) / det;
            if (cr > 0.f && cj > 0.f) {
                const float w = fminf(4.f, fmaxf(0.5f, cr / cj));
                wq = (int)(w * 256.f + 0.5f);
            }
        }
        c.cnt_next->run_wq = wq;
    }
}

// ---------------------------------------------------------------------------
// k_place: the lane offsets of the next snapshot, then the snapshot itself.
//
// A tile is a run of whole lanes [tile_cur[t], tile_cur[t+1]) with their
// vehicles, cut where 2 off[l] + PLACE_LANE_W l passes a multiple of
// 1 << tile_shift (the previous step's tiles wrote the cuts).  newsize(l) =
// size(l) - leave(l) + enter(l).  k_decide also counts how each tile grows
// (tile_delta), so the next offset of a tile's first lane is its offset now plus the growth of the
// tiles before it: every tile adds those words up for itself and no tile
// waits for another.  The vehicles of a lane lie in the tile, so a stayer's
// next slot is its own slot plus a per-lane shift, minus the leavers before it
// in the tile, plus the entrants ahead of it.
//
// The entrants of the tile are gathered in shared memory (a lane's list is
// walked once, by the lane's thread), ranked there and counted against the
// stayers eight threads each, side by side: in the flowing traffic of a city
// some lane takes several every step, and every step waits for the worst lane.
// One entrant of a lane after the other, each walking the list again, the
// kernel took 17 to 21 us between its events on cities of 50,000 to 150,000
// trips, so 10 to 12 (a step 29.5 -> 23.5 and 40.8 -> 28.8 us; by slots 26.3
// and 30.8).
//
// Bound by latency: about six dependent memory rounds and four barriers, 6 us
// on the 12x12 grid and 9 on the 30x30 grid of 70,000 vehicles, where the
// scan with look-back and the placement as two kernels took 16 and 15.5.
// Everything the step before wrote (cuts, offsets, records) is loaded before
// grid_wait, past L1: the tail of k_decide covers it.

// entrants of a list (from q on) that are ahead of (s, id); n_in: its length
template <typename Real>
__device__ __forceinline__ int entrants_ahead(const Ctx<Real>& c, int q, Real s, int id, int* n_in = nullptr) {
    int cnt = 0, guard = 0;
    for (; q >= 0; q = c.enext[q]) {
        const RecA<Real> Q = c.ea[q];
        if (ahead(Q.s, Q.id, s, id)) ++cnt;
        if (++guard > c.n_veh) { atomicOr(c.err, ERR_RANGE); break; }
    }
    if (n_in) *n_in = guard;
    return cnt;
}

constexpr int TW = TILE / 32;           // warps per block
constexpr int PLACE_ROUNDS = 16;        // slot rounds whose leaver masks are held at a time
constexpr int PLACE_LANE_W = 4;         // weight of a lane in the tiles, in half-slots (a vehicle: 2)
constexpr int PLACE_SHIFT_MAX = 10;     // a tile takes 1 << 9 or 1 << 10 half-slots
constexpr int PLACE_LANES = (1 << PLACE_SHIFT_MAX) / PLACE_LANE_W;  // lanes of the widest tile
static_assert(PLACE_LANES <= TILE, "a thread per lane");
constexpr int PLACE_ENT = 128;          // entrants that a tile holds in shared memory
template <typename Real>
__host__ __device__ constexpr size_t place_smem() {
    return PLACE_ENT * (sizeof(Real) + 4 * sizeof(int)) + sizeof(int) * (5 * PLACE_LANES + 2);
}

// the clocks of every scenario, one step on (a frozen or retiring one stands
// still; one that reaches its horizon freezes)
template <typename Real>
__device__ __forceinline__ void advance_clocks(const Ctx<Real>& c) {
    for (int s = threadIdx.x; s < c.n_scen; s += TILE) {
        if (c.scen_ctl[s]) continue;
        const long long t = c.scen_step[s] + 1;
        c.scen_step[s] = t;
        if (t == c.stop_at[s]) c.scen_ctl[s] = SC_FROZEN;
    }
}

template <typename Real, bool Pdl>
__device__ __forceinline__ void place_tile(const Ctx<Real>& c, int tile) {
    __shared__ unsigned long long s_wsum[TW];       // per warp: leavers << 32 | next size of its lanes
    __shared__ unsigned s_ball[PLACE_ROUNDS * TW];  // leaver mask of each 32 slots
    __shared__ int s_lp[PLACE_ROUNDS * TW];         // leavers of the tile before them
    __shared__ int s_sum[TW];
    __shared__ int s_ne, s_nel;                     // entrants held here, lanes whose entrants are not
    // (dynamic: with the decision's FP64 queue past what a kernel may declare)
    extern __shared__ __align__(16) unsigned char s_mem[];
    Real* const s_es = reinterpret_cast<Real*>(s_mem);               // [PLACE_ENT] entrants: position,
    int* const s_eid = reinterpret_cast<int*>(s_es + PLACE_ENT);     // id,
    int* const s_eq = s_eid + PLACE_ENT;                             // record (-1: none),
    int* const s_ek = s_eq + PLACE_ENT;                              // lane of the tile,
    int* const s_bh = s_ek + PLACE_ENT;                              // stayers of the lane behind it
    int* const s_nx = s_bh + PLACE_ENT;     // [PLACE_LANES + 1] next offset of a lane
    int* const s_ob = s_nx + PLACE_LANES + 1;  // [PLACE_LANES + 1] its offset
    int* const s_sh = s_ob + PLACE_LANES + 1;  // [PLACE_LANES] next slot - slot of a lane's first vehicle, + leavers before
                                               // the lane
    int* const s_hd = s_sh + PLACE_LANES;   // [PLACE_LANES] entrants of a lane: 0 none; > 0: 1 + (first of them here | how
                                            // many << 9); < 0: ~(their list)
    int* const s_el = s_hd + PLACE_LANES;   // [PLACE_LANES] lanes with a list
    const int tid = threadIdx.x, ln = tid & 31, w = tid >> 5;
    // ---- what the previous step wrote
    const int tag = __ldcg(&c.cnt->tag);
    const int L0 = __ldcg(&c.tile_cur[tile]), L1 = __ldcg(&c.tile_cur[tile + 1]);
    const int S0 = __ldcg(&c.cur.off[L0]), S1 = __ldcg(&c.cur.off[L1]);
    // (a step that reported ERR_RANGE may have left cuts of two steps: this
    // one ends below, past the writes to the arrays above)
    const int m = min(L1 - L0, PLACE_LANES);
    const int l = L0 + tid;  // the thread's lane of the tile (tid < m)
    int o0 = 0, o1 = 0;
    if (tid < m) {
        o0 = __ldcg(&c.cur.off[l]);
        o1 = __ldcg(&c.cur.off[l + 1]);
    }
    int2 al = make_int2(-1, -1);  // id, lane of the first round's record
    int4 ab = make_int4(0, 0, 0, 0);
    if (S0 + tid < S1) {
        al = __ldcg(reinterpret_cast<const int2*>(&c.cur.a[S0 + tid].id));
        ab = __ldcg(reinterpret_cast<const int4*>(&c.cur.b[S0 + tid]));
    }
    if (tid == 0) s_ne = s_nel = 0;
    if (tid < PLACE_ENT) s_eq[tid] = -1;
    __syncthreads();
    if (Pdl) {
        grid_wait();
        grid_release();
    }
    const int poison = tid == 0 ? *c.err & ERR_POISON : 0;
    // ---- lanes: sizes, leavers, entrant lists; prefixes within the warp
    SV<Real> st0;
    int8_t code0 = C_STAY;
    if (S0 + tid < S1) {
        code0 = c.code[S0 + tid];
        st0 = c.stay[S0 + tid];
    }
    int grown = 0;
    for (int p = tid; p < tile; p += TILE) grown += c.tile_delta[p];
    unsigned long long x = 0;
    if (tid < m) {
        const int lv = c.leave[l], en = c.enter[l];
        const unsigned long long h = c.head[l];
        if (lv) c.leave[l] = 0;
        int hd = 0;
        if (en) {
            c.enter[l] = 0;
            if ((int)(h >> 32) == tag) {
                int q = (int)(unsigned)(h & 0xffffffffull);
                const int j = atomicAdd(&s_ne, en);
                if (j + en <= PLACE_ENT) {
                    hd = 1 + (j | en << 9);
                    for (int t = 0; t < en; ++t) {
                        s_eq[j + t] = q;
                        s_ek[j + t] = tid;
                        if (t + 1 < en && (q = c.enext[q]) < 0) { atomicOr(c.err, ERR_RANGE); break; }
                    }
                } else {
                    hd = ~q;
                    s_el[atomicAdd(&s_nel, 1)] = tid;
                }
            }
        }
        s_hd[tid] = hd;
        s_ob[tid] = o0;
        s_ob[tid + 1] = o1;
        x = ((unsigned long long)(unsigned)lv << 32) | (unsigned)(o1 - o0 - lv + en);
    }
    unsigned long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (ln >= o) incl += y;
    }
    if (ln == 31) s_wsum[w] = incl;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) grown += __shfl_xor_sync(0xffffffffu, grown, o);
    if (ln == 0) s_sum[w] = grown;
    // ---- the leavers of the first slot rounds
    const int nr = min((S1 - S0 + TILE - 1) / TILE, PLACE_ROUNDS);
    for (int r = 0; r < nr; ++r) {
        const int i = S0 + r * TILE + tid;
        const int8_t code = r == 0 ? code0 : (i < S1 ? c.code[i] : (int8_t)C_STAY);
        const unsigned b = __ballot_sync(0xffffffffu, code != C_STAY);
        if (ln == 0) s_ball[r * TW + w] = b;
    }
    if (__syncthreads_or(poison)) return;
    unsigned long long wb = 0, tot = 0;
    int prefix = S0;
#pragma unroll
    for (int k = 0; k < TW; ++k) {
        const unsigned long long x = s_wsum[k];
        if (k < w) wb += x;
        tot += x;
        prefix += s_sum[k];
    }
    if (w == TW - 1) {  // leavers before each 32 slots
        int carry = 0;
        for (int k0 = 0; k0 < nr * TW; k0 += 32) {
            const int x = k0 + ln < nr * TW ? __popc(s_ball[k0 + ln]) : 0;
            int incl = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (ln >= o) incl += y;
            }
            if (k0 + ln < nr * TW) s_lp[k0 + ln] = carry + incl - x;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    const unsigned long long ex = wb + incl - x;  // leavers << 32 | next size of the lanes before the thread's
    if (tid < m) {
        const int nx = prefix + (int)(unsigned)(ex & 0xffffffffull);
        c.nxt.off[l] = nx;
        s_nx[tid] = nx;
        s_sh[tid] = nx + (int)(ex >> 32) - o0;
    }
    if (tid == 0) s_nx[m] = prefix + (int)(unsigned)(tot & 0xffffffffull);
    if (tid < PLACE_ENT && s_eq[tid] >= 0) {
        const RecA<Real> Q = c.ea[s_eq[tid]];
        s_es[tid] = Q.s;
        s_eid[tid] = Q.id;
    }
    __syncthreads();
    // ---- the next step's tile cuts and the ends of the snapshot
    if (tid < m) {
        const int q0 = tile_key(c, s_nx[tid], l), q1 = tile_key(c, s_nx[tid + 1], l + 1);
        for (int q = q0 + 1; q <= q1; ++q) c.tile_nxt[q] = l + 1;
        if (l + 1 == c.n_lanes) {
            c.nxt.off[l + 1] = s_nx[tid + 1];
            c.cnt_next->n_cur = s_nx[tid + 1];
            c.tile_nxt[q1 + 1] = l + 1;
        }
    }
    // ---- entrants: eight threads each, four at a time in a warp.  The stayers
    // of a lane keep their order (nobody overtakes within a lane, R13), so the
    // stayers behind an entrant form the rear of the lane's old segment: they
    // are counted from the segment's end, 8 slots per round, up to the first
    // round that holds a stayer ahead of the entrant (entrants join mostly at
    // the rear of a lane: one round).  Stayers ahead = the lane's stayers (its
    // next size minus its entrants) minus those behind.
    const int sub = ln >> 3, sl = ln & 7, ne = min(s_ne, PLACE_ENT), nel = s_nel;
    const auto stayers_behind = [&](bool open, int b, int e, Real s, int id) {
        int bh = 0;
        for (int x0 = e - 1; __any_sync(0xffffffffu, open); x0 -= 8) {
            const int x = x0 - sl;
            bool st = false, ah = false;
            if (open && x >= b) {
                st = c.code[x] == C_STAY;  // (the other loads go out with this one)
                ah = ahead(c.stay[x].s, c.cur.a[x].id, s, id) && st;
            }
            const unsigned mb = (__ballot_sync(0xffffffffu, st && !ah) >> (8 * sub)) & 0xffu;
            const unsigned ma = (__ballot_sync(0xffffffffu, ah) >> (8 * sub)) & 0xffu;
            if (open) bh += __popc(mb);
            if (ma || x0 - 8 < b) open = false;
        }
        return bh;
    };
    for (int j0 = 4 * w; j0 < ne; j0 += 4 * TW) {
        const int j = j0 + sub, q = j < ne ? s_eq[j] : -1;
        int k = 0, id = 0;
        Real s = Real(0);
        RecA<Real> Q;
        RecB QB;
        if (q >= 0) {
            k = s_ek[j]; s = s_es[j]; id = s_eid[j];
            if (sl == 0) { Q = c.ea[q]; QB = c.eb[q]; }
        }
        const int bh = stayers_behind(q >= 0, s_ob[k], s_ob[k + 1], s, id);
        if (q < 0 || sl) continue;
        s_bh[j] = bh;
        const int n = (s_hd[k] - 1) >> 9, f = (s_hd[k] - 1) & 511;
        int pos = s_nx[k + 1] - n - bh;
        for (int t = f; t < f + n; ++t) pos += ahead(s_es[t], s_eid[t], s, id);
        if (pos < s_nx[k] || pos >= s_nx[k + 1] || pos >= c.n_veh) {
            atomicOr(c.err, ERR_RANGE);
        } else {
            c.nxt.a[pos] = Q;
            c.nxt.b[pos] = QB;
        }
    }
    // the lanes whose entrants did not fit, one entrant of a lane after the other
    for (int j0 = 4 * w; j0 < nel; j0 += 4 * TW) {
        int q = -1, k = 0;
        if (j0 + sub < nel) {
            k = s_el[j0 + sub];
            q = ~s_hd[k];
        }
        const int q0 = q;
        int n_in = 0;
        while (__any_sync(0xffffffffu, q >= 0)) {
            RecA<Real> Q;
            Q.s = Real(0); Q.id = 0;
            int nq = -1;
            if (q >= 0) {
                Q = c.ea[q];
                nq = c.enext[q];
            }
            const int bh = stayers_behind(q >= 0, s_ob[k], s_ob[k + 1], Q.s, Q.id);
            if (q >= 0) {
                if (sl == 0) {
                    int len = 0;
                    const int ent = entrants_ahead(c, q0, Q.s, Q.id, &len);
                    const int pos = s_nx[k + 1] - len - bh + ent;
                    if (pos < s_nx[k] || pos >= s_nx[k + 1] || pos >= c.n_veh) {
                        atomicOr(c.err, ERR_RANGE);
                    } else {
                        c.nxt.a[pos] = Q;
                        c.nxt.b[pos] = c.eb[q];
                    }
                }
                q = nq;
                if (++n_in > c.n_veh) { atomicOr(c.err, ERR_RANGE); q = -1; }
            }
        }
    }
    __syncthreads();
    // ---- stayers
    int lcarry = 0;  // leavers of the rounds before the held ones
    for (int r0 = 0; S0 + r0 * TILE < S1; r0 += PLACE_ROUNDS) {
        const int nh = min((S1 - S0 + TILE - 1) / TILE - r0, PLACE_ROUNDS);
        if (r0) {  // (a lane of thousands of vehicles)
            __syncthreads();
            for (int r = 0; r < nh; ++r) {
                const int i = S0 + (r0 + r) * TILE + tid;
                const unsigned b = __ballot_sync(0xffffffffu, i < S1 && c.code[i] != C_STAY);
                if (ln == 0) s_ball[r * TW + w] = b;
            }
            __syncthreads();
            if (tid == 0) {
                int x = 0;
                for (int k = 0; k < nh * TW; ++k) {
                    s_lp[k] = x;
                    x += __popc(s_ball[k]);
                }
            }
            __syncthreads();
        }
#pragma unroll 2
        for (int r = 0; r < nh; ++r) {
            const int i = S0 + (r0 + r) * TILE + tid;
            const unsigned ball = s_ball[r * TW + w];
            if (i >= S1 || ((ball >> ln) & 1u)) continue;
            SV<Real> sv = st0;
            if (r0 + r > 0) {
                al = *reinterpret_cast<const int2*>(&c.cur.a[i].id);
                ab = *reinterpret_cast<const int4*>(&c.cur.b[i]);
                sv = c.stay[i];
            }
            const int lane = al.y, k = lane - L0;
            const int o = s_nx[k], end = s_nx[k + 1], h = s_hd[k];
            int pos = s_sh[k] + i - (lcarry + s_lp[r * TW + w] + __popc(ball & ((1u << ln) - 1u)));
            if (h > 0) {  // an entrant is ahead of the stayers behind it
                const int n = (h - 1) >> 9, f = (h - 1) & 511, behind = end - n - 1 - pos;
                for (int t = f; t < f + n; ++t) pos += s_bh[t] > behind;
            } else if (h < 0) {
                pos += entrants_ahead(c, ~h, sv.s, al.x);
            }
            if (pos < o || pos >= end || pos >= c.n_veh) {
                atomicOr(c.err, ERR_RANGE);
            } else {
                RecA<Real> O;
                O.s = sv.s; O.v = sv.v; O.id = al.x; O.lane = lane;
                c.nxt.a[pos] = O;
                *reinterpret_cast<int4*>(&c.nxt.b[pos]) = ab;
            }
        }
        lcarry += s_lp[nh * TW - 1] + __popc(s_ball[nh * TW - 1]);
    }
}

// Block vb of the first n_junc_chunks + 1 blocks of the kernel after k_decide:
// the signal states of the next step (JUNC_CHUNK junctions each; with Clocks
// the last of them to finish advances the clocks, which nothing else of the
// kernel reads), then the run-weight fit with the next step's counters.  Pdl:
// the kernel may have started before k_decide ended.
template <typename Real, bool Pdl, bool Clocks>
__device__ __forceinline__ void close_step(const Ctx<Real>& c, int vb) {
    const int nj = c.n_junc_chunks;
    if (Pdl) {
        grid_wait();
        grid_release();
    }
    if (__syncthreads_or(threadIdx.x == 0 ? *c.err & ERR_POISON : 0)) return;
    if (vb < nj) {
        __shared__ int s_clocks;
        const int j = vb * JUNC_CHUNK + threadIdx.x;
        if (j < c.n_junctions && !c.scen_ctl[c.junc[j].scen])
            c.junc_state[j] = c.junc_policy[j] == POL_MAXP ? mp_advance(c, j) : junction_state_at(c, j, 1);
        if (!Clocks) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            s_clocks = nj == 1 || atomicAdd(&c.cnt->junc_done, 1) == nj - 1;
            __threadfence();
        }
        __syncthreads();
        if (s_clocks) advance_clocks(c);
        return;
    }
    if (threadIdx.x == 0) {
        const int tag = c.cnt->tag;
        c.cnt_next->n_ent = 0;
        c.cnt_next->n_cand = 0;
        c.cnt_next->junc_done = 0;
        c.cnt_next->tag = tag >= 0x3fffffff ? 1 : tag + 1;
    }
    if (Clocks && nj == 0) advance_clocks(c);
    run_fit(c);
}

// Virtual block vb of the fused form: close_step's, then the tiles.
template <typename Real, bool Pdl>
__device__ __forceinline__ void place_block(const Ctx<Real>& c, int vb) {
    const int tile = vb - c.n_junc_chunks - 1;
    if (tile < 0) {
        close_step<Real, Pdl, true>(c, vb);
        return;
    }
    if (threadIdx.x == 0) c.delta_nxt[tile] = 0;  // (last read by the step before)
    if (tile > tile_key(c, __ldcg(&c.cnt->n_cur), c.n_lanes)) return;
    place_tile<Real, Pdl>(c, tile);
}

#ifndef MOSS_PLACE_MIN_BLOCKS
#define MOSS_PLACE_MIN_BLOCKS 6
#endif
template <typename Real>
__global__ void __launch_bounds__(TILE, MOSS_PLACE_MIN_BLOCKS) k_place(Ctx<Real> c) {
    place_block<Real, true>(c, blockIdx.x);
}

// ---------------------------------------------------------------------------
// The form for large networks, where the work of a tile no longer hides behind
// its latencies: the offsets in a kernel of their own (k_lanescan), then one
// thread per slot and one warp per entrant, whatever their lanes
// (k_place_slots).  Here a tile is 1 << tile_shift consecutive lanes (slot_w
// is 0): one round of 8 or 16 lanes per thread, more rounds where the handle has so
// many lanes that there would be more than SCAN_MAX_TILES tiles, each of
// which adds up the growth of those before it.
constexpr int SCAN_Q = 4;  // a thread takes 4 consecutive lanes Q times per round: SCAN_Q, or 2 by schedule
constexpr int SCAN_MAX_TILES = 1024;
// log2 of the lanes of a round
__host__ __device__ constexpr int scan_round_log2(int q) { return q == 4 ? 12 : 11; }
static_assert((1 << scan_round_log2(4)) == 16 * TILE && (1 << scan_round_log2(2)) == 8 * TILE,
              "the threads cover a round");

// One lane tile: newsize(l) = size(l) - leave(l) + enter(l), its prefix sum
// within the tile, and the growth of the tiles before it (tile_delta).  A warp
// takes 128 Q consecutive lanes of a round, 4 per thread and Q times, so that
// its 16-byte accesses cover 512 contiguous bytes and all loads of a round are
// in flight together.
//
// Bound by one memory round trip behind k_decide, by HBM (24 B a lane) for the
// millions of lanes of a pool of slots.  The growth words are loaded before
// the counts are cleared: loads issued behind the clearing stores wait for
// them.  A pool of 1,673,184 lanes, 627,900 of them in use by 32 scenarios:
// 12 us (40 MB), where tiles of 4 lanes per thread that cleared first took 37
// and the scan with look-back 20; the same order with 4 / 8 lanes per thread:
// 14 / 12, 16 lanes that clear first: 17.  The city's step 139.3 -> 136.2 us.
template <typename Real, int Q, bool Pdl>
__device__ __forceinline__ void scan_tile(const Ctx<Real>& c, int tile) {
    constexpr int ROUND = 1 << scan_round_log2(Q);
    __shared__ int s_w[2][TW], s_g[TW];
    const int ln = threadIdx.x & 31, w = threadIdx.x >> 5, nl = c.n_lanes;
    const int t0 = tile << c.tile_shift;
    const int rounds = ((min(nl - t0, 1 << c.tile_shift)) + ROUND - 1) / ROUND;
    if (threadIdx.x == 0) c.delta_nxt[tile] = 0;  // (last read by the step before)
    // offsets (written by the step before): o[q][4] is the end of the fourth lane
    int o[Q][5];
    const auto load_offsets = [&](int r0) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int l0 = r0 + 128 * q;
            if (l0 + 4 <= nl) {
                const int4 x = __ldcg(reinterpret_cast<const int4*>(c.cur.off + l0));
                o[q][0] = x.x; o[q][1] = x.y; o[q][2] = x.z; o[q][3] = x.w;
                o[q][4] = __ldcg(c.cur.off + l0 + 4);
            } else {
#pragma unroll
                for (int j = 0; j < 5; ++j) o[q][j] = l0 + j <= nl ? __ldcg(c.cur.off + l0 + j) : 0;
            }
        }
    };
    int r0 = t0 + w * (128 * Q) + 4 * ln;  // the thread's first lane of the round
    load_offsets(r0);
    int at = __ldcg(c.cur.off + t0);  // next offset of the round's first lane
    if (Pdl) {
        grid_wait();
        grid_release();
        if (*c.err & ERR_POISON) return;  // (set by a kernel that has ended)
    }
    int grown = 0;
    for (int r = 0; r < rounds; ++r, r0 += ROUND) {
        if (r) load_offsets(r0);
        int lv[Q][4], en[Q][4];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int l0 = r0 + 128 * q;
            if (l0 + 4 <= nl) {
                const int4 x = *reinterpret_cast<const int4*>(c.leave + l0), y = *reinterpret_cast<const int4*>(c.enter + l0);
                lv[q][0] = x.x; lv[q][1] = x.y; lv[q][2] = x.z; lv[q][3] = x.w;
                en[q][0] = y.x; en[q][1] = y.y; en[q][2] = y.z; en[q][3] = y.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    lv[q][j] = l0 + j < nl ? c.leave[l0 + j] : 0;
                    en[q][j] = l0 + j < nl ? c.enter[l0 + j] : 0;
                }
            }
        }
        if (r == 0)
            for (int p = threadIdx.x; p < tile; p += TILE) grown += c.tile_delta[p];
        int pre[Q], run = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int l0 = r0 + 128 * q;
            int sum = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int ns = l0 + j < nl ? o[q][j + 1] - o[q][j] - lv[q][j] + en[q][j] : 0;
                o[q][j] = ns;
                sum += ns;
            }
            if (l0 + 4 <= nl) {
                *reinterpret_cast<int4*>(c.leave + l0) = make_int4(0, 0, 0, 0);
                *reinterpret_cast<int4*>(c.enter + l0) = make_int4(0, 0, 0, 0);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (l0 + j < nl) { c.leave[l0 + j] = 0; c.enter[l0 + j] = 0; }
            }
            int incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (ln >= d) incl += y;
            }
            pre[q] = run + incl - sum;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (r == 0) {
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) grown += __shfl_xor_sync(0xffffffffu, grown, d);
            if (ln == 0) s_g[w] = grown;
        }
        if (ln == 0) s_w[r & 1][w] = run;
        __syncthreads();
        int wb = 0, total = 0;
#pragma unroll
        for (int k = 0; k < TW; ++k) {
            const int x = s_w[r & 1][k];
            if (k < w) wb += x;
            total += x;
            if (r == 0) at += s_g[k];
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int l0 = r0 + 128 * q;
            int on[5];
            on[0] = at + wb + pre[q];
#pragma unroll
            for (int j = 0; j < 4; ++j) on[j + 1] = on[j] + o[q][j];
            if (l0 + 4 <= nl) {
                *reinterpret_cast<int4*>(c.nxt.off + l0) = make_int4(on[0], on[1], on[2], on[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (l0 + j < nl) c.nxt.off[l0 + j] = on[j];
            }
            if (l0 < nl && nl <= l0 + 4) {  // this thread holds the last lane (on[] stays at the end past it)
                c.nxt.off[nl] = on[4];
                c.cnt_next->n_cur = on[4];
            }
        }
        at += total;
    }
}

// Virtual block vb of the scan: close_step's, then the lane tiles.
template <typename Real, int Q, bool Pdl>
__device__ __forceinline__ void scan_block(const Ctx<Real>& c, int vb) {
    const int tile = vb - c.n_junc_chunks - 1;
    if (tile < 0) close_step<Real, Pdl, false>(c, vb);
    else scan_tile<Real, Q, Pdl>(c, tile);
}

template <typename Real, int Q>
__global__ void __launch_bounds__(TILE) k_lanescan(Ctx<Real> c, int n_scan) {
    for (int vb = blockIdx.x; vb < n_scan; vb += gridDim.x) {
        scan_block<Real, Q, true>(c, vb);
        __syncthreads();  // shared memory serves the next one
    }
}

// The next snapshot.  Stayer tiles (one per block iteration): a vehicle that
// kept its lane goes to off'[lane] + (stayers ahead of it in the lane) +
// (entrants ahead of it), its stayers ahead counted in its tile (below).
// Then the entrants: rank = stayers ahead + entrants ahead.  Block 0 advances
// the clocks, which k_lanescan reads and this does not.
template <typename Real>
__device__ __forceinline__ void place_slots(const Ctx<Real>& c, int vb, int nvb) {
    if (vb == 0) advance_clocks(c);
    __shared__ int s_warp[TILE / 32];
    const int n = c.cnt->n_cur;
    const int n_ent = c.cnt->n_ent;
    const int tag = c.cnt->tag;
    const int n_tiles = (n + TILE - 1) / TILE;
    const int lane_id = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int s_lpre[TILE + 1];  // leavers among the tile's slots before each slot (and in all)
    __shared__ int s_first[2];        // start and end of the lane that holds the tile's first slot
    for (int tile = vb; tile < n_tiles; tile += nvb) {
        const int t0 = tile * TILE;
        const int i = t0 + threadIdx.x;
        const bool valid = i < n;
        const int8_t code = valid ? c.code[i] : C_STAY;
        RecA<Real> A;
        RecB B;
        SV<Real> w;
        if (valid) {  // issued before the tile's leaver scan
            A = c.cur.a[i];
            B = c.cur.b[i];
            w = c.stay[i];
        }
        const int leaver = (valid && code != C_STAY) ? 1 : 0;
        const unsigned ball = __ballot_sync(0xffffffffu, leaver);
        const int wpre = __popc(ball & ((1u << lane_id) - 1));
        if (lane_id == 0) s_warp[warp] = __popc(ball);
        if (threadIdx.x == 0) {
            s_first[0] = c.cur.off[A.lane];
            s_first[1] = c.cur.off[A.lane + 1];
        }
        __syncthreads();
        int wbase = 0;
        for (int w = 0; w < warp; ++w) wbase += s_warp[w];
        s_lpre[threadIdx.x] = wbase + wpre;
        if (threadIdx.x == TILE - 1) s_lpre[TILE] = wbase + wpre + leaver;
        // a lane that covers the whole tile: its leavers before the tile
        const int f0 = s_first[0], f1 = s_first[1];
        int pre0 = 0;
        if (f0 < t0 && f1 > t0 + TILE)
            for (int k0 = t0; k0 > f0; k0 -= TILE) {
                const int k = k0 - 1 - (int)threadIdx.x;
                pre0 += __syncthreads_count(k >= f0 && c.code[k] != C_STAY);
            }
        __syncthreads();
        if (valid && code == C_STAY) {
            // its rank among the lane's stayers: from the lane's start (slots
            // ahead of it minus the leavers among them) when the lane starts
            // in the tile; from the lane's end (the lane's stayers minus
            // those behind it) when the lane started before the tile and
            // ends in it; else with the leavers before the tile counted above
            const int lane = A.lane;
            const int ob = c.cur.off[lane], oe = c.cur.off[lane + 1];
            const int o0 = c.nxt.off[lane], o1 = c.nxt.off[lane + 1];
            int n_in = 0;
            const int ent = entrants_ahead(c, list_head(c.head, lane, tag), w.s, A.id, &n_in);
            const int x = threadIdx.x;
            int stay_rank;
            if (ob >= t0) {
                stay_rank = (i - ob) - (s_lpre[x] - s_lpre[ob - t0]);
            } else if (oe <= t0 + TILE) {
                const int behind = (oe - 1 - i) - (s_lpre[oe - t0] - s_lpre[x + 1]);
                stay_rank = (o1 - o0 - n_in) - 1 - behind;
            } else {
                stay_rank = (i - ob) - (pre0 + s_lpre[x]);
            }
            const int pos = o0 + stay_rank + ent;
            if (pos < o0 || pos >= o1) {
                atomicOr(c.err, ERR_RANGE);
            } else {
                RecA<Real> O;
                O.s = w.s; O.v = w.v; O.id = A.id; O.lane = lane;
                c.nxt.a[pos] = O;
                c.nxt.b[pos] = B;
            }
        }
        __syncthreads();  // s_warp, s_lpre and s_first serve the next tile
    }
    // entrants: one warp per entrant.  The stayers of a lane keep their
    // order (nobody overtakes within a lane, R13), so the stayers behind an
    // entrant form the rear of the lane's old segment: the warp counts them
    // from the segment's end, 32 slots per round, and stops at the first
    // round that holds a stayer ahead of the entrant (entrants join mostly
    // at the rear of a lane: one round).  Stayers ahead = the lane's stayers
    // (its next size minus its entrants) minus those behind.
    const int gwarp = vb * (TILE / 32) + warp, nwarps = nvb * (TILE / 32);
    for (int q = gwarp; q < n_ent; q += nwarps) {
        const RecA<Real> Q = c.ea[q];
        const int lane = Q.lane;
        const int b = c.cur.off[lane], e = c.cur.off[lane + 1];
        int behind = 0;
        for (int k0 = e - 1; k0 >= b; k0 -= 32) {
            const int k = k0 - lane_id;
            bool st = false, ah = false;
            if (k >= b && c.code[k] == C_STAY) {
                st = true;
                ah = ahead(c.stay[k].s, c.cur.a[k].id, Q.s, Q.id);
            }
            behind += __popc(__ballot_sync(0xffffffffu, st && !ah));
            if (__any_sync(0xffffffffu, ah)) break;
        }
        if (lane_id == 0) {
            int n_in = 0;
            const int ent_ahead = entrants_ahead(c, list_head(c.head, lane, tag), Q.s, Q.id, &n_in);
            const int o0 = c.nxt.off[lane], o1 = c.nxt.off[lane + 1];
            const int pos = o0 + (o1 - o0 - n_in - behind) + ent_ahead;
            if (pos < o0 || pos >= o1) {
                atomicOr(c.err, ERR_RANGE);
            } else {
                c.nxt.a[pos] = Q;
                c.nxt.b[pos] = c.eb[q];
            }
        }
    }
}

template <typename Real>
__global__ void __launch_bounds__(TILE) k_place_slots(Ctx<Real> c) {
    grid_wait();
    grid_release();
    if (__syncthreads_or(threadIdx.x == 0 ? *c.err & ERR_POISON : 0)) return;
    place_slots(c, blockIdx.x, gridDim.x);
}

// tile cuts of the current snapshot's offsets (after creation, a state reset
// or a change of the tile size; one thread per lane)
template <typename Real>
__global__ void k_tile_cuts(Ctx<Real> c) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l == 0) c.tile_cur[0] = c.tile_nxt[0] = 0;
    if (l >= c.n_lanes) return;
    const int q0 = tile_key(c, c.cur.off[l], l), q1 = tile_key(c, c.cur.off[l + 1], l + 1);
    for (int q = q0 + 1; q <= q1; ++q) c.tile_cur[q] = l + 1;
    if (l + 1 == c.n_lanes) c.tile_cur[q1 + 1] = l + 1;
}

// ---------------------------------------------------------------------------
// The whole step as one cooperative launch (every block resident at once):
// the work of the kernels of the handle's form as phases separated by
// grid-wide barriers (n_scan > 0: k_decide, k_lanescan and k_place_slots; else
// k_decide and k_place).  A barrier is a count of arrived blocks and a
// generation word; a wait that exceeds SPIN_LIMIT sets ERR_TIMEOUT and every
// block leaves the step.  The city as one launch takes 192 us a step with the
// placement by tiles, 162 in its own form.
__device__ __forceinline__ bool grid_sync(unsigned* bar, int* err) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        cuda::atomic_ref<unsigned, cuda::thread_scope_device> gen(bar[1]);
        const unsigned g = gen.load(cuda::memory_order_relaxed);
        __threadfence();
        if (atomicAdd(&bar[0], 1u) == gridDim.x - 1) {
            bar[0] = 0u;
            gen.store(g + 1u, cuda::memory_order_release);
        } else {
            long long spins = 0;
            while (gen.load(cuda::memory_order_acquire) == g) {
                if (++spins > SPIN_LIMIT) { atomicOr(err, ERR_TIMEOUT); break; }
                if (spins > 16) __nanosleep(32);
            }
        }
        __threadfence();
        s_ok = !(*((volatile int*)err) & ERR_POISON);
    }
    __syncthreads();
    return s_ok != 0;
}

#ifndef MOSS_COOP_MIN_BLOCKS
#define MOSS_COOP_MIN_BLOCKS 4
#endif
template <typename Real, bool Groups>
__global__ void __launch_bounds__(TILE, MOSS_COOP_MIN_BLOCKS) k_step_coop(Ctx<Real> c, int n_work, int n_ins,
                                                                          int n_scan, int n_place, unsigned* bar) {
    if (*c.err & ERR_POISON) return;
    // decide: n_work tile runs, then n_ins insertion blocks, as virtual blocks
    for (int vb = blockIdx.x; vb < n_work + n_ins; vb += gridDim.x)
        decide_block<Real, Groups>(c, n_work, vb, n_work + n_ins);
    if (!grid_sync(bar, c.err)) return;
    if (n_scan) {
        for (int vb = blockIdx.x; vb < n_scan; vb += gridDim.x) {
            scan_block<Real, SCAN_Q, false>(c, vb);
            __syncthreads();  // shared memory serves the next one
        }
        if (grid_sync(bar, c.err)) place_slots(c, blockIdx.x, gridDim.x);
        return;
    }
    for (int vb = blockIdx.x; vb < n_place; vb += gridDim.x) {
        place_block<Real, false>(c, vb);
        __syncthreads();  // shared memory serves the next one
    }
}

// signal states for the current step of every junction (after creation or
// a state reset)
template <typename Real>
__global__ void k_junction_init(Ctx<Real> c, int j0, int j1) {
    for (int j = j0 + blockIdx.x * blockDim.x + threadIdx.x; j < j1; j += gridDim.x * blockDim.x)
        c.junc_state[j] = junction_state_at(c, j, 0);
}

// setter: policy (and manual phase) of n junctions, effective from the
// current step (the state of the step is recomputed)
template <typename Real>
__global__ void k_set_signal(Ctx<Real> c, int n, const int32_t* ids, const int32_t* phases, int policy) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int j = ids[k];
    if (policy == POL_MAXP) {
        // starts, green, the phase the junction shows at this step (R23)
        const int st = c.junc_state[j];
        c.mp[j] = make_int4((st & 512) ? 0 : (st & 15), 1, -1, 0);
    }
    const int was = c.junc_policy[j] == POL_MAXP, now = policy == POL_MAXP;
    if (was != now) atomicAdd(c.n_mp, now - was);
    c.junc_policy[j] = policy;
    if (policy == POL_MANUAL) c.junc_manual[j] = phases[k];
    c.junc_state[j] = junction_state_at(c, j, 0);
}

// lane setters (R25): speed limit (mode 0, value as float bits) or
// restriction flag (mode 1) of n lanes, effective from the next step
template <typename Real>
__global__ void k_set_lane(Ctx<Real> c, int n, const int32_t* ids, const int32_t* vals, int mode) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    LaneInfo* li = const_cast<LaneInfo*>(c.lane) + ids[k];
    if (mode == 0) li->vmax = __int_as_float(vals[k]);
    else li->flags = vals[k] ? (li->flags | LF_RESTRICTED) : (li->flags & ~LF_RESTRICTED);
}

// The end of a getter whose outputs lie in pinned host memory: the last block
// to have stored its own stores the ticket that the host waits for.
struct Ticket {
    int* done;
    long long* word;  // null: no ticket
    long long value;
};
__device__ __forceinline__ void give_ticket(const Ticket& tk) {
    if (!tk.word) return;
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(tk.done, 1) == (int)gridDim.x - 1) {
        *tk.done = 0;
        __threadfence_system();
        cuda::atomic_ref<long long, cuda::thread_scope_system> word(*tk.word);
        word.store(tk.value, cuda::memory_order_release);
    }
}

// metrics of the current snapshot (R24): queue length of lanes [l0, l1) —
// vehicles with v < 0.1 m/s within the last 50 m (the lane's segment is
// ordered from its end, so the scan stops at the first vehicle farther away).
// err_out (pinned host memory): the device error word, so that the getter
// needs no copy of its own for it.
template <typename Real>
__global__ void k_lane_queue(Ctx<Real> c, int l0, int l1, int32_t* out, long long* err_out, Ticket tk) {
    const int l = l0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (l == l0) *(int*)err_out = *c.err;
    if (l < l1) {
        const double L = (double)c.lane[l].L;
        int q = 0;
        for (int k = c.cur.off[l]; k < c.cur.off[l + 1]; ++k) {
            const RecA<Real> a = c.cur.a[k];
            if (L - (double)a.s > 50.0) break;
            if ((double)a.v < 0.1) ++q;
        }
        out[l - l0] = q;
    }
    give_ticket(tk);
}

// average vehicle speed of roads [r0, r1) (R24): mean speed of the vehicles
// on the road's lanes, the mean speed limit of its lanes when it is empty.
// The lanes of a road are neighbours, so its vehicles are one run of slots:
// ROAD_SPEED_THREADS threads take it together (one thread per road waited
// for one load after the other: the call on the 39,600 roads of the city
// 105 -> 69 us, on the grid's 3,480 62 -> 26 us, with its waits).
constexpr int ROAD_SPEED_THREADS = 8;
template <typename Real>
__global__ void k_road_speed(Ctx<Real> c, int r0, int r1, double* out, long long* err_out, Ticket tk) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) *(int*)err_out = *c.err;
    const int r = r0 + t / ROAD_SPEED_THREADS, p = t % ROAD_SPEED_THREADS;
    double sum = 0.0;
    int cnt = 0;
    int2 sp = make_int2(0, 0);
    if (r < r1) {
        sp = c.road_span[r];
        const int b = c.cur.off[sp.x], e = c.cur.off[sp.y];
        cnt = e - b;
        for (int k = b + p; k < e; k += ROAD_SPEED_THREADS) sum += (double)c.cur.a[k].v;
    }
#pragma unroll
    for (int o = ROAD_SPEED_THREADS / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (r < r1 && p == 0) {
        if (cnt > 0) {
            out[r - r0] = sum / (double)cnt;
        } else {
            double lim = 0.0;
            for (int l = sp.x; l < sp.y; ++l) lim += (double)c.lane[l].vmax;
            out[r - r0] = lim / (double)(sp.y - sp.x);
        }
    }
    give_ticket(tk);
}

// metric record, step and error word of a scenario into pinned host memory,
// then the ticket that the host waits for
__global__ void k_readback(const long long* metrics, const long long* step, const int* err, long long* out,
                           long long ticket) {
    grid_wait();
    grid_release();
    const int k = threadIdx.x;
    if (k < M_NFIELDS) out[k] = metrics[k];
    else if (k == M_NFIELDS) out[k] = *step;
    else if (k == M_NFIELDS + 1) *(int*)(out + k) = *err;
    __threadfence_system();
    __syncwarp();
    if (k == 0) {
        cuda::atomic_ref<long long, cuda::thread_scope_system> word(out[M_NFIELDS + 2]);
        word.store(ticket, cuda::memory_order_release);
    }
}

// The per-vehicle state of a scenario (vehicles [v0, v0 + nv)) by id, for the
// state getter: k_state_fill writes what the vehicle tables hold and the
// values of vehicles that are not on a lane, k_state_gather the values of
// those in the snapshot (the slots of the scenario's lanes [lo, lo + nl)).
// Bound by the transfer to the host and the pages it touches there: the call
// takes 0.45 ms for 500,009 vehicles and 1.9 ms for 2,464,950 (both
// snapshot records copied and scattered on the host: 6.2 and 40.7 ms).
struct StateOut {
    double *s, *v;
    int32_t *status, *lane, *rc, *flags;
};

template <typename Real>
__global__ void k_state_fill(Ctx<Real> c, int sc, int v0, int nv, StateOut o, long long* err_out) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *(int*)err_out = *c.err;
    const long long step = c.scen_step[sc];
    const int tag = (int)((step - 1) & 0xFFFFFF);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += gridDim.x * blockDim.x) {
        const int f = c.vflags[v0 + i];
        o.status[i] = c.vstatus[v0 + i];
        o.flags[i] = step > 0 && (int)((unsigned)f >> 8) == tag ? (f & 255) : 0;
        o.lane[i] = -1; o.rc[i] = 0;
        o.s[i] = 0.0; o.v[i] = 0.0;
    }
}

template <typename Real>
__global__ void k_state_gather(Ctx<Real> c, int v0, int nv, int lo, int nl, StateOut o) {
    const int b = c.cur.off[lo], e = c.cur.off[lo + nl];
    for (int k = b + blockIdx.x * blockDim.x + threadIdx.x; k < e; k += gridDim.x * blockDim.x) {
        const RecA<Real> a = c.cur.a[k];
        const int i = a.id - v0;
        if (i < 0 || i >= nv) continue;
        o.lane[i] = a.lane - lo;
        o.s[i] = (double)a.s;
        o.v[i] = (double)a.v;
        o.rc[i] = c.cur.b[k].rptr - c.route_span[a.id].x;
    }
}

// Re-routing (R26): mark the requested vehicles (req[vid] = their index in
// the request, -1 otherwise), find the lanes of the active ones, and give
// them their new routes (route spans; for the active ones the snapshot
// record's route cursor, last road and next lane).
__global__ void k_mark_vehicles(int32_t* req, int n, const int32_t* vids, int on) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) req[vids[k]] = on ? k : -1;
}

template <typename Real>
__global__ void k_find_lanes(Ctx<Real> c, const int32_t* req, int32_t* lane_out) {
    const int n = c.cnt->n_cur;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const RecA<Real> a = c.cur.a[i];
        const int k = req[a.id];
        if (k >= 0) lane_out[k] = a.lane;
    }
}

template <typename Real>
__global__ void k_apply_routes(Ctx<Real> c, const int32_t* req, int nv, const int32_t* vids, const int2* spans) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nv; k += gridDim.x * blockDim.x)
        const_cast<int2*>(c.route_span)[vids[k]] = spans[k];
    const int n = c.cnt->n_cur;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const RecA<Real> a = c.cur.a[i];
        const int k = req[a.id];
        if (k < 0) continue;
        RecB b = c.cur.b[i];
        b.rptr = spans[k].x;
        b.rlast = spans[k].y - 1;
        const LaneInfo li = c.lane[a.lane];
        if (li.lo >= 0) b.nl = b.rptr < b.rlast ? jl_toward(c, li, c.routes[b.rptr + 1]) : -1;
        c.cur.b[i] = b;
    }
}

// Lane plans (R28): road roads[k] switches to plan plans[k] (junction lanes
// outside it get LF_OFF) and is marked; then the vehicles on the marked
// roads' lanes get their next lane again; then the marks are cleared.
template <typename Real>
__global__ void k_set_plan(Ctx<Real> c, int n, const int32_t* roads, const int32_t* plans, const int32_t* jl_plans,
                           int8_t* road_mark) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int r = roads[k], p = plans[k];
    const int2 sp = c.road_span[r];
    LaneInfo* lanes = const_cast<LaneInfo*>(c.lane);
    for (int l = sp.x; l < sp.y; ++l)
        for (int j = lanes[l].jb; j < lanes[l].je; ++j) {
            const bool on = (jl_plans[j] >> p) & 1;
            lanes[j].flags = on ? (lanes[j].flags & ~LF_OFF) : (lanes[j].flags | LF_OFF);
        }
    road_mark[r] = 1;
}

template <typename Real>
__global__ void k_plan_next_lanes(Ctx<Real> c, const int8_t* road_mark) {
    const int n = c.cnt->n_cur;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const RecA<Real> a = c.cur.a[i];
        const LaneInfo li = c.lane[a.lane];
        if (li.lo < 0 || !road_mark[li.road]) continue;
        RecB b = c.cur.b[i];
        b.nl = b.rptr < b.rlast ? jl_toward(c, li, c.routes[b.rptr + 1]) : -1;
        c.cur.b[i] = b;
    }
}

__global__ void k_unmark_roads(int n, const int32_t* roads, int8_t* road_mark) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) road_mark[roads[k]] = 0;
}

// single values written in stream order (slot control, horizons)
__global__ void k_put_i32(int32_t* p, int32_t v) { *p = v; }
__global__ void k_put_i64(long long* p, long long v) { *p = v; }

// Failure-detection self-test: the look-back of tile 1 waits on tile word 0,
// which nothing publishes, so the bounded wait must give up and report.
__global__ void k_selftest_wait(unsigned long long* words, int* err) {
    bool timeout = false;
    warp_lookback(words, 1, &timeout);
    if (threadIdx.x == 0 && timeout) atomicOr(err, ERR_TIMEOUT);
}

}  // namespace moss
