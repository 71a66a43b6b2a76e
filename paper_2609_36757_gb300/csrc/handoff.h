// The hand-offs of the attention kernels through named (hardware) barriers:
// which barrier, in which order, and what a role owes after a failed wait.
//
// The MMA warp of each kernel syncs on named barriers at which the other roles
// arrive.  A named barrier has no time limit, and it counts arrivals without
// looking at who made them: a warp that arrives twice before the MMA warp has
// synced stands in for a warp that has not arrived, a generation completes
// without the MMA warp, and its next sync waits for ever.  So on every barrier
//   1. each warp of the arriving role arrives once per generation, and
//   2. it arrives for the next one only after the MMA warp has synced on this.
// In normal operation the data see to 2: what a warp waits for before its next
// arrival is committed by MMAs that were issued after the sync.  After a failed
// (timed-out or aborted) wait a role does no more work, but it still makes
// every arrival that it owes, each behind that same proof: a wait for the
// commit, deaf to the abort flag.  An MMA warp that gave up before its first
// MMA goes through its hand-offs and commits with nothing issued between them.
// Everyone then leaves in step, with undefined data and the failure recorded.
// (A blocking sync for each owed arrival is not enough: a warp may have arrived
// once ahead of the MMA warp, and its sync would pair with that arrival.)  The
// proofs are commits of the tensor pipe alone, so they come also where a copy
// never lands; should the pipe itself stop, the waits end at their time limit.
//
// Plain C++ (no CUDA types): tests/handoff_model.cpp runs these same functions
// on the host, under random schedules with waits that fail anywhere.
#pragma once

#ifdef __CUDACC__
#define FASTVR_HANDOFF __device__ __forceinline__
#else
#define FASTVR_HANDOFF inline
#endif

namespace fastvr {
namespace handoff {

// ------------------------------------------------------------------ forward
constexpr int kFwdKStages = 3;  // depth of the K ring
constexpr int kFwdVStages = 2;  // depth of the V ring
// S_t read (free for the next QK^T) and P_t stored: the four softmax warps of
// query tile t arrive.  Where the two tiles share S (own_s false) they share
// its barrier, in turn.
FASTVR_HANDOFF constexpr int fwd_s_free(int t, bool own_s) {
  return own_s && t ? 11 : 1;
}
FASTVR_HANDOFF constexpr int fwd_p_full(int t) { return 2 + t; }
constexpr int kFwdSoftmaxWarps = 5;  // of a generation: four, and the MMA warp
// K (V) of a ring stage has landed: the relay warp arrives.
constexpr int kFwdKFull0 = 4;  // + stage
constexpr int kFwdVFull0 = 7;  // + stage
constexpr int kRelayWarps = 2;  // of a generation: the relay and the MMA warp
FASTVR_HANDOFF int fwd_k(int j) { return kFwdKFull0 + j % kFwdKStages; }
FASTVR_HANDOFF int fwd_v(int j) { return kFwdVFull0 + j % kFwdVStages; }

// The MMA warp over n key tiles: QK_0(j), PV_0(j-1), QK_1(j), PV_1(j-1).  S is
// one buffer for both query tiles, or one each (own_s); a QK^T follows the read
// of what its buffer held.  qk and pv get the tile, the ring stage (worked out
// ahead of the syncs: the MMA warp sets the pace), for pv whether O holds
// something, and whether the stage is read for the last time.  (The loop is
// written as the compiler lays it out best: an S buffer's uses counted, with
// tests of j in their place the training clip's forward took 520 us in place of
// 501; the PV's tile as jp, without it 110 CTAs of 63 tiles took 77.3 us in place
// of 77.0.)
template <class Ops>
FASTVR_HANDOFF void fwd_mma_steps(int n, bool two, bool own_s, Ops& ops) {
  int s_uses[2] = {0, 0};
  for (int j = 0; j <= n; ++j) {
    const bool has_qk = j < n;
    const int jp = j - 1;  // the key tile whose PV runs now
    const int ks = j % kFwdKStages, vs = jp % kFwdVStages;
    if (has_qk) {
      ops.relay_sync(kFwdKFull0 + ks);
      if (s_uses[0]++ > 0) ops.softmax_sync(fwd_s_free(0, own_s));
      ops.qk(0, ks, !two);
    }
    if (jp >= 0) {
      ops.relay_sync(kFwdVFull0 + vs);
      ops.softmax_sync(fwd_p_full(0));
      ops.pv(0, vs, jp > 0, !two);
    }
    if (two) {
      if (has_qk) {
        if (s_uses[own_s]++ > 0) ops.softmax_sync(fwd_s_free(1, own_s));
        ops.qk(1, ks, true);
      }
      if (jp >= 0) {
        ops.softmax_sync(fwd_p_full(1));
        ops.pv(1, vs, jp > 0, true);
      }
    }
  }
}

// "S read" arrivals of query tile t: one per S except the last that the MMA
// warp has no QK^T to write behind (with one S for both tiles, the second's).
FASTVR_HANDOFF int fwd_s_arrivals(int n, int t, int tiles, bool own_s) {
  return own_s || t == tiles - 1 ? n - 1 : n;
}

// A softmax warp of tile t whose wait failed, s_done and p_done arrivals made.
// wait_s(j): QK_t(j) was committed, so the S before it has been synced on;
// wait_p(j): PV_t(j) was, and with it P_t(j).
template <class Ops>
FASTVR_HANDOFF void fwd_softmax_rest(int n, int t, bool own_s, int s_total,
                                     int s_done, int p_done, Ops ops) {
  for (int j = p_done; j < n; ++j) {
    if (j >= s_done) {
      ops.wait_s(j);
      if (j < s_total) ops.arrive(fwd_s_free(t, own_s));
    }
    if (j > 0) ops.wait_p(j - 1);
    ops.arrive(fwd_p_full(t));
  }
}

// The relay warp: K(j), then V(j-1).  A failed wait for the tile leaves the
// one for its slot, free once the MMAs of the tile before it have run.
template <class Ops>
FASTVR_HANDOFF void fwd_relay_steps(int n, Ops& ops) {
  bool ok = true;
  for (int j = 0; j <= n; ++j) {
    if (j < n) {
      ok = ok && ops.wait_k(j);
      if (!ok) ops.wait_k_slot(j);
      ops.arrive(fwd_k(j));
    }
    if (j > 0) {
      ok = ok && ops.wait_v(j - 1);
      if (!ok) ops.wait_v_slot(j - 1);
      ops.arrive(fwd_v(j - 1));
    }
  }
}

// ----------------------------------------------------------------- backward
constexpr int kBwdStages0 = 3;  // depth of ring 0 (dK/dV: Q; dQ: K)
constexpr int kBwdStages1 = 2;  // depth of ring 1 (dK/dV: dO; dQ: V)
// P stored (or, dQ, read into registers) and dS stored: the eight compute
// warps arrive.  The dQ kernel hands dS over through two barriers in turn: its
// next S and dP do not wait for dS, so a warp can be done with the next dS
// while another has yet to arrive for this one.  It cannot be two ahead: the S
// after that follows the MMA warp's wait for this dS.
constexpr int kBwdP = 1;
constexpr int kBwdComputeWarps = 9;  // of a generation: eight, and the MMA warp
// A ring's stage has landed: the relay warp arrives.
FASTVR_HANDOFF int bwd_ring0(int j) { return 3 + j % kBwdStages0; }
FASTVR_HANDOFF int bwd_ring1(int j) { return 6 + j % kBwdStages1; }
// two_ds: the dQ kernel's two barriers.
FASTVR_HANDOFF int bwd_ds(int j, bool two_ds) {
  return two_ds && (j & 1) ? 9 : 2;
}

// The MMA warps over n tiles: s and dp issue S(j) and dP(j) (transposed in
// dK/dV), dv dV, out dK or dQ.
template <class Ops>
FASTVR_HANDOFF void dkdv_mma_steps(int n, Ops& ops) {
  ops.relay_sync(bwd_ring0(0));
  ops.s(0);
  ops.relay_sync(bwd_ring1(0));
  ops.dp(0);
  for (int j = 0; j < n; ++j) {
    ops.compute_sync(kBwdP);
    ops.dv(j);
    if (j + 1 < n) {
      ops.relay_sync(bwd_ring0(j + 1));
      ops.s(j + 1);
    }
    ops.compute_sync(bwd_ds(j, false));
    ops.out(j);
    if (j + 1 < n) {
      ops.relay_sync(bwd_ring1(j + 1));
      ops.dp(j + 1);
    }
  }
}

template <class Ops>
FASTVR_HANDOFF void dq_mma_steps(int n, Ops& ops) {
  ops.relay_sync(bwd_ring0(0));
  ops.s(0);
  ops.relay_sync(bwd_ring1(0));
  ops.dp(0);
  for (int j = 0; j < n; ++j) {
    ops.compute_sync(kBwdP);
    if (j + 1 < n) {
      ops.relay_sync(bwd_ring0(j + 1));
      ops.s(j + 1);
      ops.relay_sync(bwd_ring1(j + 1));
      ops.dp(j + 1);
    }
    ops.compute_sync(bwd_ds(j, true));
    ops.out(j);
  }
}

// A compute warp whose wait failed, p_done and ds_done arrivals made.
// wait_s(j), wait_dp(j): S(j) and dP(j) were committed; they were issued behind
// the sync on P(j-1), and, for dP, on the dS before on the same barrier.
template <class Ops>
FASTVR_HANDOFF void bwd_compute_rest(int n, bool two_ds, int p_done, int ds_done,
                                     Ops ops) {
  for (int j = ds_done; j < n; ++j) {
    if (j >= p_done) {
      ops.wait_s(j);
      ops.arrive(kBwdP);
    }
    ops.wait_dp(j);
    ops.arrive(bwd_ds(j, two_ds));
  }
}

// The relay warp: ring 0, then ring 1 of each step; a failed wait as above.
template <class Ops>
FASTVR_HANDOFF void bwd_relay_steps(int n, Ops& ops) {
  bool ok = true;
  for (int j = 0; j < n; ++j) {
    ok = ok && ops.wait(0, j);
    if (!ok) ops.wait_slot(0, j);
    ops.arrive(bwd_ring0(j));
    ok = ok && ops.wait(1, j);
    if (!ok) ops.wait_slot(1, j);
    ops.arrive(bwd_ring1(j));
  }
}

}  // namespace handoff
}  // namespace fastvr
