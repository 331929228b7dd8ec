// gv_state.cuh -- device-resident state of a transport call: the
// double-buffered per-type track queues (the StackBuffer / stage baskets of
// GeantV Sec. 2.1.2, as arrays of 16-byte parts), the generation control
// block and the tally pointers.
#pragma once
#include "gv_device.cuh"

namespace gv {

// Track records.  The queue of one particle type is an array of parts: part p
// holds 16 bytes of every track, so a warp's consecutive tracks are loaded
// and stored with one coalesced 16-byte access per part and lane.
//   FP32 (64 B): {x, y} {z, id} {u, v, w, E} {n_lambda, event, step, sf}
//   FP64 (84 B): {x, y} {z, id} {u, v} {w, E} {n_lambda, event, step} and sf
// (sf = sub-slab | flags << 16) in an array of its own.
// Twelve 4- and 8-byte arrays, as before, took three times the accesses and
// address computations (see load_track).
template <typename R> struct TrackLayout {
  static constexpr int parts = sizeof(R) == 4 ? 4 : 5;
  static constexpr size_t tail = sizeof(R) == 4 ? 0 : sizeof(int);  // bytes per track past the parts
  static size_t round256(size_t n) { return (n + 255) / 256 * 256; }
  static size_t part_bytes(long long cap) { return round256(static_cast<size_t>(cap) * 16); }
  static size_t queue_bytes(long long cap) { return parts * part_bytes(cap) + round256(static_cast<size_t>(cap) * tail); }
};

// reciprocal node energies staged in shared memory, padded to 16 bytes
constexpr unsigned kInvNodeBytes = (kGridN * sizeof(float) + 15) / 16 * 16;

constexpr int kFlagPrimary = 1;
constexpr int kFlagInteracted = 2;

template <typename R> constexpr size_t track_bytes() {
  return 3 * sizeof(double) + 5 * sizeof(R) + sizeof(unsigned long long) + 3 * sizeof(unsigned);
}

// Claim counters of the work slices, one per 128-byte line.
constexpr int kNClaim = 16;
struct alignas(128) ClaimSlot {
  unsigned n;
};
// Fill counter of one output queue, in a 128-byte line of its own: every
// warp's append and every block's claim is an atomic on one of these words.
struct alignas(128) FillSlot {
  unsigned n;
};

// An interaction request of the split pipeline: the along-step kernel hands
// a track that is due a discrete interaction to the interaction kernel
// (one 16-byte-aligned record per request).
template <typename R> struct alignas(16) GReq {
  double x, y, z;
  unsigned long long id;
  R E, d0, d1, d2;
  R u2, u3;      // the sampler's uniforms of the step's counter block 0
  unsigned ev, kk;
  int sf;        // sub-slab | flags << 16
  int key;       // request key
};
// Request keys: type * 3 + process.  Electrons have two processes, and their
// third key stands for positrons that stopped and annihilate at rest.
constexpr int kNReqKey = 9;
constexpr int kKeyRest = 1 * 3 + 2;

// The plan of a generation, one 64-byte record: a block reads all of it in
// one round trip to L2 when the generation before has completed.
struct alignas(64) Plan {
  int done;                  // the transport has ended: nothing is planned
  int K;                     // rounds per claimed track
  unsigned B;                // tracks per block claim
  int book;                  // events are counted live (primaries are still waiting on the in-flight cap)
  unsigned end[4];           // cumulative chunk counts in claim order: e+, e-, gamma, primaries
  unsigned n_in[3];          // tracks in the input queues (within the capacity)
  unsigned prim_begin, prim_count;
  unsigned pad[3];
};

// Generation control block.  The last block of every generation writes the
// plan of the next one; kernels only read it.
struct Ctl {
  ClaimSlot claims[kNClaim];
  FillSlot cnt[2][3];        // queue fill per buffer parity and type
  ClaimSlot claim;           // chunk claim counter of the block claims
  Plan plan;
  unsigned prim_next;        // primaries handed out so far
  unsigned blocks_done;
  int status;
  unsigned ev_started, ev_done;  // events whose live-track count left / returned to zero
  unsigned max_in_flight;        // refill cap of this call (0: none)
  unsigned emax_bits;            // largest primary energy (FP32 bits), for the automatic cap
  unsigned long long gen;
  unsigned long long loop_iter;  // bodies of the device-side generation loop run so far
  unsigned long long live_peak;
  unsigned long long cost_started, cost_done;  // automatic cap: track budget taken by / returned from events
  unsigned long long counters[16];
  // split pipeline: requests of this generation, per key, and the claim /
  // completion counters of the interaction kernel
  unsigned req_n;
  unsigned key_n[kNReqKey];
  unsigned claim_b, blocks_done_b;
};

template <typename R> struct DevState {
  View<R> view;              // global-memory table pointers and constants
  unsigned char *qmem;       // track queues [parity][type], see TrackLayout
  unsigned long long q_bytes, q_part;  // bytes of one queue and of one of its parts
  unsigned long long capacity;
  Ctl *ctl;
  const gv_primary *prim;
  const unsigned *order;     // primary visiting order (one-event mode) or null
  unsigned n_prim, n_events;
  unsigned ev_base;          // event index of tally row 0 (the random streams use ev_base + row)
  double *edep, *cell, *escape;
  unsigned long long *evcnt;
  unsigned *evlive;          // live tracks per event (events-in-flight accounting)
  int max_in_flight;         // 0: no cap, -1: automatic from the primaries' energies
  unsigned seed_lo, seed_hi;
  int block_size, mode, K_bulk, K_tail;
  int chunk;                 // tracks per work chunk: 32 (a warp) or block_size (basketizer)
  int claim_chunks;          // chunks a warp takes per atomic claim (no basketizer)
  int along_steps;           // basketizer: steps per lane before the block basket
  int scoring;               // 0 direct atomics, 1 warp-merged (selects the kernel)
  int pipeline;              // 0 fused step kernel, 1 along-step + interaction kernels
  GReq<R> *req;              // split pipeline: request records [req_cap]
  unsigned *keyidx;          // split pipeline: request indices per key [kNReqKey][req_cap]
  unsigned long long req_cap;
  unsigned long long tail_threshold, low_water, batch, max_gen;
  int n_mat;
  unsigned xs_bytes, zb_bytes;  // staged into shared memory
  unsigned smem_req_off;        // start of the basketizer's request records
  unsigned smax_off, smax_bytes; // the integral approach's bound, staged into shared memory
  unsigned rec_off;              // sub-slab records, made in shared memory
  unsigned smem_lk_off;          // the block's secondary stack (local_stack)
  int local_stack;
  int grid, adaptive_chunk;  // blocks of the step kernel; spread small populations over all of them
  const unsigned long long *pcost;  // automatic cap: prefix sums of the primaries' track budgets [n_prim + 1], or null
  unsigned long long *evcost;       // automatic cap: budget held by each event in flight [n_events]
  int along_steps_g;                // basketizer: along-step budget of photons
};

}  // namespace gv
