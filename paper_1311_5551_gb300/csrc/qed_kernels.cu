// qed_kernels.cu -- CUDA kernels of the QED Monte-Carlo step (Sec. 3) for sm_103a.
//
// One step = one launch of step_kernel over all three species (warp-uniform chunks of 32
// consecutive particles, grid-stride over chunks) followed by one finalisation kernel that merges
// the particles created during the step in (parent species, parent index) order:
//   step_kernel      push, eta/chi, rates, tau; events collected per warp and taken 32 at a time
//                    (ballot + one atomic per warp append), per-chunk event masks and their counts
//                    per group of chunks; per-block FP64 ledger partials where the step's ledger
//                    can be read
//   finalize_kernel  checks capacities, ranks every new particle by its parent's position (a
//                    counting sort on the dense parent index), moves it into place and assigns
//                    consecutive ids; the last block sets the counters
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

#include "qed_device.cuh"

// The file is compiled three times (QED_KERNELS_PART = 1, 2, 3), so that nvcc builds the
// single-scenario step, the batch step and everything else in parallel: each part defines the
// launchers of its share and so instantiates only their kernels.  Without the macro (0) one
// translation unit holds all of them.
#ifndef QED_KERNELS_PART
#define QED_KERNELS_PART 0
#endif
#define QED_PART(p) (QED_KERNELS_PART == 0 || QED_KERNELS_PART == (p))

namespace qedlib {

namespace {
constexpr unsigned kFull = 0xffffffffu;
// Compute threads of a step block (one tile of particles), compute warps, and all threads: plus one
// producer warp that issues the tile copies.  FP64 blocks are half as large, and two of them share an SM: a
// warp instruction holds the SM's one FP64 pipe for 16 cycles however few its lanes, so a small
// population has to reach many SMs (1e4 particles are 40 tiles of 256).  On GB300 100 steps of 1e4
// electrons in a field took 4.22 ms with tiles of 256 particles, 3.65 with 128, 3.57 with 64 and 3.48
// with 32; 20 of 1e5 in a wave 2.58, 2.50, 2.56 and 2.88.
template <typename R> constexpr int kTile = sizeof(R) == 4 ? 256 : 128;
template <typename R> constexpr int kWarps = kTile<R> / 32;
template <typename R> constexpr int kStepThreads = kTile<R> + 32;

enum LedgerSlot {
  kN0 = 0, kN1, kN2, kE0, kE1, kE2, kEmitN, kEmitE, kDrop, kEmitDef, kPairN, kPairE, kPairDef, kOorEta, kOorChi
};

// Programmatic dependent launch: a kernel's blocks may start, and run what does not depend on
// earlier kernels, while the kernel before it drains; pdl_wait returns once that one has
// completed and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Compensated (Kahan) accumulation in the working precision.
template <typename R>
struct KSum {
  R s = (R)0, c = (R)0;  // value = s - c
  __device__ __forceinline__ void add(R v) { const R y = v - c, t = s + y; c = (t - s) - y; s = t; }
  // combine with another compensated sum: exact two-sum of the leading parts, errors folded in
  __device__ __forceinline__ void merge(const KSum& o) {
    const R t = s + o.s;
    const R bb = t - s;
    const R err = (s - (t - bb)) + (o.s - bb);
    c = (c + o.c) - err;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

template <typename R>
struct Acc {
  KSum<R> e[3];
  KSum<R> emit_e, emit_def, pair_e, pair_def;
  uint32_t n[3] = {0, 0, 0};
  uint32_t oor_eta = 0, oor_chi = 0;
  uint32_t pushed_ph = 0;  // photons pushed
  uint32_t emit_n = 0, drop = 0, pair_n = 0;
};

// ----------------------------------------------------------------------------- leptons
// Fields at the particle and the Boris push of Sec. 3 (the identity where the field vanishes);
// returns the field case, and what eta_after needs.
template <typename R, bool G, int FC>
struct PushState {
  R E[3], B[3], amp;
};
template <typename R, bool G, int FC>
__device__ __forceinline__ int push_at(const StepScalars<R>& S, R x, R y, R z, R q, R dt, R u[3],
                                       PushState<R, G, FC>& ps) {
  if constexpr (FC == kFieldAny) {
    ps.amp = (R)0;
    const int fc = field_at<R, G>(S, x, y, z, ps.E, ps.B, ps.amp);
    if (fc != kNoField) boris<R>(q, dt, ps.E, ps.B, u);
    return fc;
  } else {
    R ey, ez;
    if (!plane_at<R, FC>(S, x, ey, ez, ps.amp)) return kNoField;
    boris_plane<R, FC>(q, dt, ey, ez, u);
    return kPlaneWave;
  }
}
// eta from u^{n+1/2} in the fields push_at found (Sec. 2; closed form in a plane wave)
template <typename R, bool G, int FC>
__device__ __forceinline__ R eta_after(int fc, const R u[3], R gam, const PushState<R, G, FC>& ps) {
  if constexpr (FC == kFieldAny) return eta_for<R>(fc, u, gam, ps.E, ps.B, ps.amp);
  else return fc == kNoField ? (R)0 : eta_plane<R>(u, gam, ps.amp);
}
// chi of a photon at its position (Sec. 2; closed form in a plane wave), 0 where no field
template <typename R, bool G, int FC>
__device__ __forceinline__ R chi_at(const StepScalars<R>& S, R x, R y, R z, const R k[3], R eps, int& fc) {
  if constexpr (FC == kFieldAny) {
    R E[3], B[3], amp = (R)0;
    fc = field_at<R, G>(S, x, y, z, E, B, amp);
    return chi_for<R>(fc, k, eps, E, B, amp);
  } else {
    R ey, ez, amp;
    if (!plane_at<R, FC>(S, x, ey, ez, amp)) { fc = kNoField; return (R)0; }
    fc = kPlaneWave;
    return chi_plane<R>(k, eps, amp);
  }
}

// The part of a step that every e+- takes (Sec. 3): fields at (x^n, t^n), Boris push to
// u^{n+1/2}, drift to x^{n+1}, eta, and the optical-depth decrement.  Shared by the per-step
// kernel and the multi-step kernels, so both compute the same bits.
template <typename R, bool G, int FC>
__device__ __forceinline__ R lepton_advance(const StepScalars<R>& S, const TabDev<R>& tab, const R* lnh, R q, R dt,
                                            R win_v, R& x, R& y, R& z, R u[3], Tau<R>& tau, R& gam, R& u2, int& oor) {
  using N = Num<R>;
  PushState<R, G, FC> ps;
  // where the field vanishes the push is the identity and eta = 0 (no emission)
  const int fc = push_at<R, G, FC>(S, x, y, z, q, dt, u, ps);
  u2 = dot3<R>(u, u);
  R ig;
  N::root_inv_((R)1 + u2, gam, ig);
  x = N::fma_(dt, N::fma_(u[0], ig, -win_v), x);
  y = N::fma_(dt, u[1] * ig, y);
  z = N::fma_(dt, u[2] * ig, z);
  const R eta = eta_after<R, G, FC>(fc, u, gam, ps);
  oor = 0;
  if (eta > (R)0) {
    const R lam = (R)kRatePhoton * eta * ig * lookup_h<R>(tab, lnh, eta, oor);
    tau.sub(lam * dt);
  }
  return eta;
}

// ----------------------------------------------------------------------------- deferred events
// An event (Sec. 3: a Philox draw, an inverse-CDF search, the recoil or the pair split, the
// appends) is long next to the rest of a particle's step, and rare: a few per warp per step even
// at the peak of a collision.  Taken where it is found, each warp with an event would run that
// path with one lane active.  Instead every warp writes its events into a ring in shared memory
// and takes them 32 at a time, all lanes busy, whenever 32 are waiting; what is left in the block's
// rings after its last tile of a species is taken together, 32 per warp (drain_block: the few
// events of eight warps fill one batch, where each warp ran the path for its own).  An event depends only on its particle's state
// after the push (and its id and weight), so the particles get the same bits as if each event
// were taken where it was found; only the order in which the ledger sums are accumulated changes.
constexpr int kRing = 64;  // entries per warp: fewer than 32 waiting plus at most 32 from a chunk

// A warp's ledger sums, kept beside its ring (out of the registers of the hot loop) and folded into
// the block's ledger partial at the end.
template <typename R>
struct EventSums {
  KSum<R> e[3], emit_e, emit_def, pair_e, pair_def;
  uint32_t n[3], emit_n, drop, pair_n, oor_eta, oor_chi;
};

// A lane's ledger sums over the particles of one run of tiles (one species); folded into the warp's
// sums after it.  The step kernels keep them only where the ledger can be read, in tile loops of
// their own (WANT): the others have the registers.
template <typename R>
struct RunSums {
  KSum<R> e;
  uint32_t n = 0, oor = 0;
};

template <typename R>
struct __align__(16) EventRing {
  uint32_t i[kRing];  // particle index
  R v[7][kRing];      // x, y, z after the push; u after the push (photons: k); eta (photons: chi)
  EventSums<R> sums;
  uint32_t head, count;  // of the warp's queue, where other warps read it (drain_block)
};

// Compensated warp sum of one value per lane (fixed shuffle order); lane 0 holds the result.
template <typename R>
__device__ __forceinline__ KSum<R> warp_ksum(R v) {
  KSum<R> t;
  t.s = v;
  for (int off = 16; off > 0; off >>= 1) {
    KSum<R> o;
    o.s = __shfl_down_sync(kFull, t.s, off);
    o.c = __shfl_down_sync(kFull, t.c, off);
    t.merge(o);
  }
  return t;
}

// The ring of one warp with its (warp-uniform) head and fill.
template <typename R>
struct EventQueue {
  EventRing<R>* r;
  uint32_t head, count;
};

// Enqueue the warp's events of one chunk (every lane calls this with the chunk's ballot).
template <typename R>
__device__ __forceinline__ void enqueue_event(EventQueue<R>& q, unsigned evm, bool ev, int lane, uint32_t i, R x, R y,
                                              R z, R u0, R u1, R u2, R par) {
  if (ev) {
    const uint32_t p = (q.head + q.count + (uint32_t)__popc(evm & ((1u << lane) - 1u))) & (uint32_t)(kRing - 1);
    q.r->i[p] = i;
    q.r->v[0][p] = x; q.r->v[1][p] = y; q.r->v[2][p] = z;
    q.r->v[3][p] = u0; q.r->v[4][p] = u1; q.r->v[5][p] = u2;
    q.r->v[6][p] = par;
  }
  q.count += (uint32_t)__popc(evm);
}

// Adds c (mod 2^32) to the event counts, buffer ph, of the groups that hold mask word `chunk`.
template <typename R>
__device__ __forceinline__ void count_events(const SpeciesDev<R>& sp, uint32_t ph, uint32_t chunk, uint32_t c) {
  const uint32_t f = chunk >> kFineShift;
  atomicAdd(&sp.fine[ph * event_fines(sp.cap) + f], c);
  atomicAdd(&sp.coarse[ph * event_coarses(sp.cap) + (f >> kCoarseShift)], c);
}

// One particle of a 32-particle chunk (the whole warp calls this together).  The state comes
// from the shared-memory tile; results are stored straight to global memory.  A particle whose
// optical depth ran out goes to the warp's event ring; its momentum and optical depth are
// stored when the event is taken.  The chunk's event mask counts every event as a child here;
// an emission that yields no photon (below the energy cut) takes its bit back then.
template <typename R, bool G, int FC, int kind, bool WANT>
__device__ __forceinline__ void lepton_chunk(const StepArgs<R>& a, const StepScalars<R>& S, const R* lnh,
                                             uint32_t chunk, uint32_t n, int lane, RunSums<R>& sums, EventQueue<R>& q,
                                             R x, R y, R z, R v0, R v1, R v2, const double* tau_src) {
  const SpeciesDev<R>& sp = a.sp[kind];
  const uint32_t i = chunk * 32u + (uint32_t)lane;
  const bool active = i < n;
  R u[3] = {v0, v1, v2};
  Tau<R> tau = Tau<R>::load(tau_src);
  // lanes past the last particle compute on whatever their shared-memory slots hold: nothing
  // they compute is stored, counted or queued, and the table look-ups clamp their indices (a
  // NaN position maps to the first node), so no access leaves its array
  R gam, u2;
  int oor;
  const R eta = lepton_advance<R, G, FC>(S, a.tab, lnh, kind == QED_ELECTRON ? (R)-1 : (R)1, a.dt_r, a.win_v_r, x, y,
                                         z, u, tau, gam, u2, oor);
  const bool ev = active && a.emit && tau.used_up();
  const unsigned evm = __ballot_sync(kFull, ev);
  if (evm) {
    enqueue_event<R>(q, evm, ev, lane, i, x, y, z, u[0], u[1], u[2], eta);
    if (lane == 0) count_events(sp, S.phase[kind], chunk, (uint32_t)__popc(evm));
  }
  if (lane == 0) sp.evmask[chunk] = evm;
  if (active) {
    sp.x[i] = x; sp.y[i] = y; sp.z[i] = z;
    if (!ev) {
      sp.ux[i] = u[0]; sp.uy[i] = u[1]; sp.uz[i] = u[2];
      tau.store(sp.tau + i);
    }
    if (WANT) {
      if (oor > 0) sums.oor++;
      if (!ev) { sums.e.add(gam); sums.n++; }
    }
  }
}

// Takes `take` (<= 32) events, one per lane (each lane's is entry p of `ring`): photon emission
// by an e+- (Sec. 3): photon energy from the inverse CDF of P_chi, recoil, fresh optical depths
// for the emitter and the photon, the photon appended to the photon species' append region.
// A chain of dependent loads and special functions, with scattered table reads: its latency counts
// in small runs, its loads in large ones.  The loads that need no random number come first, the append
// slots are asked for before the energies are searched, both table rows are searched at once and
// from a guide (bracket2), and the block's events share batches.  On GB300 200 steps of 1e3
// electrons went from 3.69 to 3.01 ms (searched in whole rows: 3.35), 100 steps of 1e4 on the FP64
// path, where every batch costs the slow pipe, from 5.77 to 4.20, a step of 1e6 electrons in a pulse
// from 50.8 to 45.5 us (guide alone).
// Inlined, once per kernel for either lepton: as a call, the ABI's saved registers and the spills
// around the call site cost the loop more (on GB300, 3 blocks of 288 threads per SM).
template <typename R, bool WANT>
__device__ __forceinline__ void lepton_events(const StepArgs<R>& a, uint32_t phase, int kind, const EventRing<R>* ring,
                                              uint32_t p, uint32_t take, EventSums<R>& es) {
  const SpeciesDev<R>& sp = a.sp[kind];
  const SpeciesDev<R>& dst = a.sp[2];  // photon children are appended to the photon species
  const int lane = threadIdx.x & 31;
  const bool ev = (uint32_t)lane < take;
  uint32_t i = 0;
  R x = (R)0, y = (R)0, z = (R)0, u[3] = {(R)0, (R)0, (R)0}, eta = (R)0;
  if (ev) {
    i = ring->i[p];
    x = ring->v[0][p]; y = ring->v[1][p]; z = ring->v[2][p];
    u[0] = ring->v[3][p]; u[1] = ring->v[4][p]; u[2] = ring->v[5][p];
    eta = ring->v[6][p];
  }
  // gamma from u after the push, as the push computed it
  const R u2 = dot3<R>(u, u);
  R gam, ig;
  Num<R>::root_inv_((R)1 + u2, gam, ig);
  bool child = false;
  R kx = (R)0, ky = (R)0, kz = (R)0, emitted = (R)0, def = (R)0;
  Tau<R> tau = Tau<R>::one(), ctau = Tau<R>::one();
  // whether there is a photon is known before its energy: the append slots are asked for first, and
  // their answer comes while the energies are searched
  XiSampler<R> xs;
  Uniform<R> U[4];
  if (ev) {
    const uint32_t id = sp.id[i];
    xs.prepare(a.tab, Num<R>::log_(eta));
    draw4r<R>(a.seed, a.scenario, id, a.step, (uint64_t)kind, 0, U);
    child = xs.above_cut(U[0].u);
  }
  const unsigned childm = __ballot_sync(kFull, child);
  const uint32_t nc = (uint32_t)__popc(childm);
  const int leader = __ffs(childm) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(&dst.cnt->n_app, nc);
  if (ev) {
    if (child) {
      const R xi = xs.sample(a.tab, eta, U[0].u, U[0].v);
      const R eps = xi * gam;
      const R um = Num<R>::sqrt_(u2);
      const R ium = (R)1 / um;
      const R h0 = u[0] * ium, h1 = u[1] * ium, h2 = u[2] * ium;
      kx = eps * h0; ky = eps * h1; kz = eps * h2;
      // recoil p_f = p_i - (h nu/c) phat_i (Sec. 3), or energy-conserving on request
      R umf;
      if (a.recoil_energy) { const R gf = gam - eps; umf = gf > (R)1 ? Num<R>::sqrt_(gf * gf - (R)1) : (R)0; }
      else umf = um > eps ? um - eps : (R)0;
      u[0] = umf * h0; u[1] = umf * h1; u[2] = umf * h2;
      const R gf = Num<R>::sqrt_((R)1 + umf * umf);
      // energy defect (gamma_f + eps) - gamma_i (Sec. 3.1); for the momentum-conserving recoil
      // written without cancellation as 2 eps / ((gamma_i + |u_i|)(gamma_f + gamma_i - eps))
      if (!a.recoil_energy && um > eps) def = (R)2 * eps / ((gam + um) * (gf + gam - eps));
      else def = (gf + eps) - gam;
      emitted = eps;
      gam = gf;
      ctau = Tau<R>::fresh(-Num<R>::log_(U[2].u));
    } else {
      // no photon: the event is not a child after all
      atomicAnd(&sp.evmask[i >> 5], ~(1u << (i & 31u)));
      count_events(sp, phase, i >> 5, 0xffffffffu);
    }
    tau = Tau<R>::fresh(-Num<R>::log_(U[1].u));
  }
  if (WANT) {
    const KSum<R> se = warp_ksum<R>(emitted), sd = warp_ksum<R>(def), sg = warp_ksum<R>(ev ? gam : (R)0);
    if (lane == 0) {
      es.emit_e.merge(se);
      es.emit_def.merge(sd);
      es.emit_n += nc;
      es.drop += take - nc;
      es.e[kind].merge(sg);
      es.n[kind] += take;
      if (!a.drain) { es.e[2].merge(se); es.n[2] += nc; }
    }
  }
  if (childm) {
    base = __shfl_sync(kFull, base, leader);
    if (child) {
      const uint32_t slot = base + (uint32_t)__popc(childm & ((1u << lane) - 1u));
      if (slot < dst.acap) {
        dst.ax[slot] = x; dst.ay[slot] = y; dst.az[slot] = z;
        dst.aux[slot] = kx; dst.auy[slot] = ky; dst.auz[slot] = kz;
        ctau.store(dst.atau + slot);
        dst.aparent[slot] = i | ((uint32_t)kind << 31);
        if (dst.aw) dst.aw[slot] = sp.w ? sp.w[i] : (R)1;  // the photon stands for as many
      } else {
        atomicOr(&dst.cnt->err, 1u << QED_ERR_CAPACITY);
      }
    }
  }
  if (ev) {
    sp.ux[i] = u[0]; sp.uy[i] = u[1]; sp.uz[i] = u[2];
    tau.store(sp.tau + i);
  }
  __syncwarp();  // the ring slots read above may be refilled by the next chunk
}

// The same for at most kFew events, entry p of the ring on a quad's four lanes.
template <typename R, bool WANT>
__device__ __forceinline__ void lepton_events_quads(const StepArgs<R>& a, uint32_t phase, int kind,
                                                    const EventRing<R>* ring, uint32_t p, uint32_t take, EventSums<R>& es) {
  const SpeciesDev<R>& sp = a.sp[kind];
  const SpeciesDev<R>& dst = a.sp[2];  // photon children are appended to the photon species
  const int lane = threadIdx.x & 31, part = lane % kQuad;
  const bool ev = (uint32_t)(lane / kQuad) < take, lead = ev && part == 0;
  uint32_t i = 0;
  R x = (R)0, y = (R)0, z = (R)0, u[3] = {(R)0, (R)0, (R)0}, eta = (R)0;
  if (ev) {
    i = ring->i[p];
    x = ring->v[0][p]; y = ring->v[1][p]; z = ring->v[2][p];
    u[0] = ring->v[3][p]; u[1] = ring->v[4][p]; u[2] = ring->v[5][p];
    eta = ring->v[6][p];
  }
  // gamma from u after the push, as the push computed it
  const R u2 = dot3<R>(u, u);
  const R root = Num<R>::sqrt_(part == 1 ? u2 : (R)1 + u2);  // (what root_inv_ gives on the FP64 path)
  R gam = quad_get(root, 0);
  const R um = quad_get(root, 1);
  R lnU1 = (R)0, lnU2 = (R)0;
  bool child = false;
  R kx = (R)0, ky = (R)0, kz = (R)0, emitted = (R)0, def = (R)0;
  Tau<R> tau = Tau<R>::one(), ctau = Tau<R>::one();
  // whether there is a photon is known before its energy: the append slots are asked for first, and
  // their answer comes while the energies are searched
  XiSampler<R> xs;
  Uniform<R> U[4];
  if (ev) {
    const uint32_t id = sp.id[i];
    draw4r<R>(a.seed, a.scenario, id, a.step, (uint64_t)kind, 0, U);
    const R ln = Num<R>::log_(part == 0 ? eta : (part == 1 ? U[1].u : U[2].u));
    xs.prepare(a.tab, quad_get(ln, 0));
    lnU1 = quad_get(ln, 1);
    lnU2 = quad_get(ln, 2);
    child = xs.above_cut(U[0].u);
  }
  const unsigned childm = __ballot_sync(kFull, child && part == 0);
  const uint32_t nc = (uint32_t)__popc(childm);
  const int leader = __ffs(childm) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(&dst.cnt->n_app, nc);
  if (ev) {
    if (child) {
      const R xi = xs.template sample<kQuad>(a.tab, eta, U[0].u, U[0].v);
      const R eps = xi * gam;
      const R ium = (R)1 / um;
      const R h0 = u[0] * ium, h1 = u[1] * ium, h2 = u[2] * ium;
      kx = eps * h0; ky = eps * h1; kz = eps * h2;
      // recoil p_f = p_i - (h nu/c) phat_i (Sec. 3), or energy-conserving on request
      R umf;
      if (a.recoil_energy) { const R gf = gam - eps; umf = gf > (R)1 ? Num<R>::sqrt_(gf * gf - (R)1) : (R)0; }
      else umf = um > eps ? um - eps : (R)0;
      u[0] = umf * h0; u[1] = umf * h1; u[2] = umf * h2;
      const R gf = Num<R>::sqrt_((R)1 + umf * umf);
      // energy defect (gamma_f + eps) - gamma_i (Sec. 3.1); for the momentum-conserving recoil
      // written without cancellation as 2 eps / ((gamma_i + |u_i|)(gamma_f + gamma_i - eps))
      if (!a.recoil_energy && um > eps) def = (R)2 * eps / ((gam + um) * (gf + gam - eps));
      else def = (gf + eps) - gam;
      emitted = eps;
      gam = gf;
      ctau = Tau<R>::fresh(-lnU2);
    } else if (lead) {
      // no photon: the event is not a child after all
      atomicAnd(&sp.evmask[i >> 5], ~(1u << (i & 31u)));
      count_events(sp, phase, i >> 5, 0xffffffffu);
    }
    tau = Tau<R>::fresh(-lnU1);
  }
  if (WANT) {
    const KSum<R> se = warp_ksum<R>(part == 0 ? emitted : (R)0), sd = warp_ksum<R>(part == 0 ? def : (R)0),
                  sg = warp_ksum<R>(lead ? gam : (R)0);
    if (lane == 0) {
      es.emit_e.merge(se);
      es.emit_def.merge(sd);
      es.emit_n += nc;
      es.drop += take - nc;
      es.e[kind].merge(sg);
      es.n[kind] += take;
      if (!a.drain) { es.e[2].merge(se); es.n[2] += nc; }
    }
  }
  if (childm) {
    base = __shfl_sync(kFull, base, leader);
    if (child && lead) {
      const uint32_t slot = base + (uint32_t)__popc(childm & ((1u << lane) - 1u));
      if (slot < dst.acap) {
        dst.ax[slot] = x; dst.ay[slot] = y; dst.az[slot] = z;
        dst.aux[slot] = kx; dst.auy[slot] = ky; dst.auz[slot] = kz;
        ctau.store(dst.atau + slot);
        dst.aparent[slot] = i | ((uint32_t)kind << 31);
        if (dst.aw) dst.aw[slot] = sp.w ? sp.w[i] : (R)1;  // the photon stands for as many
      } else {
        atomicOr(&dst.cnt->err, 1u << QED_ERR_CAPACITY);
      }
    }
  }
  if (lead) {
    sp.ux[i] = u[0]; sp.uy[i] = u[1]; sp.uz[i] = u[2];
    tau.store(sp.tau + i);
  }
  __syncwarp();  // the ring slots read above may be refilled by the next chunk
}

// ----------------------------------------------------------------------------- photons
// The part of a step that every photon takes: chi at (x^n, t^n), the pair-rate decrement of the
// optical depth, and the drift at c along k (k does not change between events).
template <typename R, bool G, int FC>
__device__ __forceinline__ R photon_advance(const StepScalars<R>& S, const TabDev<R>& tab, const R* lnT, R dt, R win_v,
                                            R& x, R& y, R& z, const R k[3], Tau<R>& tau, R& eps, R& ie, int& oor) {
  using N = Num<R>;
  N::root_inv_(dot3<R>(k, k), eps, ie);
  int fc;
  const R chi = chi_at<R, G, FC>(S, x, y, z, k, eps, fc);
  oor = 0;
  if (chi > (R)0) {
    const R lam = (R)kAlpha * chi * ie * lookup_T<R>(tab, lnT, chi, oor);
    tau.sub(lam * dt);
  }
  x = N::fma_(dt, N::fma_(k[0], ie, -win_v), x);  // null geodesic at c along khat
  y = N::fma_(dt, k[1] * ie, y);
  z = N::fma_(dt, k[2] * ie, z);
  return chi;
}

template <typename R, bool G, int FC, bool WANT>
__device__ __forceinline__ void photon_chunk(const StepArgs<R>& a, const StepScalars<R>& S, const R* lnT,
                                             uint32_t chunk, uint32_t n, int lane, RunSums<R>& sums, uint32_t& pushed_ph,
                                             uint32_t& tau_ph, EventQueue<R>& q,
                                             R x, R y, R z, R k0, R k1, R k2, const double* tau_src) {
  const SpeciesDev<R>& sp = a.sp[2];
  const uint32_t i = chunk * 32u + (uint32_t)lane;
  Tau<R> tau = Tau<R>::load(tau_src);
  const bool alive = i < n && !tau.dead();  // converted photons stay as holes until compaction
  R k[3] = {k0, k1, k2};
  // dead or past-the-end lanes compute on what their slots hold; none of it is stored (see
  // lepton_chunk)
  R eps, ie;
  int oor;
  const R chi = photon_advance<R, G, FC>(S, a.tab, lnT, a.dt_r, a.win_v_r, x, y, z, k, tau, eps, ie, oor);
  if (alive) pushed_ph++;
  // a photon outside any field keeps its optical depth: only its position is stored
  const bool tau_moves = alive && chi > (R)0;
  if (tau_moves) tau_ph++;

  // a photon whose optical depth ran out always converts: its pair is counted here
  const bool ev = alive && a.pairs && tau.used_up();
  const unsigned evm = __ballot_sync(kFull, ev);
  if (evm) {
    enqueue_event<R>(q, evm, ev, lane, i, x, y, z, k[0], k[1], k[2], chi);
    if (lane == 0) {
      const uint32_t c = (uint32_t)__popc(evm);
      count_events(sp, S.phase[2], chunk, c);
      atomicAdd(&sp.cnt->n_dead, c);
    }
  }
  if (lane == 0) sp.evmask[chunk] = evm;
  if (alive) {
    sp.x[i] = x; sp.y[i] = y; sp.z[i] = z;  // k is unchanged between events
    if (!ev && tau_moves) tau.store(sp.tau + i);
    if (WANT) {
      if (oor > 0) sums.oor++;
      if (!ev) { sums.e.add(eps); sums.n++; }
    }
  }
}

// Takes `take` (<= 32) events, one per lane (each lane's is entry p of `ring`): pair creation
// by a photon (Sec. 3): the energy split from the inverse CDF of P_f, the electron and the
// positron along k with fresh optical depths, appended to their species' append regions; the
// photon is annihilated (its optical depth becomes +inf, a hole until compaction).  Inlined
// for the same reason as lepton_events.
template <typename R, bool WANT>
__device__ __forceinline__ void photon_events(const StepArgs<R>& a, const EventRing<R>* ring, uint32_t p, uint32_t take,
                                              EventSums<R>& es) {
  const SpeciesDev<R>& sp = a.sp[2];
  const int lane = threadIdx.x & 31;
  const bool ev = (uint32_t)lane < take;
  uint32_t i = 0;
  R x = (R)0, y = (R)0, z = (R)0, k[3] = {(R)0, (R)0, (R)1}, chi = (R)0;
  if (ev) {
    i = ring->i[p];
    x = ring->v[0][p]; y = ring->v[1][p]; z = ring->v[2][p];
    k[0] = ring->v[3][p]; k[1] = ring->v[4][p]; k[2] = ring->v[5][p];
    chi = ring->v[6][p];
  }
  // the photon energy as the push computed it
  R eps, ie;
  Num<R>::root_inv_(dot3<R>(k, k), eps, ie);
  R ue[3] = {(R)0, (R)0, (R)0}, up[3] = {(R)0, (R)0, (R)0};
  R converted = (R)0, def = (R)0, gm = (R)0, gp = (R)0;
  Tau<R> te = Tau<R>::one(), tp = Tau<R>::one();
  uint32_t be = 0, bp = 0;  // append slots, asked for first
  if (lane == 0) {
    be = atomicAdd(&a.sp[0].cnt->n_app, take);
    bp = atomicAdd(&a.sp[1].cnt->n_app, take);
  }
  if (ev) {
    Uniform<R> U[4];
    draw4r<R>(a.seed, a.scenario, sp.id[i], a.step, (uint64_t)QED_PHOTON, 0, U);
    const R f = sample_f<R>(a.tab, Num<R>::log_(chi), U[0].u, U[0].v);
    R se = (R)1 - f, sq = f;  // the positron takes f h nu (Sec. 3)
    if (a.recoil_energy && eps >= (R)2) {
      const R g1 = (R)1 + f * (eps - (R)2), g0 = (R)1 + ((R)1 - f) * (eps - (R)2);
      sq = Num<R>::sqrt_(g1 * g1 - (R)1) * ie;
      se = Num<R>::sqrt_(g0 * g0 - (R)1) * ie;
    }
    for (int c = 0; c < 3; ++c) { ue[c] = se * k[c]; up[c] = sq * k[c]; }
    const R pe = se * eps, pp = sq * eps;
    gm = Num<R>::sqrt_((R)1 + pe * pe);
    gp = Num<R>::sqrt_((R)1 + pp * pp);
    // defect (gamma_- + gamma_+) - eps (Sec. 3.1); for the momentum split it is exactly
    // 1/(gamma_- + p_-) + 1/(gamma_+ + p_+), written so to avoid cancellation
    if (!(a.recoil_energy && eps >= (R)2)) def = (R)1 / (gm + pe) + (R)1 / (gp + pp);
    else def = (gm + gp) - eps;
    converted = eps;
    te = Tau<R>::fresh(-Num<R>::log_(U[1].u));
    tp = Tau<R>::fresh(-Num<R>::log_(U[2].u));
  }
  if (WANT) {
    const KSum<R> se = warp_ksum<R>(converted), sd = warp_ksum<R>(def);
    const KSum<R> s0 = warp_ksum<R>(gm), s1 = warp_ksum<R>(gp);
    if (lane == 0) {
      es.pair_e.merge(se);
      es.pair_def.merge(sd);
      es.pair_n += take;
      es.e[0].merge(s0); es.n[0] += take;
      es.e[1].merge(s1); es.n[1] += take;
    }
  }
  be = __shfl_sync(kFull, be, 0);
  bp = __shfl_sync(kFull, bp, 0);
  if (ev) {
    const uint32_t r = (uint32_t)lane;  // the events fill lanes 0 .. take-1
    const SpeciesDev<R>& de = a.sp[0];
    const SpeciesDev<R>& dp = a.sp[1];
    if (be + r < de.acap) {
      const uint32_t s = be + r;
      de.ax[s] = x; de.ay[s] = y; de.az[s] = z;
      de.aux[s] = ue[0]; de.auy[s] = ue[1]; de.auz[s] = ue[2];
      te.store(de.atau + s);
      de.aparent[s] = i;
      if (de.aw) de.aw[s] = sp.w ? sp.w[i] : (R)1;
    } else {
      atomicOr(&de.cnt->err, 1u << QED_ERR_CAPACITY);
    }
    if (bp + r < dp.acap) {
      const uint32_t s = bp + r;
      dp.ax[s] = x; dp.ay[s] = y; dp.az[s] = z;
      dp.aux[s] = up[0]; dp.auy[s] = up[1]; dp.auz[s] = up[2];
      tp.store(dp.atau + s);
      dp.aparent[s] = i;
      if (dp.aw) dp.aw[s] = sp.w ? sp.w[i] : (R)1;
    } else {
      atomicOr(&dp.cnt->err, 1u << QED_ERR_CAPACITY);
    }
    Tau<R>::infinite().store(sp.tau + i);  // the photon is annihilated
  }
  __syncwarp();  // the ring slots read above may be refilled by the next chunk
}

// The same for at most kFew events, entry p of the ring on a quad's four lanes: the even lanes take the
// electron, the odd ones the positron.
template <typename R, bool WANT>
__device__ __forceinline__ void photon_events_quads(const StepArgs<R>& a, const EventRing<R>* ring, uint32_t p, uint32_t take,
                                                    EventSums<R>& es) {
  const SpeciesDev<R>& sp = a.sp[2];
  const int lane = threadIdx.x & 31, part = lane % kQuad, c = part & 1;
  const uint32_t r = (uint32_t)(lane / kQuad);  // the event among those taken
  const bool ev = r < take, lead = ev && part == 0;
  uint32_t i = 0;
  R x = (R)0, y = (R)0, z = (R)0, k[3] = {(R)0, (R)0, (R)1}, chi = (R)0;
  if (ev) {
    i = ring->i[p];
    x = ring->v[0][p]; y = ring->v[1][p]; z = ring->v[2][p];
    k[0] = ring->v[3][p]; k[1] = ring->v[4][p]; k[2] = ring->v[5][p];
    chi = ring->v[6][p];
  }
  // the photon energy as the push computed it
  R eps, ie;
  Num<R>::root_inv_(dot3<R>(k, k), eps, ie);
  // the lane's particle: its share of k, gamma and optical depth; the positron's gamma
  R share = (R)0, gam = (R)0, gp = (R)0, converted = (R)0, def = (R)0;
  Tau<R> tau = Tau<R>::one();
  uint32_t be = 0, bp = 0;  // append slots, asked for first
  if (lane == 0) {
    be = atomicAdd(&a.sp[0].cnt->n_app, take);
    bp = atomicAdd(&a.sp[1].cnt->n_app, take);
  }
  if (ev) {
    Uniform<R> U[4];
    draw4r<R>(a.seed, a.scenario, sp.id[i], a.step, (uint64_t)QED_PHOTON, 0, U);
    const R ln = Num<R>::log_(part == 0 ? chi : (part == 1 ? U[1].u : U[2].u));
    const R f = sample_f<R, kQuad>(a.tab, quad_get(ln, 0), U[0].u, U[0].v);
    const bool keep = a.recoil_energy && eps >= (R)2;
    const R fc = c ? f : (R)1 - f;  // the positron takes f h nu (Sec. 3)
    share = fc;
    if (keep) {
      const R g1 = (R)1 + fc * (eps - (R)2);
      share = Num<R>::sqrt_(g1 * g1 - (R)1) * ie;
    }
    const R pc = share * eps;
    gam = Num<R>::sqrt_((R)1 + pc * pc);
    gp = quad_get(gam, 1);
    const R inv = (R)1 / (gam + pc), inv_p = quad_get(inv, 1);
    tau = Tau<R>::fresh(-quad_get(ln, 1 + c));
    // defect (gamma_- + gamma_+) - eps (Sec. 3.1); for the momentum split it is exactly
    // 1/(gamma_- + p_-) + 1/(gamma_+ + p_+), written so to avoid cancellation
    def = keep ? (gam + gp) - eps : inv + inv_p;
    converted = eps;
  }
  if (WANT) {
    const KSum<R> se = warp_ksum<R>(lead ? converted : (R)0), sd = warp_ksum<R>(lead ? def : (R)0);
    const KSum<R> s0 = warp_ksum<R>(lead ? gam : (R)0), s1 = warp_ksum<R>(lead ? gp : (R)0);
    if (lane == 0) {
      es.pair_e.merge(se);
      es.pair_def.merge(sd);
      es.pair_n += take;
      es.e[0].merge(s0); es.n[0] += take;
      es.e[1].merge(s1); es.n[1] += take;
    }
  }
  be = __shfl_sync(kFull, be, 0);
  bp = __shfl_sync(kFull, bp, 0);
  if (ev && part < 2) {
    const SpeciesDev<R>& d = c ? a.sp[1] : a.sp[0];
    const uint32_t s = (c ? bp : be) + r;
    if (s < d.acap) {
      d.ax[s] = x; d.ay[s] = y; d.az[s] = z;
      d.aux[s] = share * k[0]; d.auy[s] = share * k[1]; d.auz[s] = share * k[2];
      tau.store(d.atau + s);
      d.aparent[s] = i;
      if (d.aw) d.aw[s] = sp.w ? sp.w[i] : (R)1;
    } else {
      atomicOr(&d.cnt->err, 1u << QED_ERR_CAPACITY);
    }
  }
  if (lead) Tau<R>::infinite().store(sp.tau + i);  // the photon is annihilated
  __syncwarp();  // the ring slots read above may be refilled by the next chunk
}

// One pipeline stage: a tile of consecutive particles of one species, a chunk of 32 per compute warp.

template <typename R>
struct TileBuf;

// measured on GB300 at 3 resident blocks per SM (72 registers; 4 blocks per SM spill): on the
// head-on collision of 1e6 electrons 3, 4 and 6 stages tie (2 stages are 7% slower, 8 stages, at
// 2 blocks per SM, 18%); on the 256-scenario scan 4 stages are 16% faster than 6: the shared
// memory they leave to L1 holds the spilled registers and the arguments and tables the event
// paths read
#ifndef QED_STAGES
#define QED_STAGES 4
#endif
#ifndef QED_STEP_MIN_BLOCKS
#define QED_STEP_MIN_BLOCKS 3
#endif
#ifndef QED_BATCH_MIN_BLOCKS
#define QED_BATCH_MIN_BLOCKS 3
#endif
constexpr int kStages = QED_STAGES;  // tile copies in flight per block
constexpr uint32_t kWaitLimit = 1u << 16;  // mbarrier polls (<= 20 us each) before a copy is declared lost

template <typename R>
struct TileBuf {
  R x[kTile<R>], y[kTile<R>], z[kTile<R>], ux[kTile<R>], uy[kTile<R>], uz[kTile<R>];
  double tau[kTile<R>];
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t floor16(uint32_t b) { return b & ~15u; }

// Tile t of the step (over the concatenated species) -> species and tile index in it.
__device__ __forceinline__ void decode_tile(uint32_t t, uint32_t T0, uint32_t T1, int& s, uint32_t& j) {
  if (t < T0) { s = 0; j = t; }
  else if (t < T0 + T1) { s = 1; j = t - T0; }
  else { s = 2; j = t - T0 - T1; }
}

// Source arrays of a species.
template <typename R>
struct TileSrc {
  const R *x, *y, *z, *ux, *uy, *uz;
  const double* tau;
};
template <typename R>
__device__ __forceinline__ TileSrc<R> tile_src(const SpeciesDev<R>& p) {
  return {p.x, p.y, p.z, p.ux, p.uy, p.uz, p.tau};
}

// Tiles of a photon window's conversions, each a share of its groups of 1024 photons: about two
// groups per warp, and at most one tile per block.
__device__ __forceinline__ uint32_t conversion_tiles(uint32_t win_n, uint32_t nblk) {
  return min(nblk, ((win_n >> 10) + 15u) / 16u);
}

// Thread 0 issues the bulk copies of the block's k-th tile into stage k % kStages.
template <typename R>
__device__ __forceinline__ void issue_tile(const StepArgs<R>& a, TileBuf<R>* buf, uint64_t* bar, uint32_t k, uint32_t n0,
                                        uint32_t n1, uint32_t n2, uint32_t win_n, uint32_t blk, uint32_t nblk) {
  const uint32_t T0 = (n0 + kTile<R> - 1) / kTile<R>, T1 = (n1 + kTile<R> - 1) / kTile<R>, T2 = (n2 - win_n + kTile<R> - 1) / kTile<R>;
  const uint32_t t = blk + k * nblk;
  if (t >= T0 + T1 + T2) {
    // a tile of a photon window's conversions: nothing to copy
    if (t < T0 + T1 + T2 + conversion_tiles(win_n, nblk)) mbar_arrive(&bar[k % kStages]);
    return;
  }
  int s; uint32_t j;
  decode_tile(t, T0, T1, s, j);
  const TileSrc<R> src = tile_src(a.sp[s]);
  const uint32_t ns = s == 0 ? n0 : (s == 1 ? n1 : n2);
  const uint32_t first = (s == 2 ? win_n : 0u) + j * kTile<R>;
  const uint32_t valid = min((uint32_t)kTile<R>, ns - first);
  // arrays start 16-byte aligned and tiles start at multiples of 128 particles, so every source
  // is 16-byte aligned; only whole 16-byte pieces are copied (no read past the last particle),
  // the ragged remainder of the last tile is read with plain loads by its threads
  const uint32_t br = floor16(valid * (uint32_t)sizeof(R)), bt = floor16(valid * 8u);
  TileBuf<R>& b = buf[k % kStages];
  uint64_t* bb = &bar[k % kStages];
  mbar_arrive_expect_tx(bb, 6u * br + bt);
  if (br) {
    bulk_load(b.x, src.x + first, br, bb);
    bulk_load(b.y, src.y + first, br, bb);
    bulk_load(b.z, src.z + first, br, bb);
    bulk_load(b.ux, src.ux + first, br, bb);
    bulk_load(b.uy, src.uy + first, br, bb);
    bulk_load(b.uz, src.uz + first, br, bb);
  }
  if (bt) bulk_load(b.tau, src.tau + first, bt, bb);
}

// barrier among the compute warps only (the producer warp does not take part)
template <typename R>
__device__ __forceinline__ void compute_warps_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kTile<R>) : "memory"); }

// Fixed-order block reduction of the ledger partials in the working precision: compensated
// sums are combined pairwise (two-sum), counts as integers; only the block totals become FP64
// (an FP64 shuffle tree here took a quarter of the kernel on GB300's slow FP64 pipe).
// (The multi-step passes; every thread of their W warps calls this.)
constexpr int kCounts = 8;
template <typename R, int W>
__device__ __forceinline__ void write_ledger_partial(const Acc<R>& acc, double* ledger_part, uint32_t blk) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  KSum<R> f[7] = {acc.e[0], acc.e[1], acc.e[2], acc.emit_e, acc.emit_def, acc.pair_e, acc.pair_def};
  uint32_t c[kCounts] = {acc.n[0], acc.n[1], acc.n[2], acc.emit_n, acc.drop, acc.pair_n, acc.oor_eta, acc.oor_chi};
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    KSum<R> t = f[q];
    for (int off = 16; off > 0; off >>= 1) {
      KSum<R> o;
      o.s = __shfl_down_sync(kFull, t.s, off);
      o.c = __shfl_down_sync(kFull, t.c, off);
      t.merge(o);
    }
    f[q] = t;
  }
#pragma unroll
  for (int q = 0; q < kCounts; ++q)
    for (int off = 16; off > 0; off >>= 1) c[q] += __shfl_down_sync(kFull, c[q], off);
  __shared__ KSum<R> s_fr[W][7];
  __shared__ uint32_t s_cr[W][kCounts];
  if (lane == 0) {
    for (int q = 0; q < 7; ++q) s_fr[warp][q] = f[q];
    for (int q = 0; q < kCounts; ++q) s_cr[warp][q] = c[q];
  }
  __syncthreads();
  if (threadIdx.x < kLedgerN) {
    const int k = threadIdx.x;
    int fs = -1, cs = -1;  // where ledger field k comes from
    switch (k) {
      case kN0: cs = 0; break;       case kN1: cs = 1; break;       case kN2: cs = 2; break;
      case kE0: fs = 0; break;       case kE1: fs = 1; break;       case kE2: fs = 2; break;
      case kEmitN: cs = 3; break;    case kEmitE: fs = 3; break;    case kDrop: cs = 4; break;
      case kEmitDef: fs = 4; break;  case kPairN: cs = 5; break;    case kPairE: fs = 5; break;
      case kPairDef: fs = 6; break;  case kOorEta: cs = 6; break;   case kOorChi: cs = 7; break;
      default: break;
    }
    double t = 0.0;
    if (fs >= 0) {
      KSum<R> acc_b = s_fr[0][fs];
      for (int w = 1; w < W; ++w) acc_b.merge(s_fr[w][fs]);
      t = acc_b.value();
    } else if (cs >= 0) {
      uint32_t n = 0;
      for (int w = 0; w < W; ++w) n += s_cr[w][cs];
      t = (double)n;
    }
    ledger_part[(size_t)blk * kLedgerN + k] = t;
  }
}

// The block's ledger partial from its compute warps' sums (threads 0 .. kLedgerN - 1, after a barrier):
// combined in warp order in the working precision, as write_ledger_partial does.
template <typename R>
__device__ __forceinline__ void write_step_partial(const EventRing<R>* ring, double* ledger_part, uint32_t blk) {
  const int k = threadIdx.x;
  if (k >= kLedgerN) return;
  KSum<R> t;
  uint32_t n = 0;
  for (int w = 0; w < kWarps<R>; ++w) {
    const EventSums<R>& es = ring[w].sums;
    switch (k) {
      case kN0: case kN1: case kN2: n += es.n[k - kN0]; break;
      case kE0: case kE1: case kE2: t.merge(es.e[k - kE0]); break;
      case kEmitN: n += es.emit_n; break;
      case kEmitE: t.merge(es.emit_e); break;
      case kDrop: n += es.drop; break;
      case kEmitDef: t.merge(es.emit_def); break;
      case kPairN: n += es.pair_n; break;
      case kPairE: t.merge(es.pair_e); break;
      case kPairDef: t.merge(es.pair_def); break;
      case kOorEta: n += es.oor_eta; break;
      default: n += es.oor_chi; break;
    }
  }
  ledger_part[(size_t)blk * kLedgerN + k] = n ? (double)n : t.value();
}

// The photon push counters of a block: summed over its warps in shared memory, then added to the
// scenario's work counters (the e+- pushes follow from the particle counts).
__device__ __forceinline__ void add_work(uint32_t pushed_ph, uint32_t tau_ph, uint32_t* s_work, int lane) {
  const uint32_t p = __reduce_add_sync(kFull, pushed_ph), t = __reduce_add_sync(kFull, tau_ph);
  if (lane == 0 && p) {
    atomicAdd(&s_work[0], p);
    atomicAdd(&s_work[1], t);
  }
}
__device__ __forceinline__ void flush_work(uint32_t* s_work, unsigned long long* work) {
  if (s_work[0]) atomicAdd(&work[1], (unsigned long long)s_work[0]);
  if (s_work[1]) atomicAdd(&work[5], (unsigned long long)s_work[1]);
}

// A run of tiles of one (slot, species): global tiles [g_lo, g_hi) of the step's tile space, which
// hold the species' particles [base, n); slot_lo is the slot's first tile (batches).  s = 3: tiles
// without particles, for the conversions that a photon window found among its first n photons.
struct TileRun {
  int slot = 0, s = -1;
  uint32_t g_lo = 0, g_hi = 0, slot_lo = 0;
  uint32_t n = 0, base = 0;
};

// What a block's compute warps share: the tile pipeline and the event rings.
template <typename R>
struct StepPipe {
  TileBuf<R>* buf;
  uint64_t *full, *empty;
  EventRing<R>* ring;
  const R *lnh, *lnT;
  int* abort;
  uint32_t blk, nblk;
};

// The state of one compute warp.
template <typename R>
struct WarpState {
  EventQueue<R> q;
  uint32_t pushed_ph = 0, tau_ph = 0;  // (per lane) photons pushed; those in a field
  uint32_t k = 0;        // tiles the block has passed
  bool stopped = false;  // a wait gave up: no more waits or work, but every barrier is kept
};

// Waits for the data of the block's tile w.k; false once a wait gave up.
template <typename R>
__device__ __forceinline__ bool tile_ready(const StepPipe<R>& P, WarpState<R>& w) {
  if (!w.stopped && (*P.abort || !mbar_wait_bounded(&P.full[w.k % kStages], (w.k / kStages) & 1u, kWaitLimit))) {
    *P.abort = 1;
    w.stopped = true;
  }
  return !w.stopped;
}

// Tiles of one run, from the block's w.k-th on, until 32 events wait (true: take them and call again)
// or the block's tiles of the run are done.  Compiled per field class FC and species SP, so no tile
// dispatches on either (and the species' arrays are constants); the events' code, which is long, is
// kept out of it.
template <typename R, bool G, int FC, int SP, bool WANT>
__device__ __forceinline__ bool run_tiles(const StepArgs<R>& A, const StepScalars<R>& S, const StepPipe<R>& P,
                                          const TileRun& run, WarpState<R>& w, RunSums<R>& sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t n = run.n, base = SP == 2 ? run.base : 0u;
  const uint32_t last = n > base ? (n - base - 1u) / (uint32_t)kTile<R> : 0u;  // the only tile that can be ragged
  const uint32_t valid = n - base - last * (uint32_t)kTile<R>;
  const uint32_t in_r = floor16(valid * (uint32_t)sizeof(R)) / (uint32_t)sizeof(R);
  const uint32_t in_t = floor16(valid * 8u) / 8u;
  const bool ragged = in_r < valid || in_t < valid;
  const uint32_t r = threadIdx.x;
  for (;; ++w.k) {
    const uint32_t g = P.blk + w.k * P.nblk;
    // (tested in this order, with its own return, the loop is 3% faster than with one test of the count)
    if (g >= run.g_hi) return w.q.count >= 32u;  // what is left is fewer than 32
    if (w.q.count >= 32u) return true;
    if (!tile_ready(P, w)) continue;
    const int st = (int)(w.k % kStages);
    TileBuf<R>& b = P.buf[st];
    const uint32_t j = g - run.g_lo;
    // the ragged remainder of a species' last tile: each thread reads its own particle
    if (ragged && j == last && r < valid && (r >= in_r || r >= in_t)) {
      const SpeciesDev<R>& gs = A.sp[SP];
      const uint32_t gi = base + j * kTile<R> + r;
      if (r >= in_r) {
        b.x[r] = gs.x[gi]; b.y[r] = gs.y[gi]; b.z[r] = gs.z[gi];
        b.ux[r] = gs.ux[gi]; b.uy[r] = gs.uy[gi]; b.uz[r] = gs.uz[gi];
      }
      if (r >= in_t) b.tau[r] = gs.tau[gi];
    }
    const uint32_t chunk = base / 32u + j * kWarps<R> + warp;
    if constexpr (SP == 2)
      photon_chunk<R, G, FC, WANT>(A, S, P.lnT, chunk, n, lane, sums, w.pushed_ph, w.tau_ph, w.q, b.x[r], b.y[r], b.z[r],
                                   b.ux[r], b.uy[r], b.uz[r], &b.tau[r]);
    else
      lepton_chunk<R, G, FC, SP, WANT>(A, S, P.lnh, chunk, n, lane, sums, w.q, b.x[r], b.y[r], b.z[r], b.ux[r], b.uy[r],
                                       b.uz[r], &b.tau[r]);
    __syncwarp();
    if (lane == 0) mbar_arrive(&P.empty[st]);
  }
}

// The conversions that the photon window found for this step, as a run without particles: its T tiles
// share the window's groups of 1024 photons, neighbouring groups with different warps; a group whose
// flag has the step's bit is done by the whole warp (one mask word per lane).  Makes the step's event-mask words and counts of the
// group and queues the events, as if the photons had been pushed by this step.  A converted photon
// waits with its step and its chi in the place of its optical depth, at its position after the
// push.  Returns true when 32 events wait, with its place kept in `c`.
struct ConversionState {
  bool open = false;
  uint32_t first = 0, next = 0, w = 0, m = 0;
  unsigned todo = 0;
};
template <typename R>
__device__ __forceinline__ bool run_conversions(const StepArgs<R>& a, const StepScalars<R>& S, const StepPipe<R>& P,
                                                const TileRun& run, WarpState<R>& ws, ConversionState& c) {
  const SpeciesDev<R>& sp = a.sp[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t groups = run.n >> 10, stride = (run.g_hi - run.g_lo) * kWarps<R>;
  for (;;) {
    if (!c.open) {
      const uint32_t t = P.blk + ws.k * P.nblk;
      if (t >= run.g_hi) return false;
      if (!tile_ready(P, ws)) { ++ws.k; continue; }
      c.first = c.next = (t - run.g_lo) * kWarps<R> + (uint32_t)warp;
      c.open = true;
    }
    while (__any_sync(kFull, c.m != 0u) || c.todo || c.next < groups) {
      if (!__any_sync(kFull, c.m != 0u)) {
        if (!c.todo) {  // the flags of the warp's next 32 groups
          c.first = c.next;
          c.next += 32u * stride;
          const uint32_t mine = c.first + (uint32_t)lane * stride, bit = 1u << a.win_s;
          const uint32_t fl = mine < groups ? sp.wflag[mine] : 0u;
          c.todo = __ballot_sync(kFull, (fl & bit) != 0u);
          if ((fl & bit) && !(fl >> a.win_s >> 1)) sp.wflag[mine] = 0u;  // the group's last step with conversions
          continue;
        }
        const uint32_t g = c.first + (uint32_t)(__ffs(c.todo) - 1) * stride;
        c.todo &= c.todo - 1u;
        c.w = g * 32u + (uint32_t)lane;
        for (uint32_t left = sp.cmask[c.w]; left; left &= left - 1u) {
          const uint32_t b = (uint32_t)__ffs(left) - 1u;
          if (Tau<R>::load(sp.tau + c.w * 32u + b).window_step() == a.win_s) c.m |= 1u << b;
        }
        sp.evmask[c.w] = c.m;
        const uint32_t cnt = __reduce_add_sync(kFull, (uint32_t)__popc(c.m));
        if (lane == 0) {
          count_events(sp, S.phase[2], g * 32u, cnt);
          atomicAdd(&sp.cnt->n_dead, cnt);
        }
      }
      const bool ev = c.m != 0u;
      uint32_t i = 0;
      R x = (R)0, y = (R)0, z = (R)0, k0 = (R)0, k1 = (R)0, k2 = (R)0, chi = (R)0;
      if (ev) {
        i = c.w * 32u + (uint32_t)__ffs(c.m) - 1u;
        x = sp.x[i]; y = sp.y[i]; z = sp.z[i];
        k0 = sp.ux[i]; k1 = sp.uy[i]; k2 = sp.uz[i];
        chi = Tau<R>::load(sp.tau + i).window_chi();
        c.m &= c.m - 1u;
      }
      enqueue_event<R>(ws.q, __ballot_sync(kFull, ev), ev, lane, i, x, y, z, k0, k1, k2, chi);
      __syncwarp();
      if (ws.q.count >= 32u) return true;
    }
    c.open = false;
    if (lane == 0) mbar_arrive(&P.empty[ws.k % kStages]);
    ++ws.k;
  }
}

// The lanes' sums of a run into the warp's (fixed shuffle order).
template <typename R>
__device__ __forceinline__ void fold_run_sums(const RunSums<R>& sums, int s, EventSums<R>& es) {
  KSum<R> t = sums.e;
  for (int off = 16; off > 0; off >>= 1) {
    KSum<R> o;
    o.s = __shfl_down_sync(kFull, t.s, off);
    o.c = __shfl_down_sync(kFull, t.c, off);
    t.merge(o);
  }
  const uint32_t n = __reduce_add_sync(kFull, sums.n), oor = __reduce_add_sync(kFull, sums.oor);
  if ((threadIdx.x & 31) == 0) {
    es.e[s].merge(t);
    es.n[s] += n;
    if (s == 2) es.oor_chi += oor;
    else es.oor_eta += oor;
  }
}

// Up to this many events per warp are taken in quads, on the FP64 path: what bounds a small step's events
// there is the chain of FP64 instructions (350 of them for a batch of 1 to 32 events, at some 70
// cycles each; in quads 150).  On GB300 100 steps of 1e4 electrons went from 3.65 to 3.0 ms; the
// mixed path, whose registers are full, lost 2 to 5% to the second form in the kernel and has only one.
template <typename R> constexpr uint32_t kFew = sizeof(R) == 8 ? 32 / kQuad : 0;

// The block's tiles of one run of leptons and all their events (every compute warp of the block calls
// this): a warp takes 32 events whenever it has them, and what is left in the block's rings is
// taken together, 32 per warp (or fewer, in quads): rings with fewer than 32 each make at most one
// batch per warp.
template <typename R, bool G, bool WANT>
__device__ __forceinline__ void run_leptons(const StepArgs<R>& A, const StepScalars<R>& S, const StepPipe<R>& P,
                                            const TileRun& run, WarpState<R>& w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RunSums<R> sums;
  for (bool more = true; more;) {
    if (!G && S.kind == QED_FIELD_PLANE_LP)
      more = run.s == 0 ? run_tiles<R, G, G ? kFieldAny : kFieldLP, 0, WANT>(A, S, P, run, w, sums)
                        : run_tiles<R, G, G ? kFieldAny : kFieldLP, 1, WANT>(A, S, P, run, w, sums);
    else if (!G && S.kind == QED_FIELD_PLANE_CP)
      more = run.s == 0 ? run_tiles<R, G, G ? kFieldAny : kFieldCP, 0, WANT>(A, S, P, run, w, sums)
                        : run_tiles<R, G, G ? kFieldAny : kFieldCP, 1, WANT>(A, S, P, run, w, sums);
    else
      more = run.s == 0 ? run_tiles<R, G, kFieldAny, 0, WANT>(A, S, P, run, w, sums)
                        : run_tiles<R, G, kFieldAny, 1, WANT>(A, S, P, run, w, sums);
    const EventRing<R>* src = w.q.r;
    uint32_t p = w.q.head + (uint32_t)lane, take = 32u;
    [[maybe_unused]] bool few = false;
    if (more) {  // 32 of the warp's own
      w.q.head += 32u;
      w.q.count -= 32u;
    } else {
      if (w.stopped) w.q.count = 0;  // (an unfinished step: QED_ERR_TIMEOUT)
      if (lane == 0) { w.q.r->head = w.q.head; w.q.r->count = w.q.count; }
      compute_warps_sync<R>();
      uint32_t inc = lane < kWarps<R> ? P.ring[lane].count : 0u;
#pragma unroll
      for (int off = 1; off < kWarps<R>; off <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, inc, off);
        if (lane >= off) inc += t;
      }
      const uint32_t total = __shfl_sync(kFull, inc, kWarps<R> - 1);
      if constexpr (kFew<R> != 0) few = total <= (uint32_t)kWarps<R> * kFew<R>;
      const uint32_t each = few ? kFew<R> : 32u, e0 = (uint32_t)warp * each;
      take = total > e0 ? min(each, total - e0) : 0u;
      const uint32_t e = e0 + (uint32_t)(few ? lane / kQuad : lane);
      uint32_t j = 0, before = 0;
#pragma unroll
      for (int t = 0; t < kWarps<R> - 1; ++t) {
        const uint32_t upto = __shfl_sync(kFull, inc, t);
        if (e >= upto) { j = (uint32_t)t + 1u; before = upto; }
      }
      src = P.ring + j;
      p = src->head + e - before;
    }
    if constexpr (kFew<R> != 0) {
      if (few) {
        if (take)
          lepton_events_quads<R, WANT>(A, S.phase[run.s], run.s, src, p & (uint32_t)(kRing - 1), take, w.q.r->sums);
        continue;
      }
    }
    if (take) lepton_events<R, WANT>(A, S.phase[run.s], run.s, src, p & (uint32_t)(kRing - 1), take, w.q.r->sums);
  }
  compute_warps_sync<R>();  // every ring has been read
  w.q.count = 0;
  if (WANT) fold_run_sums(sums, run.s, w.q.r->sums);
}

// The block's tiles of one run of photons, or of a window's conversions, and the warp's events.
template <typename R, bool G, bool WANT>
__device__ __forceinline__ void run_photons(const StepArgs<R>& A, const StepScalars<R>& S, const StepPipe<R>& P,
                                            const TileRun& run, WarpState<R>& w) {
  RunSums<R> sums;
  ConversionState conv;
  for (bool more = true; more;) {
    if (run.s == 3) {
      more = false;
      if constexpr (sizeof(R) == 4) more = run_conversions(A, S, P, run, w, conv);
    } else if (!G && S.kind == QED_FIELD_PLANE_LP) {
      more = run_tiles<R, G, G ? kFieldAny : kFieldLP, 2, WANT>(A, S, P, run, w, sums);
    } else if (!G && S.kind == QED_FIELD_PLANE_CP) {
      more = run_tiles<R, G, G ? kFieldAny : kFieldCP, 2, WANT>(A, S, P, run, w, sums);
    } else {
      more = run_tiles<R, G, kFieldAny, 2, WANT>(A, S, P, run, w, sums);
    }
    if (w.stopped) w.q.count = 0;
    const uint32_t take = min(w.q.count, 32u);
    const bool few = take <= kFew<R>;
    if (take && !few)
      photon_events<R, WANT>(A, w.q.r, (w.q.head + (threadIdx.x & 31u)) & (uint32_t)(kRing - 1), take, w.q.r->sums);
    if constexpr (kFew<R> != 0) {
      if (take && few)
        photon_events_quads<R, WANT>(A, w.q.r, (w.q.head + (threadIdx.x & 31u) / kQuad) & (uint32_t)(kRing - 1), take,
                                     w.q.r->sums);
    }
    w.q.head += take;
    w.q.count -= take;
  }
  if (WANT && run.s == 2) fold_run_sums(sums, 2, w.q.r->sums);
}

template <typename R, bool G, bool WANT>
__device__ __forceinline__ void run_species(const StepArgs<R>& A, const StepScalars<R>& S, const StepPipe<R>& P,
                                            const TileRun& run, WarpState<R>& w) {
  if (run.s < 2) run_leptons<R, G, WANT>(A, S, P, run, w);
  else run_photons<R, G, WANT>(A, S, P, run, w);
}

// The call's packed grid, if it has one (after pdl_wait: pack_grid_kernel writes the flag).
template <typename R>
__device__ __forceinline__ const R* packed_cells(const FieldDev& f) {
  return sizeof(R) == 4 && f.cells && *f.packed ? static_cast<const R*>(f.cells) : nullptr;
}

// The step over one scenario, run by block `blk` of the `nblk` blocks given to it: block blk
// takes the scenario's tiles blk, blk + nblk, ... and writes ledger partial number blk.
// Warp roles: all warps but the last compute (warp w takes 32-particle chunk w of each tile); the last is
// the producer: its first lane issues the bulk copies of tile k into stage k % kStages once the
// compute warps have released that stage (mbarrier `empty`, one arrival per warp); compute warps
// wait only for their tile's data (mbarrier `full`), and for each other once per species, to share
// out the events left in their rings.
template <typename R, bool G, bool WANT>
__device__ __forceinline__ void step_body(const StepArgs<R>& a, uint32_t blk, uint32_t nblk, unsigned char* smem_raw) {
  TileBuf<R>* buf = reinterpret_cast<TileBuf<R>*>(smem_raw);
  EventRing<R>* ring = reinterpret_cast<EventRing<R>*>(buf + kStages);
  R* s_lnh = reinterpret_cast<R*>(ring + kWarps<R>);
  R* s_lnT = s_lnh + a.tab.n_eta;
  __shared__ __align__(8) uint64_t full[kStages];
  __shared__ __align__(8) uint64_t empty[kStages];
  __shared__ StepScalars<R> S;
  __shared__ int s_abort;
  __shared__ uint32_t s_work[2];

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // what does not depend on the step before: barriers, rate tables (fixed after their upload) and
  // the field scalars of this step
  if (threadIdx.x == kTile<R>) {
    for (int st = 0; st < kStages; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], kWarps<R>);
    }
    mbar_fence_init();
    s_abort = 0;
    s_work[0] = s_work[1] = 0;
  }
  for (int k = threadIdx.x; k < a.tab.n_eta; k += blockDim.x) s_lnh[k] = a.tab.ln_h[k];
  for (int k = threadIdx.x; k < a.tab.n_chi; k += blockDim.x) s_lnT[k] = a.tab.ln_T[k];
  if (threadIdx.x == 0) make_scalars<R>(a.field, a.t0 + (double)a.step * a.dt, a.win_x0, a.win_v, S);
  pdl_wait();
  const uint32_t n0 = a.sp[0].cnt->n, n1 = a.sp[1].cnt->n, n2 = a.sp[2].cnt->n;
  const uint32_t win_n = sizeof(R) == 4 && a.win_s >= 0 ? a.sp[2].cnt->win_n : 0u;
  const uint32_t T0 = (n0 + kTile<R> - 1) / kTile<R>, T1 = (n1 + kTile<R> - 1) / kTile<R>, T2 = (n2 - win_n + kTile<R> - 1) / kTile<R>;
  const uint32_t T3 = conversion_tiles(win_n, nblk);
  const uint32_t ttot = T0 + T1 + T2 + T3;
  if (threadIdx.x < 3) S.phase[threadIdx.x] = a.sp[threadIdx.x].cnt->phase;
  if (G && threadIdx.x == 0) S.cells = packed_cells<R>(a.field);
  if (threadIdx.x == kTile<R>)
    for (uint32_t k = 0; k < (uint32_t)kStages; ++k) issue_tile(a, buf, full, k, n0, n1, n2, win_n, blk, nblk);
  __syncthreads();
  pdl_launch();

  WarpState<R> w;
  if (warp == kWarps<R>) {
    // ---------------- producer
    if (lane == 0) {
      uint32_t k = kStages;
      for (;; ++k) {
        if (blk + k * nblk >= ttot || s_abort) break;
        const int st = (int)(k % kStages);
        if (!mbar_wait_bounded(&empty[st], ((k / kStages) - 1u) & 1u, kWaitLimit)) { s_abort = 1; break; }
        fence_proxy_async_smem();  // the compute warps' accesses to this stage come first
        issue_tile(a, buf, full, k, n0, n1, n2, win_n, blk, nblk);
      }
      if (s_abort) {
        // a wait gave up: report it, then wait (bounded) for the copies this block issued
        atomicOr(&a.sp[0].cnt->err, 1u << QED_ERR_TIMEOUT);
        const uint32_t first = k >= (uint32_t)kStages ? k - kStages : 0u;
        for (uint32_t q = first; q < k; ++q)
          if (blk + q * nblk < ttot) mbar_wait_bounded(&full[q % kStages], (q / kStages) & 1u, kWaitLimit);
      }
    }
  } else {
    // ---------------- compute warps
    w.q = EventQueue<R>{ring + warp, 0u, 0u};
    if (lane == 0) w.q.r->sums = EventSums<R>{};
    __syncwarp();
    const StepPipe<R> P{buf, full, empty, ring, s_lnh, s_lnT, &s_abort, blk, nblk};
    TileRun run;
    for (run.s = 0; run.s < 4; ++run.s) {
      run.g_lo = run.g_hi;
      run.g_hi += run.s == 0 ? T0 : (run.s == 1 ? T1 : (run.s == 2 ? T2 : T3));
      run.n = run.s == 0 ? n0 : (run.s == 1 ? n1 : (run.s == 2 ? n2 : win_n));
      run.base = run.s == 2 ? win_n : 0u;
      if (blk + w.k * nblk < run.g_hi) run_species<R, G, WANT>(a, S, P, run, w);  // (the same for every warp)
    }
    add_work(w.pushed_ph, w.tau_ph, s_work, lane);
  }
  __syncthreads();
  if (threadIdx.x == 0) flush_work(s_work, a.work);
  if (WANT) write_step_partial<R>(ring, a.ledger_part, blk);
}

// WANT: the step's ledger can be read (the last step of a run).
template <typename R, bool G, bool WANT>
__global__ void __launch_bounds__(kStepThreads<R>, sizeof(R) == 4 ? QED_STEP_MIN_BLOCKS : 256 / kTile<double>)
step_kernel(const __grid_constant__ StepArgs<R> a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  step_body<R, G, WANT>(a, blockIdx.x, gridDim.x, smem_raw);
}

// ----------------------------------------------------------------------------- multi-step
// Several steps per pass over the particles, state in registers.  Exact only across steps in
// which no particle has an event (children would have to join and be ordered at their step), so
// it runs in two passes: the probe advances every particle up to K steps without writing
// anything and records the first step (0-based, min over all particles) at which any particle
// would have an event; the commit then advances k <= that many steps and writes the state and
// the ledger of the last of them.  Both run lepton_advance / photon_advance, the per-step
// kernel's own arithmetic, so the particles end up with the bits the per-step kernel gives.
constexpr int kMaxFuse = 64;
constexpr int kFuseThreads = 256;

// State of one particle as the multi-step passes read it (the 7 SoA columns of any species;
// for photons u holds k).
template <typename R>
struct PState {
  R x, y, z, u0, u1, u2;
  double tau;  // stored form
};

// Particle g of the concatenated species (e-, e+, photons): its column pointers.
template <typename R>
struct PCols {
  R *x, *y, *z, *ux, *uy, *uz;
  double* tau;
  uint32_t i;
  int s;
};
template <typename R>
__device__ __forceinline__ PCols<R> cols_of(const StepArgs<R>& a, uint32_t g, uint32_t n0, uint32_t nl) {
  PCols<R> c;
  c.s = g < n0 ? 0 : (g < nl ? 1 : 2);
  c.i = c.s == 0 ? g : (c.s == 1 ? g - n0 : g - nl);
  // constant indices only (no dynamic indexing of the kernel parameters)
  c.x = c.s == 0 ? a.sp[0].x : (c.s == 1 ? a.sp[1].x : a.sp[2].x);
  c.y = c.s == 0 ? a.sp[0].y : (c.s == 1 ? a.sp[1].y : a.sp[2].y);
  c.z = c.s == 0 ? a.sp[0].z : (c.s == 1 ? a.sp[1].z : a.sp[2].z);
  c.ux = c.s == 0 ? a.sp[0].ux : (c.s == 1 ? a.sp[1].ux : a.sp[2].ux);
  c.uy = c.s == 0 ? a.sp[0].uy : (c.s == 1 ? a.sp[1].uy : a.sp[2].uy);
  c.uz = c.s == 0 ? a.sp[0].uz : (c.s == 1 ? a.sp[1].uz : a.sp[2].uz);
  c.tau = c.s == 0 ? a.sp[0].tau : (c.s == 1 ? a.sp[1].tau : a.sp[2].tau);
  return c;
}
template <typename R>
__device__ __forceinline__ PState<R> load_state(const PCols<R>& c) {
  return {c.x[c.i], c.y[c.i], c.z[c.i], c.ux[c.i], c.uy[c.i], c.uz[c.i], c.tau[c.i]};
}

// True when a particle drifting at vx (relative to the window) stays outside a plane-wave
// pulse's envelope through steps 0..K-1 of the stretch: the phase omega (t - x) is linear in the
// step along a straight path, so it suffices that the first and the last step are both on the
// same side of the envelope, with a margin far above the FP32 rounding of the per-step phase
// (the field is then exactly zero at every step, as field_at would find).
template <typename R>
__device__ __forceinline__ bool outside_pulse(const StepScalars<R>* S, int K, R x, R vx, R dt) {
  if (S[0].kind != QED_FIELD_PLANE_LP && S[0].kind != QED_FIELD_PLANE_CP) return false;
  if (!(S[0].len > (R)0)) return false;
  using N = Num<R>;
  const R ph0 = N::fma_(-S[0].omega, x, S[0].phi_ref);
  const R ph1 = N::fma_(-S[0].omega, N::fma_((R)(K - 1) * dt, vx, x), S[K - 1].phi_ref);
  const R m0 = (R)1e-2 + (R)1e-5 * fabs(ph0), m1 = (R)1e-2 + (R)1e-5 * fabs(ph1);
  return (ph0 < -m0 && ph1 < -m1) || (ph0 > S[0].len + m0 && ph1 > S[0].len + m1);
}

// One scenario's multi-step pass, run by block `blk` of the `nblk` blocks given to it (all
// threads of the block call it).
template <typename R, bool G, bool COMMIT, int FC>
__device__ __forceinline__ void fused_body(const StepArgs<R>& a, int K, uint32_t* first_event, uint32_t blk,
                                           uint32_t nblk, unsigned char* smem_raw) {
  R* s_lnh = reinterpret_cast<R*>(smem_raw);
  R* s_lnT = s_lnh + a.tab.n_eta;
  __shared__ StepScalars<R> S[kMaxFuse];
  for (int k = threadIdx.x; k < a.tab.n_eta; k += blockDim.x) s_lnh[k] = a.tab.ln_h[k];
  for (int k = threadIdx.x; k < a.tab.n_chi; k += blockDim.x) s_lnT[k] = a.tab.ln_T[k];
  if ((int)threadIdx.x < K)
    make_scalars<R>(a.field, a.t0 + (double)(a.step + threadIdx.x) * a.dt, a.win_x0, a.win_v, S[threadIdx.x]);
  __syncthreads();

  const uint32_t n0 = a.sp[0].cnt->n, n1 = a.sp[1].cnt->n, n2 = a.sp[2].cnt->n;
  const uint32_t nl = n0 + n1, tot = nl + n2;
  const uint32_t stride = nblk * blockDim.x;
  const R dt = a.dt_r, wv = a.win_v_r;
  using N = Num<R>;
  Acc<R> acc;
  bool bad = false;
  uint32_t g = blk * blockDim.x + threadIdx.x;
  // the next particle's state is loaded while the current one is stepped
  PCols<R> cc = cols_of(a, g < tot ? g : 0u, n0, nl);
  PState<R> cur;
  if (g < tot) cur = load_state(cc);
  for (; g < tot; g += stride) {
    const uint32_t gn = g + stride;
    const PCols<R> nc = cols_of(a, gn < tot ? gn : g, n0, nl);
    PState<R> nxt;
    if (gn < tot) nxt = load_state(nc);
    int limit = K;
    if (!COMMIT) {
      // no need to simulate past the earliest event found so far
      limit = min(K, (int)*reinterpret_cast<volatile uint32_t*>(first_event));
      if (limit == 0) break;
    }
    R x = cur.x, y = cur.y, z = cur.z;
    Tau<R> tau = Tau<R>::from_stored(cur.tau);
    int k = 0;
    if (cc.s < 2) {
      const bool pos = cc.s == 1;
      R u[3] = {cur.u0, cur.u1, cur.u2};
      const R q = pos ? (R)1 : (R)-1;
      // lepton_advance, step by step, with the drift velocity kept while u does not change
      // (where the field vanishes the push is the identity): the same operations on the same
      // values, so the same bits
      R gam, ig;
      N::root_inv_((R)1 + dot3<R>(u, u), gam, ig);
      R vx = N::fma_(u[0], ig, -wv), vy = u[1] * ig, vz = u[2] * ig;
      int oor = 0;
      if (outside_pulse<R>(S, limit, x, vx, dt)) {
        // no field at any step of the stretch: the drift only (nothing to probe)
        if (COMMIT)
          for (; k < limit; ++k) { x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z); }
        else
          k = limit;
      }
      for (; k < limit; ++k) {
        PushState<R, G, FC> ps;
        const int fc = push_at<R, G, FC>(S[k], x, y, z, q, dt, u, ps);
        if (fc == kNoField) {
          x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z);
          oor = 0;
          continue;  // no rate, no event
        }
        N::root_inv_((R)1 + dot3<R>(u, u), gam, ig);
        vx = N::fma_(u[0], ig, -wv); vy = u[1] * ig; vz = u[2] * ig;
        x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z);
        const R eta = eta_after<R, G, FC>(fc, u, gam, ps);
        oor = 0;
        if (eta > (R)0) {
          const R lam = (R)kRatePhoton * eta * ig * lookup_h<R>(a.tab, s_lnh, eta, oor);
          tau.sub(lam * dt);
        }
        if (a.emit && tau.used_up()) break;
      }
      if (!COMMIT) {
        if (k < limit) atomicMin(first_event, (uint32_t)k);
      } else {
        bad |= k < K;  // the probe ruled this out; the arithmetic is the same
        cc.x[cc.i] = x; cc.y[cc.i] = y; cc.z[cc.i] = z;
        cc.ux[cc.i] = u[0]; cc.uy[cc.i] = u[1]; cc.uz[cc.i] = u[2];
        tau.store(cc.tau + cc.i);
        acc.e[pos ? 1 : 0].add(gam);
        acc.n[pos ? 1 : 0]++;
        if (oor > 0) acc.oor_eta++;
      }
    } else if (!tau.dead()) {  // converted photons stay as holes until compaction
      const R kv[3] = {cur.u0, cur.u1, cur.u2};
      // photon_advance, step by step: k does not change, so neither do eps, 1/eps and the drift
      R eps, ie;
      N::root_inv_(dot3<R>(kv, kv), eps, ie);
      const R vx = N::fma_(kv[0], ie, -wv), vy = kv[1] * ie, vz = kv[2] * ie;
      int oor = 0;
      if (outside_pulse<R>(S, limit, x, vx, dt)) {
        if (COMMIT)
          for (; k < limit; ++k) { x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z); }
        else
          k = limit;
      }
      for (; k < limit; ++k) {
        int fc;
        const R chi = chi_at<R, G, FC>(S[k], x, y, z, kv, eps, fc);
        oor = 0;
        if (fc != kNoField) {
          if (chi > (R)0) {
            const R lam = (R)kAlpha * chi * ie * lookup_T<R>(a.tab, s_lnT, chi, oor);
            tau.sub(lam * dt);
          }
        }
        x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z);
        if (fc != kNoField && a.pairs && tau.used_up()) break;
      }
      if (!COMMIT) {
        if (k < limit) atomicMin(first_event, (uint32_t)k);
      } else {
        bad |= k < K;
        cc.x[cc.i] = x; cc.y[cc.i] = y; cc.z[cc.i] = z;
        tau.store(cc.tau + cc.i);
        acc.e[2].add(eps);
        acc.n[2]++;
        acc.pushed_ph++;
        if (oor > 0) acc.oor_chi++;
      }
    }
    cc = nc;
    cur = nxt;
  }
  if (COMMIT) {
    if (bad) atomicOr(&a.sp[0].cnt->err, 1u << QED_ERR_NUMERIC);
    __shared__ uint32_t s_pushed;
    if (threadIdx.x == 0) s_pushed = 0;
    __syncthreads();
    const uint32_t pushed = __reduce_add_sync(kFull, acc.pushed_ph);
    if ((threadIdx.x & 31) == 0 && pushed) atomicAdd(&s_pushed, pushed);
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned long long p = (unsigned long long)s_pushed * (unsigned long long)K;
      if (p) { atomicAdd(&a.work[1], p); atomicAdd(&a.work[4], p); }
      if (blk == 0) {
        const unsigned long long l = (unsigned long long)nl * (unsigned long long)K;
        atomicAdd(&a.work[0], l);
        atomicAdd(&a.work[3], l);
      }
    }
    if (a.want) write_ledger_partial<R, kFuseThreads / 32>(acc, a.ledger_part, blk);
  }
}

template <typename R, bool G, bool COMMIT>
__global__ void __launch_bounds__(kFuseThreads) fused_kernel(const StepArgs<R> a, int K, uint32_t* first_event) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // the field class of the run (every step of a stretch has the same field)
  if (a.field.kind == QED_FIELD_PLANE_LP)
    fused_body<R, G, COMMIT, kFieldLP>(a, K, first_event, blockIdx.x, gridDim.x, smem_raw);
  else if (a.field.kind == QED_FIELD_PLANE_CP)
    fused_body<R, G, COMMIT, kFieldCP>(a, K, first_event, blockIdx.x, gridDim.x, smem_raw);
  else
    fused_body<R, G, COMMIT, kFieldAny>(a, K, first_event, blockIdx.x, gridDim.x, smem_raw);
}

__global__ void set_u32_kernel(uint32_t* p, uint32_t v) { *p = v; }

// Failure-detection self-test of the bounded mbarrier wait that every pipeline wait uses: a
// barrier whose phase completes is waited for successfully; a barrier that nothing ever arrives
// at gives up after `polls` polls instead of hanging.  bits: 1 = completed wait returned true,
// 2 = unsatisfiable wait timed out.
__global__ void selftest_wait_kernel(uint32_t polls, uint32_t* bits) {
  __shared__ __align__(8) uint64_t done_bar, never_bar;
  if (threadIdx.x == 0) {
    mbar_init(&done_bar, 1);
    mbar_init(&never_bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t out = 0;
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&done_bar)) : "memory");
    if (mbar_wait_bounded(&done_bar, 0u, polls)) out |= 1u;
    if (!mbar_wait_bounded(&never_bar, 0u, polls)) out |= 2u;
    *bits = out;
  }
}


// ----------------------------------------------------------------------------- packed grids
// Packs a cloud-in-cell grid by cells for one call (the caller updates its grid between calls).  A
// gather straight from the grid is 48 scattered 4-byte reads per particle, and the L1's one look-up
// per lane and read bounds it: on GB300 60 us for 4e5 particles on a grid of 48^3 nodes; packed it is
// 6 reads of 32 bytes, 20 us.  Packing writes 192 bytes per cell, so it pays from about a third of a
// particle-step per cell on (48^3: break-even at 3e4 particles, 64^3: 1e5); with fewer it is skipped.  (The FP64 path is
// bound by the FP64 pipe and gains nothing: 375 us a step against 391 with the packing.)  One thread per component and cell; blocks
// stand for 256 cells of one z layer of one component.
__global__ void __launch_bounds__(256) pack_grid_kernel(const StepArgs<float> a, uint64_t steps) {
  pdl_wait();
  pdl_launch();
  const FieldDev& f = a.field;
  const uint64_t cells = grid_cells(f.n);
  const uint64_t particles = (uint64_t)a.sp[0].cnt->n + a.sp[1].cnt->n + a.sp[2].cnt->n;
  const bool on = packing_pays(particles, steps, cells);
  if (blockIdx.x + blockIdx.y + blockIdx.z + threadIdx.x == 0) *f.packed = on ? 1u : 0u;
  if (!on) return;
  const int nx = f.n[0], ny = f.n[1], nz = f.n[2];
  const uint32_t q = blockIdx.x * 256u + threadIdx.x, layer = (uint32_t)(nx + 1) * (uint32_t)(ny + 1);
  if (q >= layer) return;
  const int y = (int)(q / (uint32_t)(nx + 1)) - 1, x = (int)(q % (uint32_t)(nx + 1)) - 1;
  const size_t N = (size_t)nx * ny * nz;
  const float* grid = static_cast<const float*>(f.grid) + blockIdx.z * N;
  for (int z = (int)blockIdx.y - 1; z < nz; z += (int)gridDim.y) {
    float v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = x + (t & 1), j = y + (t >> 1 & 1), k = z + (t >> 2);
      const bool in = i >= 0 && i < nx && j >= 0 && j < ny && k >= 0 && k < nz;
      v[t] = in ? grid[((size_t)k * ny + j) * nx + i] : 0.0f;
    }
    float4* out = reinterpret_cast<float4*>(static_cast<float*>(f.cells) +
                                            8 * (blockIdx.z * cells + (uint64_t)(z + 1) * layer + q));
    out[0] = make_float4(v[0], v[1], v[2], v[3]);
    out[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// ----------------------------------------------------------------------------- finalisation
// Block-wide exclusive scan of one value per thread (blockDim.x <= 1024, multiple of 32).
__device__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t s_w[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  uint32_t inc = v;
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t t = __shfl_up_sync(kFull, inc, off);
    if (lane >= off) inc += t;
  }
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nwarp ? s_w[lane] : 0u;
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, w, off);
      if (lane >= off) w += t;
    }
    s_w[lane] = w;  // inclusive prefix over warps
  }
  __syncthreads();
  const uint32_t warp_base = warp > 0 ? s_w[warp - 1] : 0u;
  if (total) *total = s_w[nwarp - 1];
  __syncthreads();
  return warp_base + inc - v;
}

// Sum of the entries [lo, hi) of a group-aligned array v (lo a multiple of 32 entries, hi - lo <= 32;
// storage is padded to whole groups), or of their popcounts: eight independent 16-byte loads.
template <bool POP>
__device__ __forceinline__ uint32_t group_sum(const uint32_t* v, uint32_t lo, uint32_t hi) {
  const uint4* p = reinterpret_cast<const uint4*>(v + lo);
  uint32_t s = 0;
  const uint32_t m = hi - lo;
#pragma unroll
  for (uint32_t q = 0; q < 8; ++q) {
    if (4 * q < m) {
      const uint4 t = p[q];
      s += POP ? (uint32_t)__popc(t.x) : t.x;
      if (4 * q + 1 < m) s += POP ? (uint32_t)__popc(t.y) : t.y;
      if (4 * q + 2 < m) s += POP ? (uint32_t)__popc(t.z) : t.z;
      if (4 * q + 3 < m) s += POP ? (uint32_t)__popc(t.w) : t.w;
    }
  }
  return s;
}

// Parents of children before parent p inside its coarse group.
template <typename R>
__device__ __forceinline__ uint32_t rank_in_coarse(const SpeciesDev<R>& sp, uint32_t phase, uint32_t p) {
  const uint32_t w = p >> 5, f = w >> kFineShift;
  const uint32_t f0 = f & ~((1u << kCoarseShift) - 1u), w0 = w & ~((1u << kFineShift) - 1u);
  return group_sum<false>(sp.fine + phase * event_fines(sp.cap), f0, f) + group_sum<true>(sp.evmask, w0, w) +
         (uint32_t)__popc(sp.evmask[w] & ((1u << (p & 31u)) - 1u));
}

// What the step leaves to merge, from the counters and the parents' totals (the same on every
// thread that computes it; the error bits are set by the one with `report`).
template <typename R>
__device__ __forceinline__ FinalizePlan make_plan(const StepArgs<R>& a, uint32_t from_electrons, bool report) {
  FinalizePlan P;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const SpeciesDev<R>& app = a.sp[d];  // append region owner
    const SpeciesDev<R>& dst = (d == 2 && a.drain) ? a.sp[3] : a.sp[d];
    P.n_old[d] = dst.cnt->n;
    P.next_id_old[d] = dst.cnt->next_id;
    P.phase[d] = app.cnt->phase;
    uint32_t m = app.cnt->n_app;
    // children beyond the append region or the destination's room: drop the step's children
    if (m > app.acap || (uint64_t)P.n_old[d] + m > dst.cap) {
      if (report) atomicOr(&dst.cnt->err, 1u << QED_ERR_CAPACITY);
      m = 0;
    }
    P.m[d] = m;
  }
  P.from_electrons = from_electrons;
  P.ticket = 0;
  return P;
}

// Child c (in destination order e-, e+, photons) of the step planned in P: its rank among the
// destination's new particles is its parent's rank (a counting sort on the dense parent index),
// which fixes its slot and its id.  coarse_before(s, c): children of species s's parents in the
// coarse groups before c.
template <typename R, typename F>
__device__ __forceinline__ void place_child(const StepArgs<R>& a, const FinalizePlan& P, uint32_t c, F coarse_before) {
  const uint32_t m0 = P.m[0], m1 = P.m[1];
  const int d = c < m0 ? 0 : (c < m0 + m1 ? 1 : 2);
  const uint32_t j = c - (d == 0 ? 0u : (d == 1 ? m0 : m0 + m1));
  // constant indices only (no dynamic indexing of the kernel parameters)
  const SpeciesDev<R>& app = d == 0 ? a.sp[0] : (d == 1 ? a.sp[1] : a.sp[2]);
  const SpeciesDev<R>& dst = (d == 2 && a.drain) ? a.sp[3] : app;
  const uint32_t par = app.aparent[j];
  const R x = app.ax[j], y = app.ay[j], z = app.az[j], ux = app.aux[j], uy = app.auy[j], uz = app.auz[j];
  const double tau = app.atau[j];
  const int ps = d < 2 ? 2 : (int)(par >> 31);
  const uint32_t p = d < 2 ? par : par & 0x7fffffffu;
  const SpeciesDev<R>& psp = ps == 0 ? a.sp[0] : (ps == 1 ? a.sp[1] : a.sp[2]);
  const uint32_t ph = ps == 0 ? P.phase[0] : (ps == 1 ? P.phase[1] : P.phase[2]);
  const uint32_t rank = coarse_before(ps, p >> (5 + kFineShift + kCoarseShift)) + rank_in_coarse(psp, ph, p) +
                        (ps == 1 ? P.from_electrons : 0u);
  const uint32_t m = d == 0 ? m0 : (d == 1 ? m1 : P.m[2]);
  if (rank >= m) { atomicOr(&dst.cnt->err, 1u << QED_ERR_NUMERIC); return; }
  const uint32_t o = (d == 0 ? P.n_old[0] : (d == 1 ? P.n_old[1] : P.n_old[2])) + rank;
  dst.x[o] = x; dst.y[o] = y; dst.z[o] = z;
  dst.ux[o] = ux; dst.uy[o] = uy; dst.uz[o] = uz;
  dst.tau[o] = tau;
  dst.id[o] = (d == 0 ? P.next_id_old[0] : (d == 1 ? P.next_id_old[1] : P.next_id_old[2])) + rank;
  if (dst.w) dst.w[o] = app.aw ? app.aw[j] : (R)1;
}

// Clears, share `i` of `n`, the event counts that the step before left in the buffer this step
// did not use.
template <typename R>
__device__ __forceinline__ void clear_other_counts(const StepArgs<R>& a, const FinalizePlan& P, uint32_t i, uint32_t n) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const SpeciesDev<R>& sp = a.sp[s];
    const uint32_t o = P.phase[s] ^ 1u, ext = sp.cnt->ext[o];
    for (uint32_t k = i; k < ext; k += n) sp.fine[o * event_fines(sp.cap) + k] = 0u;
    for (uint32_t k = i; k < (ext + 31u) >> kCoarseShift; k += n) sp.coarse[o * event_coarses(sp.cap) + k] = 0u;
  }
}

__device__ __forceinline__ uint32_t fines_of(uint32_t n) { return (((n + 31u) >> 5) + 31u) >> kFineShift; }
__device__ __forceinline__ uint32_t coarses_of(uint32_t n) { return (fines_of(n) + 31u) >> kCoarseShift; }

// The counters after the merge and the scenario's work counters (one thread).  n: the step's parents.
template <typename R>
__device__ __forceinline__ void finish_counters(const StepArgs<R>& a, const FinalizePlan& P, const uint32_t n[3]) {
  const uint32_t emitted = a.sp[2].cnt->n_app, pairs = a.sp[0].cnt->n_app;
  atomicAdd(&a.work[0], (unsigned long long)n[0] + n[1]);
  if (emitted + pairs) atomicAdd(&a.work[2], (unsigned long long)emitted + 2ull * pairs);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const SpeciesDev<R>& sp = a.sp[d];
    sp.cnt->ext[P.phase[d] ^ 1u] = 0u;
    sp.cnt->ext[P.phase[d]] = fines_of(n[d]);
    sp.cnt->phase = P.phase[d] ^ 1u;
    sp.cnt->n_app = 0u;
    const SpeciesDev<R>& dst = (d == 2 && a.drain) ? a.sp[3] : sp;
    dst.cnt->n = P.n_old[d] + P.m[d];
    dst.cnt->next_id = P.next_id_old[d] + P.m[d];
  }
}

// Fixed-order reduction of the per-block ledger partials, one warp per field (lane l sums
// partials l, l+32, ... in order, then a fixed shuffle tree): deterministic for a fixed grid.
template <typename R>
__device__ __forceinline__ void reduce_ledger(const StepArgs<R>& a, int nparts) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = warp; k < kLedgerN; k += blockDim.x >> 5) {
    double t = 0.0;
#pragma unroll 4
    for (int p = lane; p < nparts; p += 32) t += a.ledger_part[(size_t)p * kLedgerN + k];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(kFull, t, off);
    if (lane == 0) a.ledger[k] = t;
  }
}

// The merge of one step.  Every block computes the plan for itself: the counters give the totals,
// and warp s scans species s's coarse event counts (one per 32768 parents) into shared memory; a
// child's rank is then three sums of at most 32 entries each, by its own thread.
// Latency-bound: it moves a few MB at most, on every step of every run.  The form before it, a
// one-block plan, a prefix over the event masks and a scatter, were three dependent launches of
// 12, 5 and 8 us (GB300, 1e3 to 3e5 electrons); with this one, and the ledger's sums kept only
// where they can be read, a step of 1e3 electrons went from 39.8 to 18.4 us and the 4000-step
// collision of 1e3 electrons from 109 to 50 ms.
constexpr int kCoarseMax = 1024;  // prefixes per species in shared memory (larger species: groups of counts)
constexpr int kFinalThreads = 256;
template <typename R>
__global__ void __launch_bounds__(kFinalThreads) finalize_kernel(const StepArgs<R> a, int nparts) {
  __shared__ uint32_t s_pre[3][kCoarseMax];
  __shared__ uint32_t s_from;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();
  pdl_launch();
  const uint32_t n[3] = {a.sp[0].cnt->n, a.sp[1].cnt->n, a.sp[2].cnt->n};
  const bool any_ph = a.sp[2].cnt->n_app != 0u, any_pair = a.sp[0].cnt->n_app != 0u;
  uint32_t per[3];  // coarse counts per prefix entry
#pragma unroll
  for (int s = 0; s < 3; ++s) per[s] = (coarses_of(n[s]) + kCoarseMax - 1) / kCoarseMax;
  if (warp < 3) {
    const SpeciesDev<R>& sp = warp == 0 ? a.sp[0] : (warp == 1 ? a.sp[1] : a.sp[2]);
    const uint32_t* co = sp.coarse + sp.cnt->phase * event_coarses(sp.cap);
    const uint32_t nc = (warp < 2 ? any_ph : any_pair) ? coarses_of(warp == 0 ? n[0] : (warp == 1 ? n[1] : n[2])) : 0u;
    const uint32_t g = warp == 0 ? per[0] : (warp == 1 ? per[1] : per[2]);
    uint32_t run = 0;
#pragma unroll 4
    for (uint32_t e0 = 0; e0 * g < nc; e0 += 32) {
      uint32_t v = 0;
      for (uint32_t k = (e0 + lane) * g; k < min(nc, (e0 + lane + 1) * g); ++k) v += co[k];
      uint32_t inc = v;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, inc, off);
        if (lane >= off) inc += t;
      }
      if (e0 + lane < (uint32_t)kCoarseMax) s_pre[warp][e0 + lane] = run + inc - v;
      run += __shfl_sync(kFull, inc, 31);
    }
    if (warp == 0 && lane == 0) s_from = run;
  }
  __syncthreads();
  const FinalizePlan P = make_plan(a, s_from, blockIdx.x == 0 && threadIdx.x == 0);
  const uint32_t tot = P.m[0] + P.m[1] + P.m[2];
  const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t c = first; c < tot; c += stride)
    place_child<R>(a, P, c, [&](int s, uint32_t cg) {
      const uint32_t g = s == 0 ? per[0] : (s == 1 ? per[1] : per[2]);
      uint32_t r = s_pre[s][cg / g];
      if (g > 1) {
        const SpeciesDev<R>& sp = s == 0 ? a.sp[0] : (s == 1 ? a.sp[1] : a.sp[2]);
        const uint32_t* co = sp.coarse + (s == 0 ? P.phase[0] : (s == 1 ? P.phase[1] : P.phase[2])) * event_coarses(sp.cap);
        for (uint32_t k = cg / g * g; k < cg; ++k) r += co[k];
      }
      return r;
    });
  clear_other_counts(a, P, first, stride);
  if (a.want && blockIdx.x == gridDim.x - 1) {
    // (blocks without a tile have nothing to add)
    uint32_t tiles = 0;
    for (int s = 0; s < 3; ++s) tiles += (n[s] + kTile<R> - 1) / kTile<R>;
    reduce_ledger(a, (int)min((uint32_t)nparts, tiles));
  }
  // the last block to get here sets the counters: by then every block has read them
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&a.plan->ticket, 1u) == gridDim.x - 1) {
      a.plan->ticket = 0u;
      finish_counters(a, P, n);
      if (a.counter) {  // the allocation-free step: the caller's photon count, next id and error bits
        a.counter[0] = a.sp[3].cnt->n;
        a.counter[1] = a.sp[3].cnt->next_id;
        uint32_t err = 0;
        for (int k = 0; k < 4; ++k) err |= *(volatile uint32_t*)&a.sp[k].cnt->err;
        a.counter[2] |= err;
      }
    }
  }
}

// ----------------------------------------------------------------------------- photon windows
// Photons depend on no other particle, and the only thing a step does with one is to convert it.  So
// a run takes its photons several steps at a time: at the start of a window of K steps this kernel
// advances every photon held (but for the last n mod 1024) by K steps in registers, with
// photon_advance's own operations, and stops a photon at the step at which its optical depth runs
// out; the K per-step kernels that follow push the leptons and the photons made since, and take the
// conversions found for their step (run_conversions).  Particles, ids and order are those of the
// per-step path: a conversion is taken at its step, and the merge ranks it by the photon's index.
//
// A step whose ledger can be read (the last of a run) belongs to no window: its sums are taken by
// the per-step kernel over every photon, in its order.
//
// What it saves: the per-step kernel streams 44 B per photon and step and is issue-bound on the
// bookkeeping around the field evaluation; here a photon is loaded and stored (52 B) once per K.
// Issue-bound.  What it does about that:
//  - What a photon keeps over the window (energy, drift velocity, the invariant's factor) is computed
//    once; the plane wave's step-dependent phases and the T table's cells are read as pairs.
//  - A photon whose chi stays below the table's start whatever the phase (chi_bound) has rate zero:
//    it only drifts, as does one that stays outside the pulse.  Photon energies mix within every
//    chunk, so the others (about half) go to a ring per warp and are stepped 32 at a time.
//  - In a uniform field chi and the rate are constants of the photon.
// Measured on GB300 (16 steps): 2e7 cascade photons 580 us, 36 us a step against 189 us on the
// per-step kernel; 6e6 photons in a pulse 273 us, 17 us a step.  Whole runs: the collision of 1e6
// electrons 367 -> 139 ms, the cascade's 50 steps 10.2 -> 4.2 ms.
enum WindowClass { kWinLP = 0, kWinCP = 1, kWinRotating = 2, kWinUniform = 3, kWinGrid = 4 };

struct WinRing {
  uint32_t i[kRing];
  float v[8][kRing];  // x, y, z, k, optical depth (hi, lo)
};
struct WinShared {
  StepScalars<float> S[kWinMax];
  float2 pair[kWinMax];  // per step: plane waves (phi_ref, phi_ref_mod); rotating E (E_x, E_y)
  uint32_t pushed;
  WinRing ring[kFuseThreads / 32];
};

// T(chi) as lookup_T, from cells (ln T_i, ln T_i+1)
__device__ __forceinline__ float lookup_T_cells(const TabDev<float>& T, const float2* cell, float chi, int& oor) {
  oor = 0;
  if (!(chi >= T.chi_min)) return 0.0f;
  if (chi > T.chi_max) { oor = 1; return T_above<float>(T, chi); }
  int i, o; float w;
  grid_pos(Num<float>::log_tab_(chi), T.ln_chi_min, T.inv_d_chi, T.n_chi, i, w, o);
  const float2 c = cell[i];
  return Num<float>::exp_tab_(Num<float>::fma_(w, c.y, (1.0f - w) * c.x));
}

// One photon of a window with its constants.
template <int WC>
struct WinPhoton {
  float x, y, z, k[3], eps, ie, vx, vy, vz, hd;
  Tau<float> tau;
  __device__ __forceinline__ void constants(float wv) {
    using N = Num<float>;
    N::root_inv_(dot3<float>(k, k), eps, ie);
    vx = N::fma_(k[0], ie, -wv); vy = k[1] * ie; vz = k[2] * ie;
    if (WC == kWinLP || WC == kWinCP) {  // chi = hd |E| (chi_plane)
      const float d = k[0] > 0.0f ? N::div_(N::fma_(k[1], k[1], k[2] * k[2]), eps + k[0]) : eps - k[0];
      hd = 0.5f * d;
    }
  }
  __device__ __forceinline__ void drift(float dt) {
    using N = Num<float>;
    x = N::fma_(dt, vx, x); y = N::fma_(dt, vy, y); z = N::fma_(dt, vz, z);
  }
  // a bound of chi over every phase, with room for the rounding of the phase functions
  __device__ __forceinline__ float chi_bound(float E0) const {
    return (WC == kWinRotating ? 0.5f * eps : hd) * fabsf(E0) * 1.0001f;
  }
};

// Steps one photon per lane up to K steps; the step it converted at, or -1.
template <bool G, int WC>
__device__ __forceinline__ int window_steps(const StepArgs<float>& a, const WinShared& sh, const float2* cell, int K,
                                            WinPhoton<WC>& p, float& chi) {
  using N = Num<float>;
  const float dt = a.dt_r;
  const StepScalars<float>& S0 = sh.S[0];
  const float om = S0.omega, len = S0.len, inv_len = S0.inv_len, E0 = S0.E0;
  int k = 0;
  for (; k < K; ++k) {
    chi = 0.0f;
    int oor;
    if (WC == kWinLP || WC == kWinCP) {
      // plane_at and chi_plane
      const float2 ref = sh.pair[k];
      float env = 1.0f;
      bool in = true;
      if (len > 0.0f) {
        const float phi = N::fma_(-om, p.x, ref.x);
        in = phi > 0.0f && phi < len;
        const float sn = N::sin_env_((float)kPi * (phi * inv_len));
        env = sn * sn;
      }
      const float amp0 = E0 * env;
      float amp;
      if (WC == kWinLP) {
        float sn, cs;
        N::carrier_(N::fma_(-om, p.x, ref.y), &sn, &cs);
        amp = fabsf(amp0 * cs);
      } else {
        amp = amp0;
      }
      if (in) chi = p.hd * amp;
    } else if (WC == kWinRotating) {
      // chi_of with E = (E_x, E_y, 0), B = 0: the terms left out are exact zeros
      const float2 E = sh.pair[k];
      const float e0 = -(p.k[2] * E.y), e1 = p.k[2] * E.x, e2 = N::fma_(p.k[0], E.y, -(p.k[1] * E.x));
      const float c2 = N::fma_(e0, e0, N::fma_(e1, e1, e2 * e2));
      if (c2 > 0.0f) chi = 0.5f * N::sqrt_pos_(c2);
    } else {
      int fc;
      chi = chi_at<float, G, kFieldAny>(sh.S[k], p.x, p.y, p.z, p.k, p.eps, fc);
    }
    if (chi > 0.0f) {
      const float lam = (float)kAlpha * chi * p.ie * lookup_T_cells(a.tab, cell, chi, oor);
      p.tau.sub(lam * dt);
    }
    p.drift(dt);
    if (a.pairs && p.tau.used_up()) return k;
  }
  return -1;
}

// Writes one stepped photon back; a converted one waits for its step (run_conversions).
template <int WC>
__device__ __forceinline__ void window_store(const StepArgs<float>& a, uint32_t i, const WinPhoton<WC>& p,
                                             const Tau<float>& tau0, int conv, float chi, int K, uint32_t& pushed) {
  const SpeciesDev<float>& sp = a.sp[2];
  sp.x[i] = p.x; sp.y[i] = p.y; sp.z[i] = p.z;
  pushed += conv >= 0 ? (uint32_t)conv + 1u : (uint32_t)K;
  if (conv >= 0) {
    Tau<float>::window(conv, chi).store(sp.tau + i);
    atomicOr(&sp.cmask[i >> 5], 1u << (i & 31u));
    atomicOr(&sp.wflag[i >> 10], 1u << conv);
  } else if (__float_as_int(p.tau.hi) != __float_as_int(tau0.hi) || __float_as_int(p.tau.lo) != __float_as_int(tau0.lo)) {
    p.tau.store(sp.tau + i);
  }
}

// Takes `take` (<= 32) photons from the warp's ring, one per lane.
template <bool G, int WC>
__device__ __forceinline__ void window_batch(const StepArgs<float>& a, const WinShared& sh, const WinRing& r,
                                             const float2* cell, uint32_t head, uint32_t take, int K, uint32_t& pushed) {
  const int lane = threadIdx.x & 31;
  if ((uint32_t)lane < take) {
    const uint32_t q = (head + (uint32_t)lane) & (uint32_t)(kRing - 1);
    WinPhoton<WC> p;
    p.x = r.v[0][q]; p.y = r.v[1][q]; p.z = r.v[2][q];
    p.k[0] = r.v[3][q]; p.k[1] = r.v[4][q]; p.k[2] = r.v[5][q];
    const Tau<float> tau0{r.v[6][q], r.v[7][q]};
    p.tau = tau0;
    p.constants(a.win_v_r);
    float chi;
    const int conv = window_steps<G, WC>(a, sh, cell, K, p, chi);
    window_store<WC>(a, r.i[q], p, tau0, conv, chi, K, pushed);
  }
  __syncwarp();  // the ring slots read above may be refilled
}

// A warp's chunks chunk, chunk + nw, ... below `chunks`; the ring is empty after it.  Returns the
// lane's pushes.
template <bool G, int WC>
__device__ __forceinline__ uint32_t window_chunks(const StepArgs<float>& a, int K, uint32_t chunk, uint32_t chunks,
                                                  uint32_t nw, WinShared& sh, const float2* cell) {
  const SpeciesDev<float>& sp = a.sp[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float dt = a.dt_r;
  WinRing& ring = sh.ring[warp];
  uint32_t head = 0, count = 0;  // warp-uniform
  uint32_t pushed = 0;
  // the next chunk's state is loaded while the current one is stepped
  PState<float> nxt{};
  auto load = [&](uint32_t c) {
    const uint32_t i = c * 32u + (uint32_t)lane;
    nxt = {sp.x[i], sp.y[i], sp.z[i], sp.ux[i], sp.uy[i], sp.uz[i], sp.tau[i]};
  };
  if (chunk < chunks) load(chunk);
  for (; chunk < chunks; chunk += nw) {
    const PState<float> cur = nxt;
    if (chunk + nw < chunks) load(chunk + nw);
    const uint32_t i = chunk * 32u + (uint32_t)lane;
    if (lane == 0) sp.cmask[chunk] = 0u;
    __syncwarp();
    WinPhoton<WC> p;
    p.x = cur.x; p.y = cur.y; p.z = cur.z;
    p.k[0] = cur.u0; p.k[1] = cur.u1; p.k[2] = cur.u2;
    const Tau<float> tau0 = Tau<float>::from_stored(cur.tau);
    p.tau = tau0;
    const bool alive = !tau0.dead();
    bool later = false;
    if (alive) {
      p.constants(a.win_v_r);
      float chi = 0.0f;
      int oor, conv = -1;
      if (WC == kWinGrid) {
        conv = window_steps<G, WC>(a, sh, cell, K, p, chi);
      } else if (WC == kWinUniform) {
        float amp = 0.0f, E[3], B[3];
        const int fc = field_at<float, false>(sh.S[0], p.x, p.y, p.z, E, B, amp);
        chi = chi_for<float>(fc, p.k, p.eps, E, B, amp);
        float d = 0.0f;
        if (chi > 0.0f) {
          const float lam = (float)kAlpha * chi * p.ie * lookup_T_cells(a.tab, cell, chi, oor);
          d = lam * dt;
        }
        for (int k = 0; k < K; ++k) {
          if (chi > 0.0f) p.tau.sub(d);
          p.drift(dt);
          if (a.pairs && p.tau.used_up()) { conv = k; break; }
        }
      } else {
        // (an optical depth that is used up already converts at the next step, field or not)
        const bool used = tau0.used_up();
        const bool none = !used && (WC == kWinLP || WC == kWinCP) && outside_pulse<float>(sh.S, K, p.x, p.vx, dt);
        const bool soft = !used && p.chi_bound(sh.S[0].E0) < a.tab.chi_min;
        if (soft && !none) p.tau.sub(0.0f);  // (the rate is zero: the value stays)
        later = !none && !soft;
        if (!later)
          for (int k = 0; k < K; ++k) p.drift(dt);
      }
      if (!later) window_store<WC>(a, i, p, tau0, conv, chi, K, pushed);
    }
    if (WC != kWinGrid && WC != kWinUniform) {
      const unsigned m = __ballot_sync(kFull, later);
      if (later) {
        const uint32_t q = (head + count + (uint32_t)__popc(m & ((1u << lane) - 1u))) & (uint32_t)(kRing - 1);
        ring.i[q] = i;
        ring.v[0][q] = cur.x; ring.v[1][q] = cur.y; ring.v[2][q] = cur.z;
        ring.v[3][q] = cur.u0; ring.v[4][q] = cur.u1; ring.v[5][q] = cur.u2;
        ring.v[6][q] = tau0.hi; ring.v[7][q] = tau0.lo;
      }
      count += (uint32_t)__popc(m);
      __syncwarp();
      const bool end = chunk + nw >= chunks;
      while (count >= 32u || (end && count > 0u)) {
        const uint32_t take = min(count, 32u);
        window_batch<G, WC>(a, sh, ring, cell, head, take, K, pushed);
        head = (head + take) & (uint32_t)(kRing - 1);
        count -= take;
      }
    }
  }
  return pushed;
}

template <bool G>
__device__ __forceinline__ uint32_t window_photons(const StepArgs<float>& a, int K, uint32_t chunk, uint32_t chunks,
                                                   uint32_t nw, WinShared& sh, const float2* cell) {
  switch (a.field.kind) {
    case QED_FIELD_PLANE_LP: return window_chunks<G, kWinLP>(a, K, chunk, chunks, nw, sh, cell);
    case QED_FIELD_PLANE_CP: return window_chunks<G, kWinCP>(a, K, chunk, chunks, nw, sh, cell);
    case QED_FIELD_ROTATING_E: return window_chunks<G, kWinRotating>(a, K, chunk, chunks, nw, sh, cell);
    case QED_FIELD_UNIFORM: return window_chunks<G, kWinUniform>(a, K, chunk, chunks, nw, sh, cell);
    default:
      if constexpr (G) return window_chunks<G, kWinGrid>(a, K, chunk, chunks, nw, sh, cell);
      return 0;
  }
}

__device__ __forceinline__ void load_cells(const TabDev<float>& tab, float2* cell) {
  for (int k = threadIdx.x; k + 1 < tab.n_chi; k += blockDim.x) cell[k] = make_float2(tab.ln_T[k], tab.ln_T[k + 1]);
}
__device__ __forceinline__ float2 window_pair(int kind, const StepScalars<float>& S) {
  return kind == QED_FIELD_ROTATING_E ? make_float2(S.E[0], S.E[1]) : make_float2(S.phi_ref, S.phi_ref_mod);
}
__device__ __forceinline__ void add_window_work(const StepArgs<float>& a, uint32_t pushed) {
  if (!pushed) return;
  atomicAdd(&a.work[1], (unsigned long long)pushed);
  atomicAdd(&a.work[4], (unsigned long long)pushed);
}

// Shared memory: WinShared, then the T table's cells (n_chi - 1 of them).
inline size_t window_smem(int n_chi) { return sizeof(WinShared) + (size_t)n_chi * sizeof(float2); }

template <bool G>
__global__ void __launch_bounds__(kFuseThreads) window_kernel(const StepArgs<float> a, int K) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  WinShared& sh = *reinterpret_cast<WinShared*>(smem_raw);
  float2* cell = reinterpret_cast<float2*>(smem_raw + sizeof(WinShared));
  load_cells(a.tab, cell);
  if ((int)threadIdx.x < K) {
    StepScalars<float>& S = sh.S[threadIdx.x];
    make_scalars<float>(a.field, a.t0 + (double)(a.step + threadIdx.x) * a.dt, a.win_x0, a.win_v, S);
    sh.pair[threadIdx.x] = window_pair(a.field.kind, S);
  }
  if (threadIdx.x == 0) sh.pushed = 0;
  pdl_wait();
  if (G && (int)threadIdx.x < K) sh.S[threadIdx.x].cells = packed_cells<float>(a.field);
  __syncthreads();
  pdl_launch();
  constexpr uint32_t W = kFuseThreads / 32;
  const uint32_t nwin = a.sp[2].cnt->n & ~1023u;
  const uint32_t pushed = __reduce_add_sync(
      kFull, window_photons<G>(a, K, blockIdx.x * W + (threadIdx.x >> 5), nwin >> 5, gridDim.x * W, sh, cell));
  if ((threadIdx.x & 31) == 0 && pushed) atomicAdd(&sh.pushed, pushed);
  __syncthreads();
  if (threadIdx.x == 0) {
    add_window_work(a, sh.pushed);
    if (blockIdx.x == 0) a.sp[2].cnt->win_n = nwin;
  }
}

template <typename R>
__global__ void __launch_bounds__(512) ledger_kernel(const StepArgs<R> a, int nparts) {
  pdl_wait();
  reduce_ledger(a, nparts);
}

// ----------------------------------------------------------------------------- batches
// Copies one slot's arguments into shared memory (8-byte words, all threads).
template <typename R>
__device__ __forceinline__ void load_args(StepArgs<R>& dst, const StepArgs<R>* src) {
  static_assert(sizeof(StepArgs<R>) % 8 == 0, "StepArgs is a whole number of 8-byte words");
  const unsigned long long* s = reinterpret_cast<const unsigned long long*>(src);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(&dst);
  for (int k = threadIdx.x; k < (int)(sizeof(StepArgs<R>) / 8); k += blockDim.x) d[k] = s[k];
  __syncthreads();
}

// One block: which slots step now and how many step-kernel blocks each gets (proportional to
// its tiles, at least one for a slot with work, at most its ledger partials).
template <typename R>
__global__ void __launch_bounds__(1024) batch_schedule_kernel(const BatchCtl<R> c) {
  __shared__ unsigned long long s_tiles;
  if (threadIdx.x == 0) s_tiles = 0ull;
  __syncthreads();
  const int per = (c.S + blockDim.x - 1) / blockDim.x;
  unsigned long long mine = 0;
  for (int q = 0; q < per; ++q) {
    const int sl = threadIdx.x * per + q;
    if (sl >= c.S || c.remaining[sl] == 0u) continue;
    const StepArgs<R>& a = c.args[sl];
    for (int k = 0; k < 3; ++k) mine += (a.sp[k].cnt->n + kTile<R> - 1) / kTile<R>;
  }
  atomicAdd(&s_tiles, mine);
  __syncthreads();
  const double total = (double)s_tiles;
  uint32_t local = 0;
  for (int q = 0; q < per; ++q) {
    const int sl = threadIdx.x * per + q;
    if (sl >= c.S) continue;
    uint32_t b = 0;
    const bool live = c.remaining[sl] > 0u;
    if (live) {
      const StepArgs<R>& a = c.args[sl];
      uint32_t t = 0;
      for (int k = 0; k < 3; ++k) t += (a.sp[k].cnt->n + kTile<R> - 1) / kTile<R>;
      if (t > 0) {
        b = (uint32_t)(c.target_blocks * (double)t / total + 0.5);
        b = max(1u, min(b, min(t, (uint32_t)c.max_parts)));
      }
    }
    c.live[sl] = live ? 1u : 0u;
    local += b;
  }
  uint32_t tot;
  uint32_t run = block_exclusive_scan(local, &tot);
  for (int q = 0; q < per; ++q) {
    const int sl = threadIdx.x * per + q;
    if (sl >= c.S) continue;
    c.blocks[sl] = run;
    if (c.live[sl]) {
      const StepArgs<R>& a = c.args[sl];
      uint32_t t = 0;
      for (int k = 0; k < 3; ++k) t += (a.sp[k].cnt->n + kTile<R> - 1) / kTile<R>;
      if (t > 0) {
        uint32_t b = (uint32_t)(c.target_blocks * (double)t / total + 0.5);
        run += max(1u, min(b, min(t, (uint32_t)c.max_parts)));
      }
    }
  }
  if (threadIdx.x == blockDim.x - 1) c.blocks[c.S] = tot;
}

// Slot of block b: the last slot whose first block is <= b (blocks[] is non-decreasing).
__device__ __forceinline__ int slot_of_block(const uint32_t* blocks, int S, uint32_t b) {
  int lo = 0, hi = S;  // blocks[lo] <= b < blocks[hi]
  while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (blocks[mid] <= b) lo = mid; else hi = mid; }
  return lo;
}

template <typename R>
__device__ __forceinline__ bool is_call_end(const BatchCtl<R>& c, int end) {
  return end == kBatchCallEnd || (end == kBatchGroupEnd && c.tot[1] != 0u);
}
// Steps of a slot's photon window when the batch's spans W: up to the step before its last (whose
// ledger is kept), 0 if that leaves fewer than 2.  end: where the batch's window ends.
template <typename R>
__device__ __forceinline__ uint32_t win_steps(const BatchCtl<R>& c, uint32_t remaining, int W, int end) {
  const uint32_t w = (uint32_t)W - (is_call_end(c, end) ? 1u : 0u);
  const uint32_t k = remaining > 0u ? min(w, remaining - 1u) : 0u;
  return k >= 2u ? k : 0u;
}

// ---- per-step path of a batch: one tile space over all live slots
// The tile schedule (one block) lays the live slots' tiles end to end (slot order, species order
// inside a slot) and evaluates every slot's per-step field
// scalars once.  win_w, win_end, win_s: the batch's photon window and the step's place in it (-1:
// none).  end: the ledgers of all live slots can be read after the call's last step; a slot that
// ends with this step keeps its ledger too.
template <typename R>
__global__ void __launch_bounds__(1024) batch_tiles_kernel(const BatchCtl<R> c, int end, int win_w, int win_end,
                                                           int win_s) {
  pdl_wait();
  pdl_launch();
  const int per = (c.S + blockDim.x - 1) / blockDim.x;
  const int s0 = threadIdx.x * per, s1 = min(c.S, s0 + per);
  uint32_t tiles = 0;
  for (int sl = s0; sl < s1; ++sl) {
    SlotPlan q{};
    q.live = c.remaining[sl] > 0u ? 1u : 0u;
    if (q.live) {
      const StepArgs<R>& a = c.args[sl];
      const uint32_t rem = c.remaining[sl];
      // the slot's place in its photon window (its own may be shorter than the batch's)
      const bool in = win_s >= 0 && (uint32_t)win_s < win_steps(c, rem + (uint32_t)win_s, win_w, win_end);
      if (in) q.win_n = a.sp[2].cnt->win_n;
      for (int k = 0; k < 3; ++k) {
        q.n[k] = a.sp[k].cnt->n;
        q.T[k] = (q.n[k] - (k == 2 ? q.win_n : 0u) + kTile<R> - 1) / kTile<R>;
      }
      q.T[3] = conversion_tiles(q.win_n, (uint32_t)c.target_blocks);
      for (int k = 0; k < 4; ++k) tiles += q.T[k];
      c.args[sl].want = rem == 1u || is_call_end(c, end);
      c.args[sl].win_s = in ? win_s : -1;
      StepScalars<R>& S = static_cast<StepScalars<R>*>(c.scal)[sl];
      make_scalars<R>(a.field, a.t0 + (double)a.step * a.dt, a.win_x0, a.win_v, S);
      for (int k = 0; k < 3; ++k) S.phase[k] = a.sp[k].cnt->phase;
    }
    c.splan[sl] = q;
  }
  uint32_t ttot;
  uint32_t tb = block_exclusive_scan(tiles, &ttot);
  for (int sl = s0; sl < s1; ++sl) {
    SlotPlan& q = c.splan[sl];
    q.tile_base = tb;
    tb += q.T[0] + q.T[1] + q.T[2] + q.T[3];
    c.live[sl] = q.live;
  }
  if (threadIdx.x == 0) c.tot[0] = ttot;
}

// The run that global tile g of the batch step lies in.  A block's tiles increase, so the slot cursor
// only moves forward and the run is looked up again only when g leaves it.
__device__ __forceinline__ void find_run(const SlotPlan* sp, int S, uint32_t g, TileRun& r) {
  if (g >= r.g_lo && g < r.g_hi) return;
  int cur = r.slot;
  while (cur + 1 < S && sp[cur + 1].tile_base <= g) ++cur;
  const SlotPlan& q = sp[cur];
  const uint32_t local = g - q.tile_base, T0 = q.T[0], T1 = q.T[1];
  r.slot = cur;
  r.slot_lo = q.tile_base;
  r.base = 0;
  const uint32_t T2 = q.T[2];
  if (local < T0) { r.s = 0; r.g_lo = q.tile_base; r.g_hi = r.g_lo + T0; r.n = q.n[0]; }
  else if (local < T0 + T1) { r.s = 1; r.g_lo = q.tile_base + T0; r.g_hi = r.g_lo + T1; r.n = q.n[1]; }
  else if (local < T0 + T1 + T2) { r.s = 2; r.g_lo = q.tile_base + T0 + T1; r.g_hi = r.g_lo + T2; r.n = q.n[2]; r.base = q.win_n; }
  else { r.s = 3; r.g_lo = q.tile_base + T0 + T1 + T2; r.g_hi = r.g_lo + q.T[3]; r.n = q.win_n; }  // conversions
}

// Producer (thread kTile<R>): bulk copies of the block's k-th tile, global tile g, into stage
// k % kStages; as issue_tile, with the arrays of the tile's run (kept while the run lasts).
template <typename R>
__device__ __forceinline__ void issue_batch_tile(const BatchCtl<R>& c, TileBuf<R>* buf, uint64_t* bar, uint32_t k,
                                                 uint32_t g, TileRun& run, TileSrc<R>& src) {
  if (!(g >= run.g_lo && g < run.g_hi)) {
    find_run(c.splan, c.S, g, run);
    if (run.s < 3) src = tile_src(c.args[run.slot].sp[run.s]);
  }
  if (run.s == 3) {  // nothing to copy
    mbar_arrive(&bar[k % kStages]);
    return;
  }
  const TileSrc<R>& sp = src;
  const uint32_t first = run.base + (g - run.g_lo) * kTile<R>;
  const uint32_t valid = min((uint32_t)kTile<R>, run.n - first);
  const uint32_t br = floor16(valid * (uint32_t)sizeof(R)), bt = floor16(valid * 8u);
  TileBuf<R>& b = buf[k % kStages];
  uint64_t* bb = &bar[k % kStages];
  mbar_arrive_expect_tx(bb, 6u * br + bt);
  if (br) {
    bulk_load(b.x, sp.x + first, br, bb);
    bulk_load(b.y, sp.y + first, br, bb);
    bulk_load(b.z, sp.z + first, br, bb);
    bulk_load(b.ux, sp.ux + first, br, bb);
    bulk_load(b.uy, sp.uy + first, br, bb);
    bulk_load(b.uz, sp.uz + first, br, bb);
  }
  if (bt) bulk_load(b.tau, sp.tau + first, bt, bb);
}

// One batch step of every live slot in one persistent launch.  Block blk takes the global tiles
// blk, blk + G, blk + 2G, ... (G = gridDim.x), whatever slot they belong to, so every block gets
// an equal share of tiles in one wave.  Inside a slot, block blk takes exactly the slot-local
// tiles j = p, p + G, ... (p: its first one) that block p takes when the slot runs alone with the
// same grid, and writes ledger partial p: a scenario's ledger partials, and so its ledger, are the
// same alone and in any mix.  The warp roles, the pipeline and the per-warp event rings are those
// of step_body; the compute warps switch to a slot's arguments and field scalars together (named
// barrier) when their tiles move on to the next slot, after taking the events queued for it and
// writing its ledger partial.
template <typename R, bool G>
__global__ void __launch_bounds__(kStepThreads<R>, sizeof(R) == 4 ? QED_BATCH_MIN_BLOCKS : 256 / kTile<double>)
batch_step_kernel(const BatchCtl<R> c) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  TileBuf<R>* buf = reinterpret_cast<TileBuf<R>*>(smem_raw);
  EventRing<R>* ring = reinterpret_cast<EventRing<R>*>(buf + kStages);
  R* s_lnh = reinterpret_cast<R*>(ring + kWarps<R>);
  R* s_lnT = s_lnh + c.tab.n_eta;
  __shared__ __align__(8) uint64_t full[kStages];
  __shared__ __align__(8) uint64_t empty[kStages];
  __shared__ __align__(16) StepArgs<R> A;
  __shared__ __align__(16) StepScalars<R> S;
  __shared__ int s_abort;
  __shared__ uint32_t s_work[2];

  const uint32_t blk = blockIdx.x, nblk = gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < c.tab.n_eta; k += blockDim.x) s_lnh[k] = c.tab.ln_h[k];
  for (int k = threadIdx.x; k < c.tab.n_chi; k += blockDim.x) s_lnT[k] = c.tab.ln_T[k];
  if (threadIdx.x == kTile<R>) {
    for (int st = 0; st < kStages; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], kWarps<R>);
    }
    mbar_fence_init();
    s_abort = 0;
    s_work[0] = s_work[1] = 0;
  }
  pdl_wait();
  const uint32_t ttot = c.tot[0];
  __syncthreads();
  pdl_launch();
  TileRun prun;  // producer's run of tiles and its arrays
  TileSrc<R> psrc{};
  if (threadIdx.x == kTile<R>)
    for (uint32_t k = 0; k < (uint32_t)kStages && blk + k * nblk < ttot; ++k)
      issue_batch_tile(c, buf, full, k, blk + k * nblk, prun, psrc);

  if (warp == kWarps<R>) {
    // ---------------- producer
    if (lane == 0) {
      uint32_t k = kStages;
      for (;; ++k) {
        if (blk + k * nblk >= ttot || s_abort) break;
        const int st = (int)(k % kStages);
        if (!mbar_wait_bounded(&empty[st], ((k / kStages) - 1u) & 1u, kWaitLimit)) { s_abort = 1; break; }
        fence_proxy_async_smem();
        issue_batch_tile(c, buf, full, k, blk + k * nblk, prun, psrc);
      }
      if (s_abort) {
        atomicOr(&c.args[0].sp[0].cnt->err, 1u << QED_ERR_TIMEOUT);
        const uint32_t first = k >= (uint32_t)kStages ? k - kStages : 0u;
        for (uint32_t q = first; q < k; ++q)
          if (blk + q * nblk < ttot) mbar_wait_bounded(&full[q % kStages], (q / kStages) & 1u, kWaitLimit);
      }
    }
    return;  // the producer takes part in no later barrier
  }
  // ---------------- compute warps
  WarpState<R> w;
  w.q = EventQueue<R>{ring + warp, 0u, 0u};
  if (lane == 0) w.q.r->sums = EventSums<R>{};
  __syncwarp();
  const StepPipe<R> P{buf, full, empty, ring, s_lnh, s_lnT, &s_abort, blk, nblk};
  TileRun run;
  int cur = -1;
  uint32_t part = 0;
  const int nw = (int)(sizeof(StepArgs<R>) / 8), ns = (int)(sizeof(StepScalars<R>) / 8);
  static_assert(sizeof(StepArgs<R>) % 8 == 0 && sizeof(StepScalars<R>) % 8 == 0, "8-byte words");
  auto flush_slot = [&]() {
    add_work(w.pushed_ph, w.tau_ph, s_work, lane);
    w.pushed_ph = w.tau_ph = 0;
    compute_warps_sync<R>();  // every warp has added its work and its sums
    if (threadIdx.x == 0) {
      flush_work(s_work, A.work);
      s_work[0] = s_work[1] = 0;
    }
    if (A.want) {
      write_step_partial<R>(ring, A.ledger_part, part);
      compute_warps_sync<R>();
      if (lane == 0) w.q.r->sums = EventSums<R>{};
    }
  };
  for (;;) {
    const uint32_t g = blk + w.k * nblk;
    if (g >= ttot) break;
    find_run(c.splan, c.S, g, run);
    if (run.slot != cur) {
      if (cur >= 0) flush_slot();
      compute_warps_sync<R>();  // every warp is done with the previous slot's arguments
      const unsigned long long* sa = reinterpret_cast<const unsigned long long*>(c.args + run.slot);
      const unsigned long long* ss = reinterpret_cast<const unsigned long long*>(
          static_cast<const StepScalars<R>*>(c.scal) + run.slot);
      unsigned long long* da = reinterpret_cast<unsigned long long*>(&A);
      unsigned long long* ds = reinterpret_cast<unsigned long long*>(&S);
      for (int q = threadIdx.x; q < nw; q += kTile<R>) da[q] = sa[q];
      for (int q = threadIdx.x; q < ns; q += kTile<R>) ds[q] = ss[q];
      compute_warps_sync<R>();
      cur = run.slot;
      part = g - run.slot_lo;  // < G: the block's first tile of the slot
    }
    // (a batch with a grid field runs the grid-capable instantiation: the general class only)
    if (A.want) run_species<R, G, true>(A, S, P, run, w);
    else run_species<R, G, false>(A, S, P, run, w);
  }
  // a wait that gave up leaves the step unfinished (QED_ERR_TIMEOUT): events still in the rings
  // are not taken
  if (cur >= 0) flush_slot();
}

constexpr int kMaxScatterSlots = 4096;  // slots of a batch at most

// Per-slot plan (one block per live slot): the exclusive prefixes of its species' coarse event
// counts, the merge plan, the slot's ledger (from its partials 0 .. min(its tiles, G) - 1) where it
// can be read, and the counts of the step before cleared.
template <typename R>
__global__ void __launch_bounds__(256) batch_plan_kernel(const BatchCtl<R> c, int G) {
  __shared__ uint32_t s_tot;
  pdl_wait();
  pdl_launch();
  const int sl = blockIdx.x;
  const SlotPlan& q = c.splan[sl];
  if (!q.live) return;
  const StepArgs<R>& a = c.args[sl];
  for (int s = 0; s < 3; ++s) {
    const SpeciesDev<R>& sp = a.sp[s];
    if ((s < 2 ? a.sp[2] : a.sp[0]).cnt->n_app == 0u) continue;  // (uniform) no child asks for it
    const uint32_t nc = coarses_of(q.n[s]);
    const uint32_t* co = sp.coarse + sp.cnt->phase * event_coarses(sp.cap);
    uint32_t base = 0;
    for (uint32_t k0 = 0; k0 < nc; k0 += blockDim.x) {
      const uint32_t k = k0 + threadIdx.x, v = k < nc ? co[k] : 0u;
      uint32_t tot;
      const uint32_t ex = block_exclusive_scan(v, &tot);
      if (k < nc) sp.cprefix[k] = base + ex;
      base += tot;
    }
    if (s == 0 && threadIdx.x == 0) s_tot = base;
  }
  __syncthreads();
  if (threadIdx.x == 0) *a.plan = make_plan(a, a.sp[2].cnt->n_app ? s_tot : 0u, true);
  FinalizePlan P;
  for (int s = 0; s < 3; ++s) P.phase[s] = a.sp[s].cnt->phase;
  clear_other_counts(a, P, threadIdx.x, blockDim.x);
  if (a.want) reduce_ledger(a, (int)min(q.T[0] + q.T[1] + q.T[2], (uint32_t)G));
}

// The new particles of every live slot, ranked and moved into place (place_child) by a grid that
// strides through all slots' children together; the first threads of block 0 then set each
// slot's counters and advance its step.
template <typename R>
__global__ void __launch_bounds__(256) batch_scatter_kernel(const BatchCtl<R> c) {
  __shared__ uint32_t s_base[kMaxScatterSlots + 1];
  pdl_wait();
  pdl_launch();
  const int per = (c.S + blockDim.x - 1) / blockDim.x;
  const int s0 = threadIdx.x * per, s1 = min(c.S, s0 + per);
  uint32_t mine = 0;
  for (int sl = s0; sl < s1; ++sl) {
    uint32_t m = 0;
    if (c.splan[sl].live) { const FinalizePlan* P = c.args[sl].plan; m = P->m[0] + P->m[1] + P->m[2]; }
    s_base[sl] = m;
    mine += m;
  }
  __syncthreads();
  uint32_t tot;
  uint32_t run = block_exclusive_scan(mine, &tot);
  for (int sl = s0; sl < s1; ++sl) { const uint32_t m = s_base[sl]; s_base[sl] = run; run += m; }
  if (threadIdx.x == 0) s_base[c.S] = tot;
  __syncthreads();
  for (uint32_t ci = blockIdx.x * blockDim.x + threadIdx.x; ci < tot; ci += gridDim.x * blockDim.x) {
    int lo = 0, hi = c.S;  // s_base[lo] <= ci < s_base[hi]
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (s_base[mid] <= ci) lo = mid; else hi = mid; }
    const StepArgs<R>& a = c.args[lo];
    place_child<R>(a, *a.plan, ci - s_base[lo], [&](int s, uint32_t cg) { return a.sp[s].cprefix[cg]; });
  }
  if (blockIdx.x == 0)
    for (int sl = threadIdx.x; sl < c.S; sl += blockDim.x) {
      if (!c.splan[sl].live) continue;
      const StepArgs<R>& a = c.args[sl];
      finish_counters<R>(a, *a.plan, c.splan[sl].n);
      c.args[sl].step = a.step + 1;  // the slot's next step
      c.remaining[sl] -= 1u;
    }
}

// A photon window in a batch (24 scenarios of 1e3 to 2e5 electrons, 256 steps on GB300: 106 -> 82 ms
// with it, 57 ms with the block-wide event batches and the guides): first the field scalars of every live slot's window steps (one thread
// each, 16 per slot) and the photons it takes, then the photons of all slots, in units of 4096 that
// a persistent grid strides through (a unit lies in one slot; its 8 warps share its chunks).
__global__ void __launch_bounds__(128) batch_window_prepare_kernel(const BatchCtl<float> c, int W, int end) {
  pdl_wait();
  pdl_launch();
  const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x), sl = t / kWinMax, k = t % kWinMax;
  if (sl >= c.S) return;
  const StepArgs<float>& a = c.args[sl];
  const uint32_t rem = c.remaining[sl];
  if (rem == 0u) return;
  const uint32_t K = win_steps(c, rem, W, end);
  if (k == 0) a.sp[2].cnt->win_n = K ? a.sp[2].cnt->n & ~1023u : 0u;
  if ((uint32_t)k < K)
    make_scalars<float>(a.field, a.t0 + (double)(a.step + k) * a.dt, a.win_x0, a.win_v,
                        static_cast<StepScalars<float>*>(c.wscal)[sl * kWinMax + k]);
}

constexpr uint32_t kUnitChunks = 128;  // chunks of 32 photons per unit
template <bool G>
__global__ void __launch_bounds__(kFuseThreads) batch_window_kernel(const BatchCtl<float> c, int W, int end) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  WinShared& sh = *reinterpret_cast<WinShared*>(smem_raw);
  float2* cell = reinterpret_cast<float2*>(smem_raw + sizeof(WinShared));
  __shared__ __align__(16) StepArgs<float> A;
  __shared__ uint32_t s_base[kMaxScatterSlots + 1];  // exclusive prefix of the slots' units
  load_cells(c.tab, cell);
  pdl_wait();
  pdl_launch();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (c.S + kFuseThreads - 1) / kFuseThreads;
  const int s0 = threadIdx.x * per, s1 = min(c.S, s0 + per);
  uint32_t mine = 0;
  for (int sl = s0; sl < s1; ++sl) {
    uint32_t u = 0;
    if (c.remaining[sl] > 0u) u = ((c.args[sl].sp[2].cnt->win_n >> 5) + kUnitChunks - 1) / kUnitChunks;
    s_base[sl] = u;
    mine += u;
  }
  __syncthreads();
  uint32_t tot;
  uint32_t run = block_exclusive_scan(mine, &tot);
  for (int sl = s0; sl < s1; ++sl) { const uint32_t u = s_base[sl]; s_base[sl] = run; run += u; }
  if (threadIdx.x == 0) s_base[c.S] = tot;
  __syncthreads();
  int cur = -1, K = 0;
  uint32_t pushed = 0;
  for (uint32_t u = blockIdx.x; u < tot; u += gridDim.x) {
    int lo = cur < 0 ? 0 : cur, hi = c.S;  // s_base[lo] <= u < s_base[hi]
    while (hi - lo > 1) { const int mid = (lo + hi) >> 1; if (s_base[mid] <= u) lo = mid; else hi = mid; }
    if (lo != cur) {
      if (cur >= 0) {
        pushed = __reduce_add_sync(kFull, pushed);
        if (lane == 0) add_window_work(A, pushed);
        pushed = 0;
      }
      __syncthreads();
      const unsigned long long* src = reinterpret_cast<const unsigned long long*>(c.args + lo);
      for (int w = threadIdx.x; w < (int)(sizeof(StepArgs<float>) / 8); w += kFuseThreads)
        reinterpret_cast<unsigned long long*>(&A)[w] = src[w];
      K = (int)win_steps(c, c.remaining[lo], W, end);
      const StepScalars<float>* ws = static_cast<const StepScalars<float>*>(c.wscal) + lo * kWinMax;
      const unsigned long long* wsrc = reinterpret_cast<const unsigned long long*>(ws);
      for (int w = threadIdx.x; w < K * (int)(sizeof(StepScalars<float>) / 8); w += kFuseThreads)
        reinterpret_cast<unsigned long long*>(sh.S)[w] = wsrc[w];
      if ((int)threadIdx.x < K) sh.pair[threadIdx.x] = window_pair(ws[threadIdx.x].kind, ws[threadIdx.x]);
      __syncthreads();
      cur = lo;
    }
    const uint32_t c0 = (u - s_base[cur]) * kUnitChunks;
    pushed += window_photons<G>(A, K, c0 + warp, min(c0 + kUnitChunks, A.sp[2].cnt->win_n >> 5), kFuseThreads / 32, sh, cell);
  }
  if (cur >= 0) {
    pushed = __reduce_add_sync(kFull, pushed);
    if (lane == 0) add_window_work(A, pushed);
  }
}

// Multi-step passes in a batch (when fuse_k >= 2): every live slot probes up to
// min(fuse_k, remaining) steps, commits its event-free stretch and advances by it; then the
// regular batch step follows, so a batch step moves a slot by one step plus its stretch.  Each
// slot runs the single-scenario bodies, so its particles are those of qed_run.
// A probe costs a pass over the slot's particles for up to its span of steps, so the span
// adapts per slot: it doubles (up to fuse_k) after a probe that found no event, shrinks to what
// was found otherwise, and a probe that finds an event in the first step makes the slot wait
// fuse_k batch steps before probing again.
template <typename R>
__global__ void __launch_bounds__(1024) batch_probe_init_kernel(const BatchCtl<R> c) {
  for (int sl = threadIdx.x; sl < c.S; sl += blockDim.x) {
    uint32_t k = 0;
    if (c.live[sl]) {
      if (c.skip[sl] > 0) c.skip[sl] -= 1u;
      else k = min(max(c.span[sl], 2u), min((uint32_t)c.fuse_k, c.remaining[sl]));
    }
    c.first_event[sl] = k;
    c.tried[sl] = k;
  }
}

template <typename R, bool G, bool COMMIT>
__global__ void __launch_bounds__(kFuseThreads) batch_fused_kernel(const BatchCtl<R> c) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(16) StepArgs<R> A;
  __shared__ int s_K;
  const uint32_t b = blockIdx.x;
  if (b >= c.blocks[c.S]) return;
  const int sl = slot_of_block(c.blocks, c.S, b);
  // probe: the stretch still worth trying (other blocks of the slot may be lowering it right
  // now); commit: the event-free steps the probe found.  Read once, so that the whole block
  // takes the same branch and copies the arguments together.
  if (threadIdx.x == 0) s_K = (int)*reinterpret_cast<volatile uint32_t*>(c.first_event + sl);
  __syncthreads();
  const int K = s_K;
  if (K == 0) return;
  load_args(A, c.args + sl);
  if (threadIdx.x == 0) A.want = 1;  // the stretch may use up the slot's steps
  __syncthreads();
  const uint32_t bb = b - c.blocks[sl], nb = c.blocks[sl + 1] - c.blocks[sl];
  if (A.field.kind == QED_FIELD_PLANE_LP) fused_body<R, G, COMMIT, kFieldLP>(A, K, c.first_event + sl, bb, nb, smem_raw);
  else if (A.field.kind == QED_FIELD_PLANE_CP) fused_body<R, G, COMMIT, kFieldCP>(A, K, c.first_event + sl, bb, nb, smem_raw);
  else fused_body<R, G, COMMIT, kFieldAny>(A, K, c.first_event + sl, bb, nb, smem_raw);
}

template <typename R>
__global__ void __launch_bounds__(1024) batch_commit_plan_kernel(const BatchCtl<R> c) {
  __shared__ __align__(16) StepArgs<R> A;
  const int sl = blockIdx.x;
  const uint32_t k = c.first_event[sl], tried = c.tried[sl];
  if (threadIdx.x == 0 && tried > 0) {
    if (k == 0) c.skip[sl] = (uint32_t)c.fuse_k;
    c.span[sl] = k == tried ? min(2u * tried, (uint32_t)c.fuse_k) : max(k, 2u);
  }
  if (k == 0) return;
  load_args(A, c.args + sl);
  reduce_ledger(A, (int)(c.blocks[sl + 1] - c.blocks[sl]));  // no children: the ledger of the stretch's last step
  __syncthreads();
  if (threadIdx.x == 0) {
    c.args[sl].step = A.step + k;
    c.remaining[sl] -= k;
  }
}

// ----------------------------------------------------------------------------- utilities
template <typename R>
__global__ void init_tau_kernel(const SpeciesDev<R> sp, int kind, uint64_t seed, uint64_t scen) {
  const uint32_t n = sp.cnt->n;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double U[4];
    draw4(seed, scen, sp.id[i], 0, (uint64_t)kind, 1, U);
    store_tau_from_double<R>(sp.tau + i, -log(U[0]));
  }
}

template <typename R>
__global__ void eval_kernel(const TabDev<R> tab, const FieldDev f, int kind, double t, double wx0, double wv, size_t n,
                            const double* x, const double* y, const double* z, const double* ux, const double* uy,
                            const double* uz, double* oE, double* oB, double* op, double* oe, double* orate) {
  __shared__ StepScalars<R> S;
  if (threadIdx.x == 0) make_scalars<R>(f, t, wx0, wv, S);
  __syncthreads();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    R E[3], B[3], amp = (R)0, u[3] = {(R)ux[i], (R)uy[i], (R)uz[i]};
    const int fc = field_at<R, true>(S, (R)x[i], (R)y[i], (R)z[i], E, B, amp);
    int oor;
    R param, energy, inv, rate;
    // the step's own forms: energy and its inverse from one reciprocal square root, the
    // quantum parameter for the field case, the same look-ups
    if (kind == QED_PHOTON) {
      Num<R>::root_inv_(dot3<R>(u, u), energy, inv);
      param = chi_for<R>(fc, u, energy, E, B, amp);
      rate = param > (R)0 ? (R)kAlpha * param * inv * lookup_T<R>(tab, tab.ln_T, param, oor) : (R)0;
    } else {
      Num<R>::root_inv_((R)1 + dot3<R>(u, u), energy, inv);
      param = eta_for<R>(fc, u, energy, E, B, amp);
      rate = param > (R)0 ? (R)kRatePhoton * param * inv * lookup_h<R>(tab, tab.ln_h, param, oor) : (R)0;
    }
    for (int c = 0; c < 3; ++c) { oE[3 * i + c] = (double)E[c]; oB[3 * i + c] = (double)B[c]; }
    op[i] = (double)param;
    oe[i] = (double)energy;
    orate[i] = (double)rate;
  }
}

template <typename R>
__global__ void sample_kernel(const TabDev<R> tab, int which, size_t n, const double* param, const double* U,
                              double* out, int32_t* ok) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    if (which >= 2) {
      // the step's rate look-ups for a given parameter, from the tables staged as the step does
      int oor = 0;
      const R v = which == 2 ? lookup_h<R>(tab, tab.ln_h, (R)param[i], oor) : lookup_T<R>(tab, tab.ln_T, (R)param[i], oor);
      out[i] = (double)v;
      ok[i] = oor;
      continue;
    }
    const R u = (R)U[i], v = (R)(1.0 - U[i]);
    if (which == 0) {
      R xi = (R)0;
      const bool good = sample_xi<R>(tab, (R)param[i], u, v, xi);
      out[i] = good ? (double)xi : 0.0;
      ok[i] = good ? 1 : 0;
    } else {
      out[i] = (double)sample_f<R, 1, true>(tab, Num<R>::log_((R)param[i]), u, v);
      ok[i] = 1;
    }
  }
}

__global__ void philox_kernel(size_t n, const uint64_t* ctr, uint64_t k0, uint64_t k1, uint64_t* out) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    uint64_t c[4] = {ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]};
    philox4x64(c, k0, k1);
    for (int j = 0; j < 4; ++j) out[4 * i + j] = c[j];
  }
}

// ----------------------------------------------------------------------------- tau format
// In-place conversion between the C ABI's double optical depth and the stored representation
// (identical for FP64; a compensated float pair for the mixed path).  Exact round trip.
template <typename R>
__global__ void tau_from_double_kernel(double* tau, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    store_tau_from_double<R>(tau + i, tau[i]);
}
template <typename R>
__global__ void tau_to_double_kernel(double* tau, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    tau[i] = tau_to_double<R>(tau + i);
}

// ----------------------------------------------------------------------------- compaction
// Stable removal of converted photons (tau = +inf) into a second array set, three passes over
// segments of 2048 particles: count survivors, scan the counts (one block), scatter in order.
constexpr uint32_t kSeg = 2048;

template <typename R>
__global__ void __launch_bounds__(256) compact_count_kernel(const SpeciesDev<R> sp, uint32_t* seg_count) {
  const uint32_t n = sp.cnt->n, nseg = (n + kSeg - 1) / kSeg;
  for (uint32_t g = blockIdx.x; g < nseg; g += gridDim.x) {
    uint32_t c = 0;
    for (uint32_t i = g * kSeg + threadIdx.x; i < min(n, (g + 1) * kSeg); i += blockDim.x)
      c += !Tau<R>::load(sp.tau + i).dead();
    uint32_t tot;
    block_exclusive_scan(c, &tot);
    if (threadIdx.x == 0) seg_count[g] = tot;
  }
}

template <typename R>
__global__ void __launch_bounds__(1024) compact_scan_kernel(const SpeciesDev<R> sp, uint32_t* seg_count,
                                                             uint32_t* seg_prefix) {
  const uint32_t n = sp.cnt->n, nseg = (n + kSeg - 1) / kSeg;
  const uint32_t per = (nseg + blockDim.x - 1) / blockDim.x;
  const uint32_t r0 = threadIdx.x * per, r1 = min(nseg, r0 + per);
  uint32_t local = 0;
  for (uint32_t r = r0; r < r1; ++r) local += seg_count[r];
  uint32_t total;
  uint32_t run = block_exclusive_scan(local, &total);
  for (uint32_t r = r0; r < r1; ++r) { seg_prefix[r] = run; run += seg_count[r]; }
  if (threadIdx.x == 0) seg_prefix[nseg] = total;
}

template <typename R>
__global__ void __launch_bounds__(256) compact_scatter_kernel(const SpeciesDev<R> sp, SpeciesDev<R> out,
                                                              const uint32_t* seg_prefix) {
  // warp w moves the segment's particles [256 w, 256 w + 256), 32 at a time: its survivors are counted
  // first, so the block synchronises once per segment (2.4e6 of 3e6 photons: 106 -> 60 us on GB300
  // against a block-wide scan for every 256)
  __shared__ uint32_t s_w[8];
  const uint32_t n = sp.cnt->n, nseg = (n + kSeg - 1) / kSeg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kRounds = kSeg / 256;
  for (uint32_t g = blockIdx.x; g < nseg; g += gridDim.x) {
    const uint32_t first = g * kSeg + (uint32_t)warp * (kRounds * 32u) + (uint32_t)lane;
    unsigned keep[kRounds];
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
      const uint32_t i = first + 32u * q;
      keep[q] = __ballot_sync(kFull, i < n && !Tau<R>::load(sp.tau + i).dead());
      mine += (uint32_t)__popc(keep[q]);
    }
    __syncthreads();  // the last segment's counts have been read
    if (lane == 0) s_w[warp] = mine;
    __syncthreads();
    uint32_t base = seg_prefix[g];
    for (int w = 0; w < warp; ++w) base += s_w[w];
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
      const uint32_t i = first + 32u * q;
      if (keep[q] >> lane & 1u) {
        const uint32_t o = base + (uint32_t)__popc(keep[q] & ((1u << lane) - 1u));
        out.x[o] = sp.x[i]; out.y[o] = sp.y[i]; out.z[o] = sp.z[i];
        out.ux[o] = sp.ux[i]; out.uy[o] = sp.uy[i]; out.uz[o] = sp.uz[i];
        out.tau[o] = sp.tau[i]; out.id[o] = sp.id[i];
        if (sp.w) out.w[o] = sp.w[i];
      }
      base += (uint32_t)__popc(keep[q]);
    }
  }
}

// The new count, once every block of the scatter has read the old one.
template <typename R>
__global__ void compact_finish_kernel(const SpeciesDev<R> sp, const uint32_t* seg_prefix) {
  const uint32_t n = sp.cnt->n, nseg = (n + kSeg - 1) / kSeg;
  sp.cnt->n = seg_prefix[nseg];
  sp.cnt->n_dead = 0;
}

std::atomic<uint64_t> g_launches{0};
int g_sm_count = 0;

int sm_count() {
  if (g_sm_count == 0) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    g_sm_count = v > 0 ? v : 1;
  }
  return g_sm_count;
}

int small_grid(size_t n) {
  const size_t want = (n + 255) / 256;
  const size_t cap = (size_t)sm_count() * 8;
  return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}
}  // namespace

#if QED_PART(1)
void count_launch(int n) { g_launches += (uint64_t)n; }
uint64_t launch_count_value() { return g_launches.load(); }
#endif

// Launch with programmatic dependent launch: the kernel may start before the one ahead of it in
// the stream has finished, and calls pdl_wait before it touches anything that one writes.
template <typename... P, typename... A>
static void launch_pdl(void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, P(args)...);
}

// dynamic shared memory of the step kernel: the tile stages, the compute warps' event rings,
// then ln h and ln T
template <typename R>
static size_t step_smem(int n_eta, int n_chi) {
  return (size_t)kStages * sizeof(TileBuf<R>) + (size_t)kWarps<R> * sizeof(EventRing<R>) +
         (size_t)(n_eta + n_chi) * sizeof(R);
}

// Resident blocks per SM of a kernel at a given dynamic shared memory size, with its limit raised to
// it (never lowered: another thread may be about to launch with more): asked of the runtime once per
// kernel, device and size (the queries took a third of a one-step call's 12 us on the host).  Any
// thread; the limit is compared and raised under a lock.
struct Residency {
  std::atomic<uint64_t> known[128];  // per device: size << 16 | blocks (0: not asked yet)
  template <typename F>
  int operator()(F kernel, int threads, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<uint64_t>* slot = dev >= 0 && dev < 128 ? &known[dev] : nullptr;
    const uint64_t have = slot ? slot->load(std::memory_order_relaxed) : 0;
    if (have && (have >> 16) == smem) return (int)(have & 0xffffu);
    static std::mutex m;  // (one for all that ask for the same kernel type)
    std::lock_guard<std::mutex> lock(m);
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess || (size_t)fa.maxDynamicSharedSizeBytes < smem)
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess || b < 1) return 1;
    if (slot) slot->store((uint64_t)smem << 16 | (uint64_t)b, std::memory_order_relaxed);
    return b;
  }
};

#if QED_PART(1)
int step_grid_size(int precision) {
  // occupancy for the paper's table sizes (256 eta, 256 chi)
  static Residency mixed, fp64;
  const int b = precision == QED_MIXED ? mixed(step_kernel<float, false, false>, kStepThreads<float>, step_smem<float>(256, 256))
                                       : fp64(step_kernel<double, false, false>, kStepThreads<double>, step_smem<double>(256, 256));
  return sm_count() * b;
}

template <typename R>
void launch_step(const StepArgs<R>& a, int grid, int block, size_t smem_unused, cudaStream_t s) {
  (void)block;
  (void)smem_unused;
  const size_t smem = step_smem<R>(a.tab.n_eta, a.tab.n_chi);
  // the grid-capable instantiation runs in waves if it fits fewer blocks per SM; the analytic-field
  // one sets the persistent grid size
  const bool g = a.field.kind == QED_FIELD_GRID;
  const auto k = a.want ? (g ? step_kernel<R, true, true> : step_kernel<R, false, true>)
                        : (g ? step_kernel<R, true, false> : step_kernel<R, false, false>);
  static Residency known[4];
  known[(a.want ? 2 : 0) + (g ? 1 : 0)](k, kStepThreads<R>, smem);  // (raises the shared memory limit)
  launch_pdl(k, grid, kStepThreads<R>, smem, s, a);
  count_launch();
}

#endif

#if QED_PART(2)
void launch_batch_window(const BatchCtl<float>& c, int n_chi, int W, BatchEnd end, cudaStream_t s) {
  launch_pdl(batch_window_prepare_kernel, (c.S * kWinMax + 127) / 128, 128, 0, s, c, W, (int)end);
  const size_t smem = window_smem(n_chi);
  const auto k = c.grid_fields ? batch_window_kernel<true> : batch_window_kernel<false>;
  static Residency known[2];
  launch_pdl(k, sm_count() * known[c.grid_fields != 0](k, kFuseThreads, smem), kFuseThreads, smem, s, c, W, (int)end);
  count_launch(2);
}

template <typename R>
void launch_batch_step(const BatchCtl<R>& c, int n_eta, int n_chi, BatchEnd end, int win_w, BatchEnd win_end, int win_s,
                       cudaStream_t s) {
  const size_t smem = step_smem<R>(n_eta, n_chi);
  const auto k = c.grid_fields ? batch_step_kernel<R, true> : batch_step_kernel<R, false>;
  static Residency known[2];
  known[c.grid_fields != 0](k, kStepThreads<R>, smem);  // (raises the shared memory limit)
  if (c.fuse_k >= 2) {
    const size_t fsm = (size_t)(n_eta + n_chi) * sizeof(R);
    const int fgrid = c.target_blocks + c.S;
    batch_schedule_kernel<R><<<1, 1024, 0, s>>>(c);
    batch_probe_init_kernel<R><<<1, 1024, 0, s>>>(c);
    if (c.grid_fields) {
      batch_fused_kernel<R, true, false><<<fgrid, kFuseThreads, fsm, s>>>(c);
      batch_fused_kernel<R, true, true><<<fgrid, kFuseThreads, fsm, s>>>(c);
    } else {
      batch_fused_kernel<R, false, false><<<fgrid, kFuseThreads, fsm, s>>>(c);
      batch_fused_kernel<R, false, true><<<fgrid, kFuseThreads, fsm, s>>>(c);
    }
    batch_commit_plan_kernel<R><<<c.S, 1024, 0, s>>>(c);
    count_launch(5);
  }
  // the per-step path: one tile space over all live slots, strided by a persistent grid
  launch_pdl(batch_tiles_kernel<R>, 1, 1024, 0, s, c, (int)end, win_w, (int)win_end, win_s);
  launch_pdl(k, c.target_blocks, kStepThreads<R>, smem, s, c);
  launch_pdl(batch_plan_kernel<R>, c.S, 256, 0, s, c, c.target_blocks);
  launch_pdl(batch_scatter_kernel<R>, sm_count() * 4, 256, 0, s, c);
  count_launch(4);
}

#endif

#if QED_PART(1)
size_t step_scalars_bytes(int precision) {
  return precision == QED_MIXED ? sizeof(StepScalars<float>) : sizeof(StepScalars<double>);
}

// grid of the multi-step kernels: every SM full, never more blocks than ledger partials
template <typename R, bool G, bool C>
static int fused_grid(int max_parts, size_t smem) {
  static Residency known;
  return std::max(1, std::min(max_parts, sm_count() * known(fused_kernel<R, G, C>, kFuseThreads, smem)));
}

template <typename R>
int launch_fused(const StepArgs<R>& a, int K, bool commit, uint32_t* first_event, int max_parts, cudaStream_t s) {
  const size_t smem = (size_t)(a.tab.n_eta + a.tab.n_chi) * sizeof(R);
  const bool g = a.field.kind == QED_FIELD_GRID;
  int grid;
  if (!commit) {
    set_u32_kernel<<<1, 1, 0, s>>>(first_event, (uint32_t)K);
    if (g) {
      grid = fused_grid<R, true, false>(max_parts, smem);
      fused_kernel<R, true, false><<<grid, kFuseThreads, smem, s>>>(a, K, first_event);
    } else {
      grid = fused_grid<R, false, false>(max_parts, smem);
      fused_kernel<R, false, false><<<grid, kFuseThreads, smem, s>>>(a, K, first_event);
    }
    count_launch(2);
  } else {
    if (g) {
      grid = fused_grid<R, true, true>(max_parts, smem);
      fused_kernel<R, true, true><<<grid, kFuseThreads, smem, s>>>(a, K, first_event);
    } else {
      grid = fused_grid<R, false, true>(max_parts, smem);
      fused_kernel<R, false, true><<<grid, kFuseThreads, smem, s>>>(a, K, first_event);
    }
    count_launch(1);
  }
  return grid;
}

int fuse_max_steps() { return kMaxFuse; }

void launch_window(const StepArgs<float>& a, int K, cudaStream_t s) {
  const size_t smem = window_smem(a.tab.n_chi);
  const bool g = a.field.kind == QED_FIELD_GRID;
  const auto k = g ? window_kernel<true> : window_kernel<false>;
  static Residency known[2];
  launch_pdl(k, sm_count() * known[g](k, kFuseThreads, smem), kFuseThreads, smem, s, a, K);
  count_launch();
}

void launch_selftest_wait(uint32_t polls, uint32_t* bits, cudaStream_t s) {
  selftest_wait_kernel<<<1, 32, 0, s>>>(polls, bits);
  count_launch();
}

template <typename R>
void launch_finalize(const StepArgs<R>& a, int step_grid, cudaStream_t s) {
  launch_pdl(finalize_kernel<R>, sm_count(), kFinalThreads, 0, s, a, step_grid);
  count_launch();
}

void launch_pack_grid(const StepArgs<float>& a, uint64_t steps, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  const size_t layer = ((size_t)a.field.n[0] + 1) * ((size_t)a.field.n[1] + 1);
  const size_t gx = (layer + 255) / 256, room = std::max<size_t>(1, (size_t)sm_count() * 8 / (6 * gx));
  cfg.gridDim = dim3((unsigned)gx, (unsigned)std::min<size_t>((size_t)a.field.n[2] + 1, room), 6);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchKernelEx(&cfg, pack_grid_kernel, a, steps);
  count_launch();
}

template <typename R>
void launch_ledger(const StepArgs<R>& a, int parts, cudaStream_t s) {
  ledger_kernel<R><<<1, 512, 0, s>>>(a, parts);
  count_launch();
}

#endif

#if QED_PART(3)
template <typename R>
void launch_init_tau(const SpeciesDev<R>& sp, int kind, uint64_t seed, uint64_t scen, cudaStream_t s) {
  init_tau_kernel<R><<<sm_count() * 4, 256, 0, s>>>(sp, kind, seed, scen);
  count_launch();
}

template <typename R>
void launch_eval(const TabDev<R>& tab, const FieldDev& f, int kind, double t, double wx0, double wv, size_t n,
                 const double* x, const double* y, const double* z, const double* ux, const double* uy,
                 const double* uz, double* oE, double* oB, double* op, double* oe, double* orate, cudaStream_t s) {
  eval_kernel<R><<<small_grid(n), 256, 0, s>>>(tab, f, kind, t, wx0, wv, n, x, y, z, ux, uy, uz, oE, oB, op, oe, orate);
  count_launch();
}

template <typename R>
void launch_sample(const TabDev<R>& tab, int which, size_t n, const double* param, const double* U, double* out,
                   int32_t* ok, cudaStream_t s) {
  sample_kernel<R><<<small_grid(n), 256, 0, s>>>(tab, which, n, param, U, out, ok);
  count_launch();
}

void launch_philox(size_t n, const uint64_t* ctr, uint64_t k0, uint64_t k1, uint64_t* out, cudaStream_t s) {
  philox_kernel<<<small_grid(n), 256, 0, s>>>(n, ctr, k0, k1, out);
  count_launch();
}

void launch_tau_convert(int precision, double* tau, size_t n, bool to_double, cudaStream_t s) {
  if (precision != QED_MIXED || n == 0) return;
  if (to_double) tau_to_double_kernel<float><<<small_grid(n), 256, 0, s>>>(tau, n);
  else tau_from_double_kernel<float><<<small_grid(n), 256, 0, s>>>(tau, n);
  count_launch();
}

template <typename R>
void launch_compact(const SpeciesDev<R>& sp, const SpeciesDev<R>& out, uint32_t* seg_count, uint32_t* seg_prefix,
                    cudaStream_t s) {
  compact_count_kernel<R><<<sm_count() * 4, 256, 0, s>>>(sp, seg_count);
  compact_scan_kernel<R><<<1, 1024, 0, s>>>(sp, seg_count, seg_prefix);
  compact_scatter_kernel<R><<<sm_count() * 4, 256, 0, s>>>(sp, out, seg_prefix);
  compact_finish_kernel<R><<<1, 1, 0, s>>>(sp, seg_prefix);
  count_launch(4);
}

// ----------------------------------------------------------------------------- weights, merging
template <typename R>
__global__ void fill_kernel(R* p, size_t n, R v) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) p[i] = v;
}

// Per-block FP64 partials of the physical totals: sum w, sum w * energy, sum w * momentum.
template <typename R>
__global__ void __launch_bounds__(256) totals_kernel(const SpeciesDev<R> sp, int massless, double* partials) {
  const uint32_t n = sp.cnt->n;
  double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (massless && Tau<R>::load(sp.tau + i).dead()) continue;
    const double u[3] = {(double)sp.ux[i], (double)sp.uy[i], (double)sp.uz[i]};
    const double w = sp.w ? (double)sp.w[i] : 1.0;
    const double u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    t[0] += w;
    t[1] += w * (massless ? sqrt(u2) : sqrt(1.0 + u2));
    for (int c = 0; c < 3; ++c) t[2 + c] += w * u[c];
  }
  __shared__ double s_t[8][5];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = 0; c < 5; ++c) {
    double v = t[c];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(kFull, v, off);
    if (lane == 0) s_t[warp][c] = v;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double v = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) v += s_t[q][threadIdx.x];
    partials[blockIdx.x * 5 + threadIdx.x] = v;
  }
}

// Group key of a photon for merging, or ~0 when it is not merged: position cell, cube-face
// direction bin and binary-exponent energy bin, from exact operations only (divisions, floor,
// frexp) in double, so that it names the same groups as any other IEEE double implementation.
__device__ uint64_t merge_key_dev(const double x[3], const double k[3], const MergeDev& M) {
  uint64_t cell = 0;
  for (int a = 2; a >= 0; --a) {
    const double c = floor((x[a] - M.origin[a]) / M.cell[a]);
    if (!(c >= 0.0 && c < (double)M.n_cells[a])) return ~0ull;
    cell = cell * (uint64_t)M.n_cells[a] + (uint64_t)c;
  }
  int ax = 0;
  for (int a = 1; a < 3; ++a)
    if (fabs(k[a]) > fabs(k[ax])) ax = a;
  const double m = fabs(k[ax]);
  if (!(m > 0.0)) return ~0ull;
  const int face = 2 * ax + (k[ax] < 0.0 ? 1 : 0);
  int fb[2], q = 0;
  for (int a = 0; a < 3; ++a) {
    if (a == ax) continue;
    int b = (int)floor((k[a] / m + 1.0) * 0.5 * M.n_face);
    b = b < 0 ? 0 : (b >= M.n_face ? M.n_face - 1 : b);
    fb[q++] = b;
  }
  const uint64_t dir = ((uint64_t)face * M.n_face + fb[0]) * M.n_face + fb[1];
  int e2 = 0;
  const double mant = frexp(sqrt(k[0] * k[0] + k[1] * k[1] + k[2] * k[2]), &e2);
  int sub = (int)floor((mant - 0.5) * 2.0 * M.n_sub);
  if (sub >= M.n_sub) sub = M.n_sub - 1;
  const uint64_t en = (uint64_t)(e2 + 1100) * (uint64_t)M.n_sub + (uint64_t)sub;
  return (cell * M.n_dir + dir) * M.n_en + en;  // < M.none
}

// The same key from FP32 arithmetic, for FP32 particles: true where no bin edge is near enough for the
// rounding to matter (the bounds below are several times the worst error), so the bins are those of
// the exact operations.  GB300's FP64 pipe made the exact key of 3e6 photons take 620 us (five
// divisions, a square root and the conversions); with this filter, where about 1 in 1e4 photons
// needs the exact one, it is 30 us.
__device__ __forceinline__ bool sure_floor(float t, float err, int& b) {
  const float f = floorf(t);
  b = (int)f;
  return t - f > err && t - f < 1.0f - err;  // false for NaN and for |t| too large for its fraction
}
__device__ bool merge_key_fast(const float x[3], const float k[3], const MergeDev& M, uint64_t& key) {
  uint64_t cell = 0;
  bool out = false;
#pragma unroll
  for (int a = 2; a >= 0; --a) {
    const float o = (float)M.origin[a], inv = M.inv_cell[a];
    int c;
    if (!sure_floor((x[a] - o) * inv, 1e-6f + 1e-6f * (fabsf(x[a]) + fabsf(o)) * inv, c)) return false;
    out = out || c < 0 || c >= M.n_cells[a];
    cell = cell * (uint64_t)M.n_cells[a] + (uint64_t)(uint32_t)c;
  }
  const float ka[3] = {fabsf(k[0]), fabsf(k[1]), fabsf(k[2])};
  int ax = 0;
  float m = ka[0];
  if (ka[1] > m) { ax = 1; m = ka[1]; }
  if (ka[2] > m) { ax = 2; m = ka[2]; }
  if (!(m > 1e-15f && m < 1e15f)) return false;  // (zero momenta, and squares that would leave the range)
  if (out) { key = ~0ull; return true; }
  const float kx = ax == 0 ? k[0] : (ax == 1 ? k[1] : k[2]);
  const int face = 2 * ax + (kx < 0.0f ? 1 : 0);
  const float im = 1.0f / m, half = 0.5f * (float)M.n_face;
  int fb[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const float v = q == 0 ? (ax == 0 ? k[1] : k[0]) : (ax == 2 ? k[1] : k[2]);
    if (v == 0.0f) {  // exactly the middle
      fb[q] = M.n_face / 2;
    } else {
      if (!sure_floor((v * im + 1.0f) * half, 2e-6f * (float)M.n_face, fb[q])) return false;
      if (fb[q] < 0 || fb[q] >= M.n_face) return false;
    }
  }
  const uint64_t dir = ((uint64_t)face * M.n_face + fb[0]) * M.n_face + fb[1];
  const float e = sqrtf(fmaf(k[0], k[0], fmaf(k[1], k[1], k[2] * k[2])));
  const int bits = __float_as_int(e);
  const int e2 = (bits >> 23) - 126;                                      // e = mant 2^e2, mant in [1/2, 1)
  const float mant = __int_as_float((bits & 0x7fffff) | 0x3f000000);
  int sub;
  const float n_sub = (float)M.n_sub;
  if (!sure_floor((mant - 0.5f) * 2.0f * n_sub, 2e-6f * n_sub, sub)) return false;  // (power-of-two edges among them)
  const uint64_t en = (uint64_t)(e2 + 1100) * (uint64_t)M.n_sub + (uint64_t)sub;
  key = (cell * M.n_dir + dir) * M.n_en + en;
  return true;
}

template <typename R, typename K>
__global__ void merge_key_kernel(const SpeciesDev<R> sp, MergeDev M, K* keys, uint32_t* idx, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint64_t key = ~0ull;
    if (!Tau<R>::load(sp.tau + i).dead()) {
      bool sure = false;
      if constexpr (sizeof(R) == 4) {
        const float x[3] = {sp.x[i], sp.y[i], sp.z[i]}, k[3] = {sp.ux[i], sp.uy[i], sp.uz[i]};
        sure = merge_key_fast(x, k, M, key);
      }
      if (!sure) {
        const double x[3] = {(double)sp.x[i], (double)sp.y[i], (double)sp.z[i]};
        const double k[3] = {(double)sp.ux[i], (double)sp.uy[i], (double)sp.uz[i]};
        key = merge_key_dev(x, k, M);
      }
    }
    keys[i] = key == ~0ull ? (K)M.none : (K)key;
    idx[i] = i;
  }
}

// ----------------------------------------------------------------------------- radix sort
// Stable sort of (key, index) pairs by 8 bits at a time, least significant first, so equal keys keep
// their order (by index).  A pass is three launches: digit counts per segment of 4096 pairs, their
// prefixes (one block per digit), and the scatter, which ranks a segment's pairs by warp match and
// per-warp counts.  Memory-bound: a pass reads the keys twice and the indices once and writes both,
// 20 B per pair with 32-bit keys, and the merging bins in use need 29 bits, so 4 passes; the bitonic
// network before it took log2(n)(log2(n)+1)/2 passes of 24 B (253 at 3e6 photons).
constexpr uint32_t kSortItems = 16;                          // pairs per thread
constexpr uint32_t kSortSeg = 256 * kSortItems;
template <typename K>
__device__ __forceinline__ uint32_t digit_of(K key, int shift) { return (uint32_t)(key >> shift) & 255u; }

template <typename K>
__global__ void __launch_bounds__(256) radix_count_kernel(const K* keys, uint32_t n, int shift, uint32_t* hist) {
  __shared__ uint32_t s_h[256];
  s_h[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t first = blockIdx.x * kSortSeg, last = min(n, first + kSortSeg);
  for (uint32_t i = first + threadIdx.x; i < last; i += 256) atomicAdd(&s_h[digit_of(keys[i], shift)], 1u);
  __syncthreads();
  hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = s_h[threadIdx.x];
}

// Block d: exclusive prefixes of digit d's counts over the segments; totals[d] their sum.
__global__ void __launch_bounds__(256) radix_scan_kernel(uint32_t* hist, uint32_t segs, uint32_t* totals) {
  uint32_t* h = hist + (size_t)blockIdx.x * segs;
  uint32_t base = 0;
  for (uint32_t k0 = 0; k0 < segs; k0 += 1024) {
    uint32_t v[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t k = k0 + threadIdx.x * 4 + q;
      v[q] = k < segs ? h[k] : 0u;
      sum += v[q];
    }
    uint32_t tot;
    uint32_t run = base + block_exclusive_scan(sum, &tot);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t k = k0 + threadIdx.x * 4 + q;
      if (k < segs) h[k] = run;
      run += v[q];
    }
    base += tot;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = base;
}

template <typename K>
__global__ void __launch_bounds__(256) radix_scatter_kernel(const K* keys, const uint32_t* idx, K* keys_out,
                                                            uint32_t* idx_out, uint32_t n, int shift, const uint32_t* hist,
                                                            const uint32_t* totals) {
  __shared__ uint32_t s_c[8][256];  // per warp and digit: pairs seen, then where the warp's begin
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int w = 0; w < 8; ++w) s_c[w][threadIdx.x] = 0;
  __syncthreads();
  // warp w takes the segment's pairs [512 w, 512 w + 512), 32 consecutive ones at a time
  const uint32_t first = blockIdx.x * kSortSeg + (uint32_t)warp * (kSortItems * 32u) + (uint32_t)lane;
  K key[kSortItems];
  uint32_t id[kSortItems], rank[kSortItems];
#pragma unroll
  for (uint32_t q = 0; q < kSortItems; ++q) {
    const uint32_t i = first + 32u * q;
    key[q] = i < n ? keys[i] : (K)0;
    id[q] = i < n ? idx[i] : 0u;
  }
#pragma unroll
  for (uint32_t q = 0; q < kSortItems; ++q) {
    const bool in = first + 32u * q < n;
    const uint32_t d = in ? digit_of(key[q], shift) : 256u;
    const unsigned same = __match_any_sync(kFull, d);
    const uint32_t before = in ? s_c[warp][d] : 0u;
    __syncwarp();
    if (in && lane == __ffs(same) - 1) s_c[warp][d] = before + (uint32_t)__popc(same);
    __syncwarp();
    rank[q] = before + (uint32_t)__popc(same & ((1u << lane) - 1u));
  }
  __syncthreads();
  // thread d: where digit d's pairs of each warp begin
  uint32_t run = block_exclusive_scan(totals[threadIdx.x], nullptr) + hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x];
  for (int w = 0; w < 8; ++w) {
    const uint32_t c = s_c[w][threadIdx.x];
    s_c[w][threadIdx.x] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (uint32_t q = 0; q < kSortItems; ++q) {
    if (first + 32u * q >= n) continue;
    const uint32_t o = s_c[warp][digit_of(key[q], shift)] + rank[q];
    keys_out[o] = key[q];
    idx_out[o] = id[q];
  }
}

// ----------------------------------------------------------------------------- merging groups
// First positions of the groups in the sorted order (any order): heads[0 .. *count).
template <typename K>
__global__ void merge_heads_kernel(const K* keys, uint32_t n, K none, uint32_t* heads, uint32_t* count) {
  const int lane = threadIdx.x & 31;
  for (uint32_t p0 = blockIdx.x * blockDim.x; p0 < n; p0 += gridDim.x * blockDim.x) {
    const uint32_t p = p0 + threadIdx.x;
    const bool head = p < n && keys[p] != none && (p == 0 || keys[p - 1] != keys[p]);
    const unsigned m = __ballot_sync(kFull, head);
    if (!m) continue;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(count, (uint32_t)__popc(m));
    base = __shfl_sync(kFull, base, 0);
    if (head) heads[base + (uint32_t)__popc(m & ((1u << lane) - 1u))] = p;
  }
}

// A float as a double by integer operations (conversions share the FP64 pipe); the few that are
// neither zero nor normal are converted (a call, so that nothing converts ahead of the test).
__device__ __noinline__ double widen_rare(float v) { return (double)v; }
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = (uint32_t)__float_as_int(v), e = b & 0x7f800000u;
  if (e == 0x7f800000u || (e == 0u && (b & 0x7fffffffu) != 0u)) return widen_rare(v);
  if (e == 0u) return __hiloint2double((int)b, 0);
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

constexpr int kMergeSums = 8;  // W, E, P[3], X[3]
// One member's share of the group's sums.
template <typename R>
__device__ __forceinline__ void merge_member(const SpeciesDev<R>& sp, uint32_t i, int massless, double v[kMergeSums]) {
  const R w = sp.w ? sp.w[i] : (R)1;
  const double k[3] = {widen(sp.ux[i]), widen(sp.uy[i]), widen(sp.uz[i])};
  const double x[3] = {widen(sp.x[i]), widen(sp.y[i]), widen(sp.z[i])};
  double e2 = k[0] * k[0] + k[1] * k[1] + k[2] * k[2];
  if (!massless) e2 = 1.0 + e2;
  v[0] = 1.0;
  v[1] = sqrt(e2);
#pragma unroll
  for (int c = 0; c < 3; ++c) { v[2 + c] = k[c]; v[5 + c] = x[c]; }
  if (w != (R)1) {  // (unweighted photons: 7 multiplications by one)
    const double wd = widen(w);
    v[0] = wd;
#pragma unroll
    for (int c = 1; c < kMergeSums; ++c) v[c] = wd * v[c];
  }
}
// The group's survivor number `which` (0 or 1), particle i, from the group's sums.
template <typename R>
__device__ void merge_survivor(SpeciesDev<R>& sp, uint32_t i, int which, int massless, const double t[kMergeSums]) {
  const double W = t[0], E = t[1], *P = t + 2, *X = t + 5;
  // both members get energy E/W; massive ones sit on the mass shell, |u|^2 = (E/W)^2 - 1
  const double et = E / W, mv[3] = {P[0] / W, P[1] / W, P[2] / W};
  const double m2 = mv[0] * mv[0] + mv[1] * mv[1] + mv[2] * mv[2];
  const double d2 = (massless ? et * et : et * et - 1.0) - m2;
  const double dl = d2 > 0.0 ? sqrt(d2) : 0.0;
  int ax = 0;
  for (int c = 1; c < 3; ++c)
    if (fabs(mv[c]) < fabs(mv[ax])) ax = c;
  double e[3] = {0.0, 0.0, 0.0};
  e[ax] = 1.0;
  double dv[3] = {mv[1] * e[2] - mv[2] * e[1], mv[2] * e[0] - mv[0] * e[2], mv[0] * e[1] - mv[1] * e[0]};
  const double dn = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
  if (dn > 0.0) {
    for (int c = 0; c < 3; ++c) dv[c] *= dl / dn;
  } else {
    for (int c = 0; c < 3; ++c) dv[c] = 0.0;
    dv[ax] = dl;
  }
  const double sg = which == 0 ? 1.0 : -1.0;
  sp.ux[i] = (R)(mv[0] + sg * dv[0]); sp.uy[i] = (R)(mv[1] + sg * dv[1]); sp.uz[i] = (R)(mv[2] + sg * dv[2]);
  sp.x[i] = (R)(X[0] / W); sp.y[i] = (R)(X[1] / W); sp.z[i] = (R)(X[2] / W);
  if (sp.w) sp.w[i] = (R)(0.5 * W);
}

// Groups of at least min_group photons become two (the two lowest indices) that carry the group's
// weight, momentum and energy; the others become holes (tau = +inf) that compaction removes.  FP64
// species: a warp per group, 32 members at a time, sums in index order (lane c adds sum c of the
// 32), so the results are those of a plain loop.  Mixed: eight lanes per group, each sums its own
// members and the eight are added in a fixed order; groups of more than kMergeBig members, of which
// a few hold most of the photons, are left to merge_big_kernel, a block each.  The mixed path's
// conversions are integer operations (widen), which keeps them off the FP64 pipe.  3e6 photons, 3e4
// groups on GB300: 434 us, and 384 us for the big ones with 2e6 of the photons; the whole merge, with
// its upload, 15.6 -> 1.51 ms.  The FP64 pipe is busy for about half of that (4.6e6 and 4.0e6 warp
// instructions, each 16 cycles of an SM's pipe: 235 and 203 us); the rest is the wait for the members'
// scattered reads (440 MB each from DRAM, 15% of its rate; 12% and 8% of the issue slots used).
constexpr uint32_t kMergeBig = 256;
template <typename R, typename K>
__global__ void __launch_bounds__(128) merge_groups_kernel(SpeciesDev<R> sp, MergeDev M, const K* keys, const uint32_t* idx,
                                                           uint32_t n, const uint32_t* heads, const uint32_t* count,
                                                           uint32_t* big, uint32_t* n_big, int massless,
                                                           unsigned long long* groups) {
  constexpr bool kOrdered = sizeof(R) == 8;
  constexpr int L = kOrdered ? 32 : 8;  // lanes per group
  __shared__ double s_v[kOrdered ? 4 : 1][kMergeSums][33];
  const int lane = threadIdx.x & (L - 1), row = kOrdered ? threadIdx.x >> 5 : 0;
  const unsigned shift = threadIdx.x & (32u - L) & 31u;  // of the group's lanes in a warp's ballot
  const uint32_t nh = *count, stride = gridDim.x * (128u / L);
  uint32_t merged = 0, removed = 0;
  // (the groups of a warp go through their members together)
  for (uint32_t h0 = blockIdx.x * (128u / L) + (threadIdx.x & ~31u) / L; h0 < nh; h0 += stride) {
    const uint32_t h = h0 + (threadIdx.x & 31u) / L;
    bool open = h < nh, whole = open;
    const uint32_t p = open ? heads[h] : 0u;
    const K key = keys[p];
    double acc[kMergeSums];  // ordered: sum `lane` in acc[0]; else the lane's own
#pragma unroll
    for (int c = 0; c < kMergeSums; ++c) acc[c] = 0.0;
    uint32_t size = 0;
    for (uint32_t r = p + (uint32_t)lane; __any_sync(kFull, open); r += L) {
      const bool in = open && r < n && keys[r] == key;
      const unsigned m = __ballot_sync(kFull, in) >> shift;
      const uint32_t here = (uint32_t)__popc(L == 32 ? m : m & ((1u << (L & 31)) - 1u));  // (the members come first)
      size += here;
      if (here < (uint32_t)L) {
        open = false;
        whole = whole && size >= (uint32_t)M.min_group;
      }
      if (!kOrdered && size > kMergeBig) {
        if (whole && lane == 0) big[atomicAdd(n_big, 1u)] = p;
        open = whole = false;
      }
      double v[kMergeSums];
#pragma unroll
      for (int c = 0; c < kMergeSums; ++c) v[c] = 0.0;
      if (in && whole) merge_member<R>(sp, idx[r], massless, v);
      if (kOrdered) {
#pragma unroll
        for (int c = 0; c < kMergeSums; ++c) s_v[row][c][lane] = v[c];
        __syncwarp();
        if (lane < kMergeSums)
          for (uint32_t t = 0; t < here; ++t) acc[0] += s_v[row][lane][t];
        __syncwarp();
      } else {
#pragma unroll
        for (int c = 0; c < kMergeSums; ++c) acc[c] += v[c];
      }
    }
    double t[kMergeSums];
#pragma unroll
    for (int c = 0; c < kMergeSums; ++c) {
      if (kOrdered) {
        t[c] = __shfl_sync(kFull, acc[0], c);
      } else {
        double a = acc[c];
        for (int off = L / 2; off > 0; off >>= 1) a += __shfl_xor_sync(kFull, a, off);
        t[c] = a;
      }
    }
    if (!whole) continue;
    for (uint32_t r = p + 2u + (uint32_t)lane; r < p + size; r += L) Tau<R>::infinite().store(sp.tau + idx[r]);
    ++merged;
    removed += size - 2u;
    if (lane < 2) merge_survivor<R>(sp, idx[p + (uint32_t)lane], lane, massless, t);
  }
  if (lane == 0 && merged) {
    atomicAdd(&sp.cnt->n_dead, removed);
    atomicAdd(groups, (unsigned long long)merged);
  }
}

// The groups of more than kMergeBig members of the mixed path, one block each.
template <typename R, typename K>
__global__ void __launch_bounds__(512) merge_big_kernel(SpeciesDev<R> sp, MergeDev M, const K* keys, const uint32_t* idx,
                                                        uint32_t n, const uint32_t* big, const uint32_t* n_big, int massless,
                                                        unsigned long long* groups) {
  __shared__ uint32_t s_end;
  __shared__ double s_t[16][kMergeSums];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nb = *n_big;
  for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
    const uint32_t p = big[b];
    const K key = keys[p];
    if (warp == 0) {
      // the group's end, 32 probes at a time: keys[lo] belongs to it, keys[hi] (if any) does not
      uint32_t lo = p, hi = n;
      while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 32u) / 33u, q = lo + step * (uint32_t)(lane + 1);
        const uint32_t c = (uint32_t)__popc(__ballot_sync(kFull, q < hi && keys[q] == key));
        if (lo + step * (c + 1u) < hi) hi = lo + step * (c + 1u);
        lo += step * c;
      }
      if (lane == 0) s_end = lo + 1u;
    }
    __syncthreads();
    const uint32_t end = s_end;
    if (end - p < (uint32_t)M.min_group) { __syncthreads(); continue; }
    double acc[kMergeSums];
#pragma unroll
    for (int c = 0; c < kMergeSums; ++c) acc[c] = 0.0;
    for (uint32_t r = p + threadIdx.x; r < end; r += 512u) {
      double v[kMergeSums];
      merge_member<R>(sp, idx[r], massless, v);
#pragma unroll
      for (int c = 0; c < kMergeSums; ++c) acc[c] += v[c];
    }
#pragma unroll
    for (int c = 0; c < kMergeSums; ++c) {
      double a = acc[c];
      for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(kFull, a, off);
      if (lane == 0) s_t[warp][c] = a;
    }
    __syncthreads();  // the sums are there, and every member has been read
    for (uint32_t r = p + 2u + threadIdx.x; r < end; r += 512u) Tau<R>::infinite().store(sp.tau + idx[r]);
    if (threadIdx.x < 2) {
      double t[kMergeSums];
      for (int c = 0; c < kMergeSums; ++c) {
        t[c] = 0.0;
        for (int w = 0; w < 16; ++w) t[c] += s_t[w][c];
      }
      merge_survivor<R>(sp, idx[p + threadIdx.x], (int)threadIdx.x, massless, t);
    }
    if (threadIdx.x == 0) {
      atomicAdd(&sp.cnt->n_dead, end - p - 2u);
      atomicAdd(groups, 1ull);
    }
    __syncthreads();
  }
}

template <typename R>
void launch_fill(R* p, size_t n, R v, cudaStream_t s) {
  if (!n) return;
  fill_kernel<R><<<sm_count() * 4, 256, 0, s>>>(p, n, v);
  count_launch();
}

template <typename R>
void launch_totals(const SpeciesDev<R>& sp, int massless, double* partials, int blocks, cudaStream_t s) {
  totals_kernel<R><<<blocks, 256, 0, s>>>(sp, massless, partials);
  count_launch();
}

// Sorts the n (key, index) pairs of a[0]; returns which of the two buffers holds the result.
template <typename K>
static int radix_sort(K* keys[2], uint32_t* idx[2], uint32_t n, int bits, uint32_t* hist, uint32_t* totals, cudaStream_t s) {
  const uint32_t segs = (n + kSortSeg - 1) / kSortSeg;
  int cur = 0;
  for (int shift = 0; shift < bits; shift += 8, cur ^= 1) {
    radix_count_kernel<K><<<segs, 256, 0, s>>>(keys[cur], n, shift, hist);
    radix_scan_kernel<<<256, 256, 0, s>>>(hist, segs, totals);
    radix_scatter_kernel<K><<<segs, 256, 0, s>>>(keys[cur], idx[cur], keys[cur ^ 1], idx[cur ^ 1], n, shift, hist, totals);
    count_launch(3);
  }
  return cur;
}

template <typename R, typename K>
static void merge_with_keys(const SpeciesDev<R>& sp, const MergeDev& m, const MergeScratch& w, uint32_t n, int massless,
                            unsigned long long* groups, cudaStream_t s) {
  K* keys[2] = {static_cast<K*>(w.keys[0]), static_cast<K*>(w.keys[1])};
  uint32_t* idx[2] = {w.idx[0], w.idx[1]};
  merge_key_kernel<R, K><<<small_grid(n), 256, 0, s>>>(sp, m, keys[0], idx[0], n);
  const int at = radix_sort<K>(keys, idx, n, m.bits, w.hist, w.totals, s);
  uint32_t* heads = idx[at ^ 1];  // the other buffer is free now
  merge_heads_kernel<K><<<small_grid(n), 256, 0, s>>>(keys[at], n, (K)m.none, heads, w.count);
  uint32_t* big = static_cast<uint32_t*>(w.keys[at ^ 1]);  // (so is its keys' buffer)
  merge_groups_kernel<R, K><<<sm_count() * 8, 128, 0, s>>>(sp, m, keys[at], idx[at], n, heads, w.count, big, w.count + 1,
                                                           massless, groups);
  count_launch(3);
  if (sizeof(R) == 4) {
    merge_big_kernel<R, K><<<sm_count() * 2, 512, 0, s>>>(sp, m, keys[at], idx[at], n, big, w.count + 1, massless, groups);
    count_launch();
  }
}

template <typename R>
void launch_merge(const SpeciesDev<R>& sp, const MergeDev& m, const MergeScratch& w, uint32_t n, int massless,
                  unsigned long long* groups, cudaStream_t s) {
  if (m.bits <= 32) merge_with_keys<R, uint32_t>(sp, m, w, n, massless, groups, s);
  else merge_with_keys<R, uint64_t>(sp, m, w, n, massless, groups, s);
}

#endif

#if QED_PART(1)
#define QED_INSTANTIATE_STEP(R)                                                                                  \
  template void launch_step<R>(const StepArgs<R>&, int, int, size_t, cudaStream_t);                              \
  template void launch_finalize<R>(const StepArgs<R>&, int, cudaStream_t);                                       \
  template void launch_ledger<R>(const StepArgs<R>&, int, cudaStream_t);                                         \
  template int launch_fused<R>(const StepArgs<R>&, int, bool, uint32_t*, int, cudaStream_t);
QED_INSTANTIATE_STEP(float)
QED_INSTANTIATE_STEP(double)
#endif
#if QED_PART(2)
template void launch_batch_step<float>(const BatchCtl<float>&, int, int, BatchEnd, int, BatchEnd, int, cudaStream_t);
template void launch_batch_step<double>(const BatchCtl<double>&, int, int, BatchEnd, int, BatchEnd, int, cudaStream_t);
#endif
#if QED_PART(3)
#define QED_INSTANTIATE(R)                                                                                       \
  template void launch_init_tau<R>(const SpeciesDev<R>&, int, uint64_t, uint64_t, cudaStream_t);                 \
  template void launch_eval<R>(const TabDev<R>&, const FieldDev&, int, double, double, double, size_t,           \
                               const double*, const double*, const double*, const double*, const double*,        \
                               const double*, double*, double*, double*, double*, double*, cudaStream_t);        \
  template void launch_sample<R>(const TabDev<R>&, int, size_t, const double*, const double*, double*, int32_t*, \
                                 cudaStream_t);                                                                  \
  template void launch_compact<R>(const SpeciesDev<R>&, const SpeciesDev<R>&, uint32_t*, uint32_t*, cudaStream_t); \
  template void launch_fill<R>(R*, size_t, R, cudaStream_t);                                                     \
  template void launch_totals<R>(const SpeciesDev<R>&, int, double*, int, cudaStream_t);                         \
  template void launch_merge<R>(const SpeciesDev<R>&, const MergeDev&, const MergeScratch&, uint32_t, int,         \
                                unsigned long long*, cudaStream_t);
QED_INSTANTIATE(float)
QED_INSTANTIATE(double)
#endif

}  // namespace qedlib
