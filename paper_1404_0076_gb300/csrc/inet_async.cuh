// Asynchronous driver of the reduction loop: the same interaction (Sec. 2.2,
// ->int), allocation and linking (->com) as the step kernels, but without
// steps.  Active pairs are independent (Sec. 2.1: reducing one cannot
// affect another), so nothing forces all pairs of a "loop iteration" to
// finish before the next begins: every warp of one cooperative launch loops
// on its own, each lane holding at most one active pair.  An interaction
// that creates active pairs keeps the first as the lane's next pair (and
// starts loading its records at once), so a sequential chain of
// interactions never leaves its lane; further pairs go to idle lanes of the
// same warp, and the rest to a FIFO of tickets that idle lanes claim: a
// bounded ring whose cells carry a 64-bit sequence number each, so that a
// producer and a consumer of the same cell in different laps can never be
// confused.  The loop ends when no active pair is left anywhere (the count
// of pairs in flight reaches zero), as in Sec. 3.6; a time slice or an error
// instead drains every pair back to a frontier buffer so that the host can
// resume.
//
// Ordering without barriers: a lane writes its new agent records and fresh
// names, then one fence, then the exchanges on name slots that publish
// references to them; the queue publishes a cell with a release store of its
// sequence and is read with an acquire load; pairs handed to lanes of the
// same warp pass through shared memory and __syncwarp.  A lane that learns
// of an agent through an exchange loads its record only after the exchange
// returned (address dependency), so it sees the record written before the
// fence.
//
// kTrack (contexts created with INET_ARENA_FREE_NETS): the kernel also keeps
// what inet_free_nets scans for: the owning net of every name it creates,
// the free mark of every agent slot it frees, and both marks on the unused
// slots its warps return at the end.  The other instantiation has none of
// that code in its loop (code the loop does not run still costs this kernel
// time through instruction fetch and scheduling).
//
// Rules (a rule set known when the kernel is compiled, see inet_jit.h): the
// library compiles k_async<kTrack, Rules> at run time for the loaded rule
// set; each lane then runs its own rule's straight-line code (one_step), and
// a rule that repeats itself along a list many interactions at a time
// (run_rule, pass_rule, end_run).  NoRules is the general kernel built with
// the library, which interprets the templates.
//
// What bounds the loop is latency: of a warp's turn (load, slots, rules,
// fence, exchanges, hand-on; 8 000 to 50 000 cycles) and of the dependent
// loads inside a run.  The design follows from that: many interactions per
// turn where a rule allows it, one fence for the whole warp, nothing between
// lanes but the hand-on.  With one interaction per turn / now: 2048 Mul nets
// 9.9 / 4.4 ms, Ackermann(3, 4..8) 66 / 45 ms, Fibonacci(20..25) 81 / 17.4 ms,
// 16 x Fibonacci(25) 93 / 23 ms, a chain of 20 000 Add 27 / 2.2 ms, 512 trees
// 1.5 / 1.1 ms, L-System(13) and (22) 0.20 / 0.20 and 0.43 / 0.42 ms.  The
// figures at the constants below are of the same batches.
#pragma once

#include "inet_kernels.cuh"

namespace inet {

constexpr int kVRes = 8;       // free name slots a lane keeps for itself
// Slots of each kind a lane keeps of those it frees; the rest is the warp's.
// 2048 Mul nets 4.5 ms with 2, 4.4 with 4; 4.3 with 8, which holds twice as many
// back from the others.
constexpr int kKeep = 4;
// Interactions after which a run ends (pass_rule looks once a block of 4; a rule
// that ends the list adds one): of a warp's only lane, of one lane among
// several, and where most of the warp's lanes reduce rules that do not run and
// wait for the run.  Lone: the chain 2.2 ms, 3.1 with 64.  Among several, with
// 32 / 64 / 128: 2048 Mul nets 4.9 / 4.4 / 5.1, Fibonacci 19.8 / 17.4 / 16.6,
// trees 1.06 / 1.12 / 1.29.  Mixed: trees 1.12 ms, 1.17 with 64.
constexpr uint32_t kRunLone = 512, kRunMany = 64, kRunMixed = 16;
constexpr unsigned long long kNoTicket = ~0ull;
// Slots fetched beyond the need when a warp's stack runs dry (two L2 round
// trips): L-System(19) 0.30 ms, 0.33 with half as many.
constexpr uint32_t kFetchA = 64, kFetchV = 32;

// Shared memory of one warp.  kTable: with the value table of the general
// kernel, which interprets every rule.
template <bool kTable>
struct ValueTable {
  static constexpr bool kHasTable = false;
};
template <>
struct ValueTable<true> {
  static constexpr bool kHasTable = true;
  uint32_t vals[kNumVals][32];   // a column per lane
};
template <bool kTable>
struct alignas(16) WarpMem : ValueTable<kTable> {
  // Agent slots of a lane, agents and names of the warp's stack.  A column of 16
  // lets a run of Dup go on for 16 copies and lays them out side by side.  The
  // general kernel has no runs: what one step of the warp can need.
  static constexpr int kARes = kTable ? 8 : 16, kAStack = kTable ? 192 : 576, kVStack = kTable ? 256 : 288;
  static_assert(kARes >= kMaxNew - 2 && kVRes >= kMaxFresh, "a lane's slots serve any one interaction");
  static_assert(kAStack >= 32 * (kTable ? kMaxNew - 2 : kARes) && kVStack >= 32 * kVRes, "a warp's stacks serve any one step");
  uint32_t ares[kARes][32];      // lane-private free slots, a column per lane
  uint32_t vres[kVRes][32];
  Pair out[kMaxLink][32];        // new active pairs of one step
  union {
    uint2 eq[kMaxLink][32];        // equations of one step left to link after the fence
    Pair xl[(kMaxLink - 1) * 32];  // extra pairs of one iteration, in lane order
  };
  uint32_t astk[kAStack];
  uint32_t vstk[kVStack];
  int an, vn, pad[2];            // entries of the warp's stacks (above the size: pushes that went to the ring)
};

__host__ __device__ constexpr size_t async_smem_bytes(uint32_t block, uint32_t n_labels, uint32_t n_tmpl, bool table) {
  size_t b = 0;
  auto take = [&](size_t n, size_t align) { b = (b + align - 1) / align * align; b += n; };
  take(sizeof(PackedTpl) * (n_tmpl ? n_tmpl : 1), 16);
  take((table ? sizeof(WarpMem<true>) : sizeof(WarpMem<false>)) * (block / 32), 16);
  take(sizeof(uint32_t) * INET_MAX_RULES, 16);
  take(sizeof(int16_t) * n_labels * n_labels, 16);
  return b + 16;
}
// Two blocks share an SM whatever the rule set: the general kernel's batch of
// 2048 Mul nets takes 12.9 ms under 64 rules and 57 symbols, as under the 18
// alone, where one block an SM took 16.8 (and 13.8 two that leave L1 only 28 of
// the 256 KB, hence 97 KB).  Each block takes 1 KB besides its own.
static_assert(async_smem_bytes(256, kMaxLabels, INET_MAX_RULES, true) <= 97 * 1024 &&
              async_smem_bytes(256, kMaxLabels, INET_MAX_RULES, false) <= 113 * 1024, "two blocks per SM");

__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Ticket queue: ticket t lives in cell t % cap, whose sequence number
// moves t -> t + 1 (the producer wrote the pair) -> t + cap (the consumer
// took it, so the cell is free for ticket t + cap).  A producer writes only
// when the sequence equals its own ticket, a consumer takes only at its
// ticket + 1; both compare all 64 bits, so no lap can be mistaken for
// another however far ahead tickets were claimed.

// Free slots.  A lane takes the slots of its interactions from a private
// column of the warp's shared memory and puts the slots it frees back there,
// so that lanes reducing different rules, or runs of different lengths, need
// no agreement; what does not fit goes to the warp's stack, then to the ring.
// Only refill() moves slots into the columns, for all lanes of the warp at
// once.
struct Lane {
  int na, nv;       // slots in this lane's columns
  long long live;   // change of live agents by this lane
};

// What a lane does not keep of the slots it frees: to the warp's stack, else
// to the ring.  Out of line, like the other rare paths here: the kernel holds
// a copy of the common path for every rule, and its size counts (instruction
// cache).
template <class WM>
__device__ __noinline__ void spill_agent(const Dev& d, WM& W, uint32_t slot) {
  const int pos = atomicAdd(&W.an, 1);
  if (pos < WM::kAStack) {
    W.astk[pos] = slot;
  } else {
    const unsigned long long tp = atomicAdd(&d.ctrl->a_tail, 1ull);
    __stcg(d.afree + tp % d.cap_agents, slot);
  }
}
template <class WM>
__device__ __noinline__ void spill_name(const Dev& d, WM& W, uint32_t x) {
  const int pos = atomicAdd(&W.vn, 1);
  if (pos < WM::kVStack) {
    W.vstk[pos] = x;
  } else {
    const unsigned long long tp = atomicAdd(&d.ctrl->v_tail, 1ull);
    __stcg(d.vfree + tp % d.cap_vars, x);
  }
}
__device__ __noinline__ void report(const Dev& d, int32_t code, uint32_t info) { set_error(d.ctrl, code, info); }

template <bool kTrack, class WM>
__device__ __forceinline__ void put_agent(const Dev& d, WM& W, Lane& L, int lane, uint32_t slot) {
  if constexpr (kTrack) __stcg(&d.node[slot].head, kFreeHead);
  if (L.na < kKeep) W.ares[L.na++][lane] = slot;
  else spill_agent(d, W, slot);
}

// A second arrival at name slot x: the slot is finished (its owner mark
// cleared) and free again.
template <bool kTrack, class WM>
__device__ __forceinline__ void release_name(const Dev& d, WM& W, Lane& L, int lane, uint32_t x) {
  __stcg(d.var + x, kEmpty);
  if constexpr (kTrack) __stcg(d.vown + x, kNoNet);
  if (L.nv < kKeep) W.vres[L.nv++][lane] = x;
  else spill_name(d, W, x);
}

template <class WM>
__device__ __forceinline__ uint32_t take_agent(const WM& W, Lane& L, int lane) { return W.ares[--L.na][lane]; }

// A free name slot is empty: never used, or cleared when it was released
// (by a lane of this warp, or before this launch), so nothing is stored here.
template <bool kTrack, class WM>
__device__ __forceinline__ uint32_t take_name(const Dev& d, const WM& W, Lane& L, int lane, uint32_t net) {
  const uint32_t x = W.vres[--L.nv][lane];
  if constexpr (kTrack) __stcg(d.vown + x, net);
  return x;
}

// One pop of the global pools for the warp's stacks (ac agents, vc names
// now): up to Ka and Kv and a few more, but no more than a warp's share of
// half of what is left, in the ring of recycled slots and above the bump
// pointer together, so that no warp starves the others, and from the bump
// pointer no more than a share of its own room; but at least what one step
// needs (Ma, Mv), and no more agents than that once a share is below 32, when
// what warps keep for later is what the nets lack (256 Mul nets then reduce
// over and over in 1.06 times their peak, else in 1.12).  With a share of the
// bump pointer's room alone, every pop of a context that runs on recycled slots
// was a bare step's need: 2048 Mul nets loaded, reduced and freed over and over
// in 1.1 times their peak 9.0 ms, now 5.5.  Returns false when the arena is full
// (fatal: the loop stops).  Warp-collective.
template <class WM>
__device__ __noinline__ bool fill_stacks(const Dev& d, WM& W, uint32_t ac, uint32_t vc, uint32_t Ka, uint32_t Kv,
                                         uint32_t Ma, uint32_t Mv) {
  Ctrl* c = d.ctrl;
  const int lane = threadIdx.x & 31;
  // lane 0 serves the agents, lane 1 the names: their counters in one load
  const unsigned long long* p = lane == 0 ? &c->a_head : lane == 1 ? &c->v_head : lane == 2 ? &c->a_pub
                              : lane == 3 ? &c->v_pub : lane == 4 ? &c->a_bump : &c->v_bump;
  unsigned long long cnt = 0;
  if (lane < 6) cnt = ld_volatile64(p);
  const unsigned long long pub = __shfl_down_sync(kFull, cnt, 2), bump = __shfl_down_sync(kFull, cnt, 4);
  const unsigned long long cap = lane == 0 ? d.cap_agents : d.cap_vars;
  const uint32_t have = lane == 0 ? ac : vc, want = lane == 0 ? Ka : Kv, least = lane == 0 ? Ma : Mv;
  const uint32_t size = lane == 0 ? (uint32_t)WM::kAStack : (uint32_t)WM::kVStack;
  uint32_t ok = 1, av = 0, k = 0;
  unsigned long long rb = 0, bb = 0;
  if (lane < 2 && want > have) {
    const unsigned long long room = bump < cap ? cap - bump : 0ull;
    const unsigned long long ring = cnt < pub ? pub - cnt : 0ull;  // a ring seen empty is left alone
    const unsigned long long shares = 2ull * gridDim.x * (blockDim.x / 32);
    const uint32_t need = least > have ? least - have : 0u;
    k = want - have + (lane == 0 ? kFetchA : kFetchV);
    if (ring + room < k * shares) {
      const uint32_t share = (uint32_t)((ring + room) / shares);
      k = lane == 0 && share < 32 ? need : max(share, need);
    }
    k = min(k, size - have);
    if (k && ring) {
      const unsigned long long h = atomicAdd(lane == 0 ? &c->a_head : &c->v_head, (unsigned long long)k);
      av = h < pub ? (uint32_t)min((unsigned long long)k, pub - h) : 0u;
      rb = h % cap;
    }
    uint32_t u = k - av;
    if (room < u * shares) u = max((uint32_t)(room / shares), need > av ? need - av : 0u);
    if (u) {
      bb = atomicAdd(lane == 0 ? &c->a_bump : &c->v_bump, (unsigned long long)u);
      if (bb + u > cap) {
        ok = 0;
        set_error(c, INET_ERR_ARENA_FULL, 0);
      }
    }
    k = av + u;
  }
  if (!__all_sync(kFull, ok)) return false;
  // on top of the stacks, the lowest slot last, so that slots from the bump
  // pointer are taken in ascending order
#pragma unroll 1
  for (int w = 0; w < 2; w++) {
    const uint32_t n = __shfl_sync(kFull, k, w), a = __shfl_sync(kFull, av, w), h = __shfl_sync(kFull, have, w);
    const unsigned long long r = __shfl_sync(kFull, rb, w), u = __shfl_sync(kFull, bb, w);
    const unsigned long long cp = __shfl_sync(kFull, cap, w);
#pragma unroll 1
    for (uint32_t j = (uint32_t)lane; j < n; j += 32) {
      uint32_t sl = pool_slot(w ? d.vfree : d.afree, cp, r, a, u, j);
      if (sl >= cp) {
        set_error(c, INET_ERR_STATE, 4);
        sl = 0;
      }
      (w ? W.vstk : W.astk)[h + n - 1 - j] = sl;
    }
    if (lane == 0) (w ? W.vn : W.an) = (int)(h + n);
  }
  __syncwarp();
  return true;
}

// Slots for the lanes that lack some for their next interaction (need_a
// agents, need_v names, 0 for the others; runs: the rule is reduced in runs;
// more: what a lane of another rule takes at least), from the warp's stacks into
// the lanes' columns.  Returns false when the arena is full.  Warp-collective.
template <class WM>
__device__ __forceinline__ bool refill(const Dev& d, WM& W, Lane& L, bool runs, uint32_t more, uint32_t need_a,
                                       uint32_t need_v, int lane) {
  __syncwarp();
  uint32_t ac = (uint32_t)min(W.an, WM::kAStack), vc = (uint32_t)min(W.vn, WM::kVStack);
  // what the step needs, and for a run a whole column and 4 names (with 2, runs
  // of Dup and Mul stop for lack of them: 2048 Mul nets 5.5 ms instead of 4.4)
  const uint32_t least_a = (uint32_t)L.na < need_a ? need_a - (uint32_t)L.na : 0u;
  const uint32_t least_v = (uint32_t)L.nv < need_v ? need_v - (uint32_t)L.nv : 0u;
  uint32_t wa = least_a ? (runs ? (uint32_t)WM::kARes : max(need_a, more)) - (uint32_t)L.na : 0u;
  uint32_t wv = least_v ? max(need_v, runs ? 4u : more) - (uint32_t)L.nv : 0u;
  uint32_t inc, packed, Ka, Kv;
  // offsets of this lane among the warp's wants
  auto scan = [&]() {
    packed = inc = wa | (wv << 16);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += t;
    }
    const uint32_t tot = __shfl_sync(kFull, inc, 31);
    Ka = tot & 0xFFFFu;
    Kv = tot >> 16;
  };
  scan();
  if (Ka > ac || Kv > vc) {
    // what lanes with no use for them now keep from an earlier run goes back
    // to the warp before the pools are asked
    const uint32_t ga = need_a == 0 && L.na > kKeep ? (uint32_t)(L.na - kKeep) : 0u;
    const uint32_t gv = need_v == 0 && L.nv > kKeep ? (uint32_t)(L.nv - kKeep) : 0u;
    if (__any_sync(kFull, (ga | gv) != 0)) {
      uint32_t g = ga | (gv << 16);
      const uint32_t own = g;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFull, g, o);
        if (lane >= o) g += t;
      }
      const uint32_t at_a = ac + ((g - own) & 0xFFFFu), at_v = vc + ((g - own) >> 16);
      uint32_t da = 0, dv = 0;
#pragma unroll 1
      for (; da < ga && at_a + da < (uint32_t)WM::kAStack; da++) W.astk[at_a + da] = W.ares[--L.na][lane];
#pragma unroll 1
      for (; dv < gv && at_v + dv < (uint32_t)WM::kVStack; dv++) W.vstk[at_v + dv] = W.vres[--L.nv][lane];
      const uint32_t tot = __shfl_sync(kFull, g, 31);
      ac = min(ac + (tot & 0xFFFFu), (uint32_t)WM::kAStack);
      vc = min(vc + (tot >> 16), (uint32_t)WM::kVStack);
      __syncwarp();
    }
  }
  if (Ka > ac || Kv > vc) {
    const uint32_t Ma = __reduce_add_sync(kFull, least_a), Mv = __reduce_add_sync(kFull, least_v);
    if (!fill_stacks(d, W, ac, vc, Ka, Kv, Ma, Mv)) return false;
    ac = (uint32_t)min(W.an, WM::kAStack);
    vc = (uint32_t)min(W.vn, WM::kVStack);
    if (Ka > ac || Kv > vc) {
      wa = least_a;
      wv = least_v;
      scan();
    }
  }
  const uint32_t oa = ac - ((inc - packed) & 0xFFFFu), ov = vc - ((inc - packed) >> 16);
#pragma unroll 1
  for (uint32_t k = 0; k < wa; k++) W.ares[L.na + (int)(wa - 1 - k)][lane] = W.astk[oa - 1 - k];
#pragma unroll 1
  for (uint32_t k = 0; k < wv; k++) W.vres[L.nv + (int)(wv - 1 - k)][lane] = W.vstk[ov - 1 - k];
  L.na += (int)wa;
  L.nv += (int)wv;
  __syncwarp();
  if (lane == 0) {
    W.an = (int)(ac - Ka);
    W.vn = (int)(vc - Kv);
  }
  __syncwarp();
  return true;
}

// ->com for the asynchronous kernel (the chase after a second arrival):
// link_eq with freed name slots kept by the lane.  The lane has fenced its
// new records before linking; a lane that receives a reference through an
// exchange loads the referenced record only after the exchange returned
// (address dependency), so it sees the record written before the fence.
template <bool kTrack, class WM>
__device__ __forceinline__ bool link_async(const Dev& d, WM& W, Lane& L, int lane, uint32_t t, uint32_t u,
                                           Pair* out) {
#pragma unroll 1
  for (uint32_t guard = 0;; guard++) {
    if (is_agent(t) && is_agent(u)) {
      out->a = idx_of(t);
      out->b = idx_of(u);
      return true;
    }
    if (!is_var(t)) {
      uint32_t w = t;
      t = u;
      u = w;
    }
    if (!is_var(t) || guard > (1u << 24) || idx_of(t) >= d.cap_vars) {
      report(d, INET_ERR_STATE, 1);
      return false;
    }
    const uint32_t x = idx_of(t);
    const uint32_t old = atomicExch(d.var + x, u);
    if (old == kEmpty) return false;
    release_name<kTrack>(d, W, L, lane, x);
    t = old;
  }
}

// What one lane's step leaves: new active pairs in W.out[0 .. np)[lane],
// equations to link after the fence in W.eq[0 .. ne)[lane], how many times
// the rule was applied, and, when fwd is set, the records of pair 0 (ra always,
// rb when have_b).
struct Step {
  uint32_t np, ne, steps;
  bool fwd, have_b;
  int fin;          // rule that ended a run inside it, -1: none
  int4 ra, rb;
};

// One equation of Theta': two agents are an active pair at once, anything
// else waits for the fence.
template <class WM>
__device__ __forceinline__ void put_equation(WM& W, Step& S, int lane, uint32_t t, uint32_t u) {
  const bool pair = is_agent(t) && is_agent(u);
  uint2* to = pair ? reinterpret_cast<uint2*>(&W.out[S.np][lane]) : &W.eq[S.ne][lane];
  *to = pair ? make_uint2(idx_of(t), idx_of(u)) : make_uint2(t, u);
  S.np += pair ? 1u : 0u;
  S.ne += pair ? 0u : 1u;
}

// ->com of one lane's equations left by its step, after the fence (which
// makes its new records and fresh names visible before an exchange can
// publish a reference to them): the first exchange of each of the first
// kBatch equations is issued back to back, and only second arrivals continue
// (rarely) with a chase.
template <bool kTrack, class WM>
__device__ __forceinline__ void link_lane(const Dev& d, WM& W, Lane& L, Step& S, int lane) {
  constexpr uint32_t kBatch = 3;
  uint32_t lt[kBatch], lu[kBatch], lo[kBatch];
  bool more = S.ne > kBatch;
  uint32_t pend = S.ne > kBatch ? ~0u << kBatch : 0u;  // equations still to chase
#pragma unroll
  for (uint32_t k = 0; k < kBatch; k++) {
    lt[k] = lu[k] = 0;
    lo[k] = kEmpty;
    if (k < S.ne) {
      const uint2 e = W.eq[k][lane];
      uint32_t t = e.x, u = e.y;
      if (!is_var(t)) {
        const uint32_t w = t;
        t = u;
        u = w;
      }
      if (is_var(t) && idx_of(t) < d.cap_vars) lo[k] = atomicExch(d.var + idx_of(t), u);
      else report(d, INET_ERR_STATE, 1);
      lt[k] = t;
      lu[k] = u;
    }
  }
#pragma unroll
  for (uint32_t k = 0; k < kBatch; k++) {
    if (k < S.ne && lo[k] != kEmpty) {
      // second arrival: the slot is finished; continue with old = u
      release_name<kTrack>(d, W, L, lane, idx_of(lt[k]));
      const uint32_t t = lo[k], u = lu[k];
      if (is_agent(t) && is_agent(u)) {
        W.out[S.np][lane] = Pair{idx_of(t), idx_of(u)};
        S.np++;
      } else {
        more = true;
        W.eq[k][lane] = make_uint2(t, u);
        pend |= 1u << k;
      }
    }
  }
  if (more) {
#pragma unroll 1
    for (uint32_t k = 0; k < S.ne; k++) {
      if (!((pend >> k) & 1u)) continue;
      const uint2 e = W.eq[k][lane];
      Pair out;
      if (link_async<kTrack>(d, W, L, lane, e.x, e.y, &out)) {
        W.out[S.np][lane] = out;
        S.np++;
      }
    }
  }
}

// The rule set a kernel is specialised for: kN templates known at compile
// time (kT, in rule-table order, some with active pairs of their own
// right-hand side already reduced: kMore[I] = how many, and by which rules)
// and kKey, the hash of the loaded templates that the host passes in
// Dev::rules_key.  NoRules (kN = 0): the general kernel, which
// reads the templates from shared memory.
struct NoRules {
  static constexpr int kN = 0;
  static constexpr unsigned long long kKey = 0;
  static constexpr Template kT[1] = {};
  static constexpr unsigned char kMore[1][3] = {{0, 0, 0}};
};

// At most this many rules get their own code (the first in rule-table
// order): every one adds to the run-time compile and to the kernel's code;
// the others are interpreted.
constexpr int kSpecialisedMaxRules = 32;

// How rule I repeats itself along a list.  A rule does when one equation of
// its right-hand side joins a new agent of one of its own left-hand side's
// symbols (the walker, new agent jc, side cs) to a port e of the other agent
// (Add(y, w) = x of Add(y, r) = S(x) -> Add(y, w) = x, r = S(w): the walker
// Add goes on to whatever x is), and every other equation is the head of an
// output stream: a walker's port p is one when its new value is a fresh name
// whose other occurrence is port q of another new agent js, and the
// remaining equation kl joins that agent to the walker's old port p
// (r = S(w) with w in the walker's port).  Along a list of k such partners
// the streams then spell js(js(..js(w)..)), with the names between two steps
// seen by nobody but the lane that reduces them.  Both sides may qualify (S
// is a walker along the chain of adders that r leads to): the symbol written
// first on the left-hand side is taken, by custom the one that does the
// walking.
struct ChainInfo {
  bool ok = false;
  int kc = 0, jc = 0, e = 0, cs = 0;
  int js[3] = {-1, -1, -1}, q[3] = {0, 0, 0};
  int other = -1;                           // the new agent that takes the partner's slot, -1: none
  bool same[3] = {false, false, false};     // js is the partner again, in its slot, but for port q
};
__host__ __device__ constexpr ChainInfo chain_info(const Template& R) {
  ChainInfo none;
  for (int cand = 0; cand < 2 * R.n_link; cand++) {
    const int kc = cand % R.n_link;
    const int c0 = R.link[kc][0], c1 = R.link[kc][1];
    const bool e0 = c0 < kValNew, e1 = c1 < kValNew;
    if (e0 == e1) continue;
    ChainInfo C;
    C.kc = kc;
    C.e = e0 ? c0 : c1;
    C.jc = (e0 ? c1 : c0) - kValNew;
    if (R.lab[C.jc] != R.lhs[0] && R.lab[C.jc] != R.lhs[1]) continue;
    C.cs = R.lab[C.jc] == R.lhs[0] ? 0 : 1;
    if (C.cs != cand / R.n_link || C.e / 3 == C.cs) continue;
    int heads = 0;
    for (int p = 0; p < 3; p++) {
      const int f = R.src[C.jc][p];
      if (f < kValFresh || f == kValNone) continue;
      for (int j = 0; j < R.n_new; j++)
        for (int q = 0; q < 3; q++) {
          if (j == C.jc || R.src[j][q] != f) continue;
          for (int k = 0; k < R.n_link; k++) {
            const int a = R.link[k][0], b = R.link[k][1];
            const int ext = kValExt + C.cs * 3 + p, agent = kValNew + j;
            if ((a == ext && b == agent) || (a == agent && b == ext)) {
              C.js[p] = j;
              C.q[p] = q;
              heads++;
            }
          }
        }
    }
    if (heads != R.n_link - 1 || (C.cs == 1 && heads == 0)) continue;
    for (int j = R.n_new - 1; j >= 0; j--)
      if (j != C.jc) C.other = j;
    for (int p = 0; p < 3; p++) {
      if (C.js[p] < 0) continue;
      const int ps = 1 - C.cs;
      bool same = C.js[p] == C.other && R.lab[C.js[p]] == R.lhs[ps];
      for (int r = 0; r < 3; r++) {
        if (r == C.q[p]) continue;
        const int c = R.src[C.js[p]][r];
        if (c != kValNone && c != kValExt + ps * 3 + r) same = false;
      }
      C.same[p] = same;
    }
    C.ok = true;
    return C;
  }
  return none;
}

// Ports of the left-hand side's agent `side` (each is used once on the
// right-hand side).
__host__ __device__ constexpr int chain_arity(const Template& R, int side) {
  int n = 0;
  for (int j = 0; j < R.n_new; j++)
    for (int p = 0; p < 3; p++)
      if (R.src[j][p] < kValNew && R.src[j][p] / 3 == side) n++;
  for (int k = 0; k < R.n_link; k++)
    for (int i = 0; i < 2; i++)
      if (R.link[k][i] < kValNew && R.link[k][i] / 3 == side) n++;
  return n;
}
// The record of a partner, or its first half when that is all it holds.
template <bool kNarrow>
__device__ __forceinline__ int4 ld_partner(const Node* p) {
  if constexpr (kNarrow) {
    const uint2 v = __ldcg(reinterpret_cast<const uint2*>(p));
    return make_int4((int)v.x, (int)v.y, 0, 0);
  } else {
    return ld_node(p);
  }
}

// The walker leaves every partner of a run in its slot as it is: one output
// stream, of the partners themselves, no other new agent, the walker's other
// ports unchanged.
__host__ __device__ constexpr bool chain_passes(const Template& R, const ChainInfo& C) {
  if (!C.ok || R.n_new != 2 || R.n_fresh != 1) return false;
  for (int p = 0; p < 3; p++) {
    if (C.js[p] >= 0) {
      if (!C.same[p] || C.q[p] != C.e % 3) return false;
    } else if (R.src[C.jc][p] != kValNone && R.src[C.jc][p] != kValExt + C.cs * 3 + p) {
      return false;
    }
  }
  return true;
}

// Component q of a record's auxiliary words (q is a constant where it is used).
__device__ __forceinline__ void set_aux(int4& r, int q, uint32_t w) {
  if (q == 0) r.y = (int32_t)w;
  else if (q == 1) r.z = (int32_t)w;
  else r.w = (int32_t)w;
}
__device__ __forceinline__ uint32_t get_aux(const int4& r, int q) {
  return (uint32_t)(q == 0 ? r.y : q == 1 ? r.z : r.w);
}

// Rule I of a specialised rule set for one lane (Sec. 2.2, ->int): the
// template is a constant, so the values live in registers and every loop
// over agents, ports, names and equations is unrolled.  Records are stored,
// equations are left for the fence that the whole warp shares.
template <bool kTrack, class Rules, int I, class WM>
__device__ __forceinline__ void one_step(const Dev& d, WM& W, Lane& L, int lane, uint32_t a, uint32_t b,
                                         const int4& ra, const int4& rb, uint32_t net, Step& S) {
  constexpr Template R = Rules::kT[I];
  uint32_t v[kNumVals];
#pragma unroll
  for (int q = 0; q < 3; q++) {
    v[kValExt + q] = get_aux(ra, q);
    v[kValExt + 3 + q] = get_aux(rb, q);
  }
#pragma unroll
  for (int j = kValNew; j < kNumVals; j++) v[j] = 0;
  if (R.n_new > 0) v[kValNew + 0] = mk_agent(a);
  if (R.n_new > 1) v[kValNew + 1] = mk_agent(b);
#pragma unroll
  for (int j = 2; j < (int)R.n_new; j++) v[kValNew + j] = mk_agent(take_agent(W, L, lane));
#pragma unroll
  for (int f = 0; f < (int)R.n_fresh; f++) v[kValFresh + f] = mk_var(take_name<kTrack>(d, W, L, lane, net));
#pragma unroll
  for (int j = 0; j < (int)R.n_new; j++) {
    int4 rec;
    rec.x = (int32_t)((net << 8) | R.lab[j]);
    rec.y = R.src[j][0] == kValNone ? 0 : (int32_t)v[R.src[j][0]];
    rec.z = R.src[j][1] == kValNone ? 0 : (int32_t)v[R.src[j][1]];
    rec.w = R.src[j][2] == kValNone ? 0 : (int32_t)v[R.src[j][2]];
    st_node(d.node + idx_of(v[kValNew + j]), rec);
  }
  if (R.n_new == 0) put_agent<kTrack>(d, W, L, lane, a);
  if (R.n_new < 2) put_agent<kTrack>(d, W, L, lane, b);
  L.live += (int)R.n_new - 2;
  S.steps = 1;
#pragma unroll
  for (int k = 0; k < (int)R.n_link; k++) put_equation(W, S, lane, v[R.link[k][0]], v[R.link[k][1]]);
}

// Rule J can end a run of rule I inside it: the walker meets an agent that
// the list ends with (Add(y, r) = Z -> r = y after Add(y, r) = S(x)), and J
// joins each of the run's output streams to something it has at hand, which
// then goes straight into the open port of the stream's last agent.  That
// saves a name, the walker's record and a whole step at every list's end, and
// leaves lists with fewer names in them for whoever walks them next: trees 1.7
// -> 1.1 ms, Fibonacci 20.0 -> 17.4, 2048 Mul nets 4.8 -> 4.4.
template <class Rules, int I, int J>
__host__ __device__ constexpr bool ends_run() {
  constexpr Template R = Rules::kT[I], T = Rules::kT[J];
  constexpr ChainInfo C = chain_info(R);
  if (I == J || T.n_fresh != 0 || T.n_new > 2) return false;
  const int wl = R.lhs[C.cs];
  if (T.lhs[0] != wl && T.lhs[1] != wl) return false;
  const int side = T.lhs[0] == wl ? 0 : 1;
  for (int p = 0; p < 3; p++) {
    if (C.js[p] < 0) continue;
    int uses = 0;
    for (int k = 0; k < T.n_link; k++)
      for (int i = 0; i < 2; i++) {
        if (T.link[k][i] != kValExt + side * 3 + p) continue;
        const int o = T.link[k][1 - i];
        for (int r = 0; r < 3; r++)
          if (C.js[r] >= 0 && o == kValExt + side * 3 + r) return false;
        uses++;
      }
    if (uses != 1) return false;
  }
  return true;
}

// At the end of a run of rule I: the walker (slot cslot, ports c) has come to
// agent `at` with record nb (its first half when kNarrow) of another label;
// hs, hr: the streams' last agents.  True when a rule ended the run here.
template <bool kTrack, class Rules, int I, bool kNarrow, int J = 0, class WM>
__device__ __forceinline__ bool end_run(const Dev& d, WM& W, Lane& L, int lane, uint32_t net, uint32_t cslot,
                                        const uint32_t (&c)[3], uint32_t at, int4 nb, const uint32_t (&hs)[3],
                                        int4 (&hr)[3], Step& S) {
  if constexpr (J < Rules::kN && J < kSpecialisedMaxRules) {
    if constexpr (ends_run<Rules, I, J>()) {
      constexpr Template R = Rules::kT[I], T = Rules::kT[J];
      constexpr ChainInfo C = chain_info(R);
      constexpr int side = T.lhs[0] == R.lhs[C.cs] ? 0 : 1;
      if (((uint32_t)nb.x & 0xFFu) == T.lhs[1 - side]) {
        if constexpr (kNarrow && chain_arity(T, 1 - side) > 1) nb = ld_node(d.node + at);
        uint32_t v[kNumVals];
#pragma unroll
        for (int q = 0; q < 3; q++) {
          v[side * 3 + q] = c[q];
          v[(1 - side) * 3 + q] = get_aux(nb, q);
        }
        v[kValNew + 0] = mk_agent(cslot);
        v[kValNew + 1] = mk_agent(at);
#pragma unroll
        for (int j = 0; j < (int)T.n_new; j++) {
          int4 rec;
          rec.x = (int32_t)((net << 8) | T.lab[j]);
          rec.y = T.src[j][0] == kValNone ? 0 : (int32_t)v[T.src[j][0]];
          rec.z = T.src[j][1] == kValNone ? 0 : (int32_t)v[T.src[j][1]];
          rec.w = T.src[j][2] == kValNone ? 0 : (int32_t)v[T.src[j][2]];
          st_node(d.node + idx_of(v[kValNew + j]), rec);
        }
#pragma unroll
        for (int k = 0; k < (int)T.n_link; k++) {
          bool stream = false;
#pragma unroll
          for (int p = 0; p < 3; p++) {
            if (C.js[p] < 0) continue;
#pragma unroll
            for (int i = 0; i < 2; i++)
              if (T.link[k][i] == kValExt + side * 3 + p) {
                set_aux(hr[p], C.q[p], v[T.link[k][1 - i]]);
                st_node(d.node + hs[p], hr[p]);
                stream = true;
              }
          }
          if (!stream) put_equation(W, S, lane, v[T.link[k][0]], v[T.link[k][1]]);
        }
        if (T.n_new == 0) put_agent<kTrack>(d, W, L, lane, cslot);
        if (T.n_new < 2) put_agent<kTrack>(d, W, L, lane, at);
        L.live += (int)T.n_new - 2;
        S.fin = J;
        return true;
      }
    }
    return end_run<kTrack, Rules, I, kNarrow, J + 1>(d, W, L, lane, net, cslot, c, at, nb, hs, hr, S);
  }
  return false;
}

// Rule I along a list (see ChainInfo): up to `lim` interactions without
// leaving the lane.  The walker keeps its slot and its ports stay in
// registers; each step loads the next partner (in flight ahead, see below),
// and the record an output stream's last agent waits for gets that step's
// agent in its open port.  The names between two steps are never created,
// the records of agents that come out as they went in (the S of Add(y, r) =
// S(x)) are not rewritten, and the streams' heads are linked once at the
// end, with one fence and one exchange for the whole run instead of one per
// interaction.  What bounds it: about 70 instructions a step of one lane
// (500 cycles alone), then the round trips of partners that do not lie side
// by side.
//
// Partners ahead: lists are mostly laid out in slot order (numerals as they
// were loaded, copies as they were allocated), so each load of a partner
// also loads the next slots in the direction the list last went; they are
// used only if the list really leads there.  Such an early load is as good
// as a late one: an agent that a record already reached names directly is
// owned by this lane, was written before that record was published and does
// not change (a name in between ends the window).
template <bool kTrack, class Rules, int I, class WM>
__device__ __forceinline__ void run_rule(const Dev& d, WM& W, Lane& L, int lane, uint32_t a, uint32_t b,
                                         const int4& ra, const int4& rb, uint32_t net, uint32_t lim, Step& S) {
  constexpr Template R = Rules::kT[I];
  constexpr ChainInfo C = chain_info(R);
  constexpr int kWalk = kValExt + C.cs * 3, kPart = kValExt + (1 - C.cs) * 3;
  constexpr int kNeedA = R.n_new > 2 ? R.n_new - 2 : 0;
  const uint32_t cslot = C.cs == 0 ? a : b;
  uint32_t pslot = C.cs == 0 ? b : a;
  uint32_t v[kNumVals];
  const int4 rw = C.cs == 0 ? ra : rb;
  int4 rp = C.cs == 0 ? rb : ra;
#pragma unroll
  for (int q = 0; q < 3; q++) v[kWalk + q] = get_aux(rw, q);
#pragma unroll
  for (int j = kValNew; j < kNumVals; j++) v[j] = 0;
  v[kValNew + C.jc] = mk_agent(cslot);
  // streams: the equation of the head, and the last agent with its open port
  uint32_t r0[3], h0[3], hs[3], hold[3];
  int4 hr[3];
#pragma unroll
  for (int p = 0; p < 3; p++) {
    r0[p] = h0[p] = hs[p] = hold[p] = 0;
    hr[p] = make_int4(0, 0, 0, 0);
  }
  constexpr uint32_t kWin = 4;
  int4 w0 = rp, w1 = rp, w2 = rp, w3 = rp;
  uint32_t wn = 0, wi = 0, dir = 1;
  uint32_t steps = 0, x = 0;
  bool ready = true;  // the partner rp at pslot is there to be reduced
  S.have_b = false;
  for (uint32_t guard = 0;; guard++) {
    if (ready) {
#pragma unroll
    for (int q = 0; q < 3; q++) v[kPart + q] = get_aux(rp, q);
#pragma unroll
    for (int j = 0; j < (int)R.n_new; j++)
      if (j != C.jc) v[kValNew + j] = mk_agent(j == C.other ? pslot : take_agent(W, L, lane));
    if (C.other < 0) put_agent<kTrack>(d, W, L, lane, pslot);
    // fresh names, but for the ones between this step and the next
#pragma unroll
    for (int f = 0; f < (int)R.n_fresh; f++) {
      bool open = false;
#pragma unroll
      for (int p = 0; p < 3; p++)
        if (C.js[p] >= 0 && R.src[C.jc][p] == kValFresh + f) open = true;
      if (!open) v[kValFresh + f] = mk_var(take_name<kTrack>(d, W, L, lane, net));
    }
    // the streams' previous agents get this step's in their open ports
#pragma unroll
    for (int p = 0; p < 3; p++) {
      if (C.js[p] < 0) continue;
      const uint32_t w = v[kValNew + (C.js[p] < 0 ? 0 : C.js[p])];
      if (steps == 0) {
        r0[p] = v[kWalk + p];
        h0[p] = w;
      } else if (!C.same[p] || hold[p] != w) {
        set_aux(hr[p], C.q[p], w);
        st_node(d.node + hs[p], hr[p]);
      }
    }
    // this step's new agents
#pragma unroll
    for (int j = 0; j < (int)R.n_new; j++) {
      if (j == C.jc) continue;
      int4 rec;
      rec.x = (int32_t)((net << 8) | R.lab[j]);
      rec.y = R.src[j][0] == kValNone ? 0 : (int32_t)v[R.src[j][0]];
      rec.z = R.src[j][1] == kValNone ? 0 : (int32_t)v[R.src[j][1]];
      rec.w = R.src[j][2] == kValNone ? 0 : (int32_t)v[R.src[j][2]];
      bool open = false;
#pragma unroll
      for (int p = 0; p < 3; p++)
        if (C.js[p] == j) {
          hr[p] = rec;
          hs[p] = idx_of(v[kValNew + j]);
          hold[p] = get_aux(rp, C.q[p]);
          open = true;
        }
      if (!open) st_node(d.node + idx_of(v[kValNew + j]), rec);
    }
    // the walker's ports
    uint32_t nx[3];
#pragma unroll
    for (int p = 0; p < 3; p++)
      nx[p] = R.src[C.jc][p] == kValNone || C.js[p] >= 0 ? 0u : v[R.src[C.jc][p] == kValNone ? 0 : R.src[C.jc][p]];
    x = v[C.e];
#pragma unroll
    for (int p = 0; p < 3; p++) v[kWalk + p] = nx[p];
    steps++;
    ready = false;
    }
    // one round trip for every lane of the warp, whatever it waits for: a
    // name (see pass_rule), or the next partner
    const uint32_t at = idx_of(x);
    const bool name = is_var(x);
    if (name ? at >= d.cap_vars || guard > 2 * lim
             : !is_agent(x) || at >= d.cap_agents || steps >= lim || L.na < kNeedA || L.nv < (int)R.n_fresh)
      break;
    uint32_t old = kEmpty;
    if (name) {
      old = ld_volatile(d.var + at);
    } else if (wn == 0 || at != wi) {
      dir = at == pslot - 1 ? ~0u : at == pslot + 1 ? 1u : dir;
      w0 = ld_node(d.node + at);
      const uint32_t i1 = at + dir, i2 = i1 + dir, i3 = i2 + dir;
      w1 = ld_node(d.node + (i1 < d.cap_agents ? i1 : at));
      w2 = ld_node(d.node + (i2 < d.cap_agents ? i2 : at));
      w3 = ld_node(d.node + (i3 < d.cap_agents ? i3 : at));
      wn = kWin;
      wi = at;
    }
    if (name) {
      if (old == kEmpty) break;
      release_name<kTrack>(d, W, L, lane, at);
      x = old;
      wn = 0;
    } else {
      rp = w0;
      w0 = w1;
      w1 = w2;
      w2 = w3;
      wn--;
      wi += dir;
      pslot = at;
      ready = ((uint32_t)rp.x & 0xFFu) == R.lhs[1 - C.cs];
      if (!ready) {
        S.have_b = true;
        break;
      }
    }
  }
  L.live += (long long)((int)R.n_new - 2) * (long long)steps;
  S.steps = steps;
  bool ended = false;
  if (S.have_b) {
    const uint32_t c[3] = {v[kWalk + 0], v[kWalk + 1], v[kWalk + 2]};
    ended = end_run<kTrack, Rules, I, false>(d, W, L, lane, net, cslot, c, pslot, rp, hs, hr, S);
  }
  if (!ended) {
    // each stream's last agent and the walker's port get a name, the
    // walker's record is stored
#pragma unroll
    for (int p = 0; p < 3; p++) {
      if (C.js[p] < 0) continue;
      const uint32_t w = mk_var(take_name<kTrack>(d, W, L, lane, net));
      set_aux(hr[p], C.q[p], w);
      st_node(d.node + hs[p], hr[p]);
      v[kWalk + p] = w;
    }
    int4 rec;
    rec.x = (int32_t)((net << 8) | R.lab[C.jc]);
    rec.y = (int32_t)v[kWalk + 0];
    rec.z = (int32_t)v[kWalk + 1];
    rec.w = (int32_t)v[kWalk + 2];
    st_node(d.node + cslot, rec);
    put_equation(W, S, lane, mk_agent(cslot), x);
    if (S.np) {  // the walker's next pair
      S.fwd = true;
      S.ra = rec;
      S.rb = rp;
    }
  }
#pragma unroll
  for (int p = 0; p < 3; p++)
    if (C.js[p] >= 0) put_equation(W, S, lane, r0[p], h0[p]);
}

// A run of a rule that leaves its partners as they are (chain_passes): the
// walker only has to find where the list ends, so the loop is a walk: along
// neighbouring slots (numerals as they were loaded, copies as they were
// allocated) kBlock partners at a time, their loads in flight together and
// used as far as the list really goes through them; else one by one.  A
// record loaded before the list was seen to lead to it is as good as one
// loaded after: an agent that a record already reached names directly is
// owned by this lane, was written before that record was published and does
// not change.  What bounds it: one L2 round trip (337 ns) per block, partner
// or name, so a turn of the loop issues whatever each lane waits for at once.
// The chain of 20 000 Add takes 0.11 us an interaction (0.34 in run_rule, 1.3
// with one a turn), 4096 short sums 0.12 ms (0.69).  Blocks of 4 against 8: 2048
// Mul nets 4.4 / 5.0 ms, the chain 2.2 / 2.0, Fibonacci the same.
template <bool kTrack, class Rules, int I, class WM>
__device__ __forceinline__ void pass_rule(const Dev& d, WM& W, Lane& L, int lane, uint32_t a, uint32_t b,
                                          const int4& ra, const int4& rb, uint32_t net, uint32_t lim, Step& S) {
  constexpr Template R = Rules::kT[I];
  constexpr ChainInfo C = chain_info(R);
  constexpr int kPort = C.e % 3;                                // the partner's port the walker goes on to
  constexpr int kOut = C.js[0] >= 0 ? 0 : C.js[1] >= 0 ? 1 : 2;  // the walker's port of the output stream
  constexpr uint32_t kLabel = R.lhs[1 - C.cs];
  constexpr bool kNarrow = chain_arity(R, 1 - C.cs) == 1;       // head and one port hold a whole partner
  constexpr uint32_t kBlock = 4;
  const uint32_t cslot = C.cs == 0 ? a : b;
  const uint32_t first = C.cs == 0 ? b : a;
  const uint32_t cap = (uint32_t)d.cap_agents;
  uint32_t cur = first;
  int4 rc = C.cs == 0 ? rb : ra;  // the partner the walker is at, and its record
  uint32_t x = get_aux(rc, kPort), steps = 1;
  int end = 0;  // the walker has come to an agent of another label: 1: its record is nb, 2: the record's first half
  int4 nb = make_int4(0, 0, 0, 0);
  for (uint32_t guard = 0;; guard++) {
    // one round trip for every lane of the warp, whatever it waits for: a
    // name, or the next partners
    const uint32_t at = idx_of(x);
    const bool name = is_var(x);
    if (name ? at >= d.cap_vars || guard > 2 * lim : !is_agent(x) || at >= cap || steps >= lim) break;
    // neighbouring slots: the whole block
    const uint32_t dir = at - cur;
    const bool block = !name && ((dir == 1u && at + kBlock <= cap) || (dir == ~0u && at + 1 >= kBlock));
    uint32_t old = kEmpty;
    int4 w[kBlock];
    if (name) old = ld_volatile(d.var + at);
    else w[0] = ld_partner<kNarrow>(d.node + at);
    if (block) {
#pragma unroll
      for (int j = 1; j < (int)kBlock; j++) w[j] = ld_partner<kNarrow>(d.node + (at + (uint32_t)j * dir));
    }
    if (name) {
      // one whose other occurrence has arrived: this one is the second (the
      // slot is finished, nobody else refers to it), so the walker goes on
      // without being published; an empty one ends the run
      if (old == kEmpty) break;
      release_name<kTrack>(d, W, L, lane, at);
      x = old;
      if (is_agent(x)) {
        set_aux(rc, kPort, x);
        st_node(d.node + cur, rc);
      }
      continue;
    }
    if (((uint32_t)w[0].x & 0xFFu) != kLabel) {
      end = kNarrow ? 2 : 1;
      nb = w[0];
      break;
    }
    steps++;
    cur = at;
    rc = w[0];
    x = get_aux(rc, kPort);
    if (block) {
      bool on = true, other = false;
#pragma unroll
      for (int j = 1; j < (int)kBlock; j++) {
        on = on && x == mk_agent(at + (uint32_t)j * dir);
        if (on && ((uint32_t)w[j].x & 0xFFu) != kLabel) {
          on = false;
          other = true;
          nb = w[j];
        }
        if (on) {
          steps++;
          cur = at + (uint32_t)j * dir;
          x = get_aux(w[j], kPort);
          rc = w[j];
        }
      }
      if (other) {
        end = kNarrow ? 2 : 1;
        break;
      }
    }
  }
  const int4& rw = C.cs == 0 ? ra : rb;
  const uint32_t r0 = get_aux(rw, kOut);
  S.steps = steps;
  bool ended = false;
  if (end) {
    const uint32_t c[3] = {get_aux(rw, 0), get_aux(rw, 1), get_aux(rw, 2)};
    const uint32_t hs[3] = {cur, cur, cur};
    int4 hr[3] = {rc, rc, rc};
    ended = end_run<kTrack, Rules, I, kNarrow>(d, W, L, lane, net, cslot, c, idx_of(x), nb, hs, hr, S);
  }
  if (!ended) {
    // the last partner's and the walker's port get a name
    const uint32_t w = mk_var(take_name<kTrack>(d, W, L, lane, net));
    set_aux(rc, kPort, w);
    st_node(d.node + cur, rc);
    S.ra = rw;
    set_aux(S.ra, kOut, w);
    st_node(d.node + cslot, S.ra);
    put_equation(W, S, lane, mk_agent(cslot), x);
    S.fwd = S.np != 0;  // the walker's next pair
    S.have_b = end == 1;
    S.rb = nb;
  }
  put_equation(W, S, lane, r0, mk_agent(first));
}

// The templates of the rules with their own code (which may hold reduced
// pairs) in place of the loaded ones.
template <class Rules, int I = 0>
__device__ __forceinline__ void spec_templates(PackedTpl* tmpl) {
  if constexpr (I < Rules::kN && I < kSpecialisedMaxRules) {
    constexpr Template R = Rules::kT[I];
    constexpr uint32_t kIn = Rules::kMore[I][0] | (Rules::kMore[I][1] << 8) | (Rules::kMore[I][2] << 16);
    if (threadIdx.x == I) tmpl[I] = pack_template(R, kIn);
    spec_templates<Rules, I + 1>(tmpl);
  }
}
static_assert(kSpecialisedMaxRules <= 32, "one thread of the smallest block per rule");

// Some rule other than I that repeats itself along lists has label B on its
// left-hand side.
template <class Rules, int B, int I, int J = 0>
__host__ __device__ constexpr bool walked() {
  if constexpr (J < Rules::kN && J < kSpecialisedMaxRules) {
    constexpr Template T = Rules::kT[J];
    return (J != I && (T.lhs[0] == B || T.lhs[1] == B) && chain_info(T).ok) || walked<Rules, B, I, J + 1>();
  } else {
    return false;
  }
}

// Rule I is reduced in runs.  A run holds its output back until it ends, which
// costs nothing where the list is walked as a whole again; where every other
// rule takes the stream's agents one at a time, each could have had its own as
// soon as it was made, so such a rule makes one interaction a turn: the
// L-System's Dup, whose copies only SymA and SymB take (with the smaller refills,
// 13 steps 0.30 -> 0.20 ms, 22 steps 0.61 -> 0.42).  The arithmetic rules' Dup, whose copies Mul and
// Add walk, is the faster in runs: 2048 Mul nets 4.4 ms against 11.5.
template <class Rules, int I>
__host__ __device__ constexpr bool runs_along() {
  constexpr Template R = Rules::kT[I];
  constexpr ChainInfo C = chain_info(R);
  if (!C.ok || chain_passes(R, C)) return C.ok;
  constexpr int j0 = C.js[0] < 0 ? 0 : C.js[0], j1 = C.js[1] < 0 ? 0 : C.js[1], j2 = C.js[2] < 0 ? 0 : C.js[2];
  return (C.js[0] < 0 || walked<Rules, R.lab[j0], I>()) && (C.js[1] < 0 || walked<Rules, R.lab[j1], I>()) &&
         (C.js[2] < 0 || walked<Rules, R.lab[j2], I>());
}

// Bit I set: rule I is reduced in runs.
template <class Rules, int I = 0>
__device__ constexpr uint32_t run_mask() {
  if constexpr (I < Rules::kN && I < kSpecialisedMaxRules)
    return (runs_along<Rules, I>() ? 1u << I : 0u) | run_mask<Rules, I + 1>();
  else return 0u;
}

// One interaction of a rule read from shared memory.  The general kernel
// keeps the values in a table; a specialised one, where few lanes come here,
// finds each where it is: the arguments in
// registers, the new slots on top of the lane's columns.
template <bool kTrack, class WM>
__device__ __forceinline__ void interpret(const Dev& d, WM& W, Lane& L, int lane, const PackedTpl& T, uint32_t a,
                                          uint32_t b, const int4& ra, const int4& rb, uint32_t net, Step& S) {
  const uint32_t hdr = T.hdr;
  const uint32_t n_new = hdr & 0xFFu, n_fresh = (hdr >> 8) & 0xFFu, n_link = (hdr >> 16) & 0xFFu;
  const int ta = L.na, tv = L.nv;
  auto value = [&](uint32_t c) -> uint32_t {
    if constexpr (WM::kHasTable) {
      return W.vals[c][lane];
    } else {
      if (c < (uint32_t)kValNew) {
        const uint32_t q = c < 3 ? c : c - 3;
        return get_aux(c < 3 ? ra : rb, (int)q);
      }
      if (c < (uint32_t)kValFresh) {
        const int j = (int)c - kValNew;
        return mk_agent(j == 0 ? a : j == 1 ? b : W.ares[ta - 1 - (j - 2)][lane]);
      }
      return mk_var(W.vres[tv - 1 - ((int)c - kValFresh)][lane]);
    }
  };
  auto port = [&](uint32_t c) -> int32_t { return c == kValNone ? 0 : (int32_t)value(c); };
  if constexpr (WM::kHasTable) {
    W.vals[kValExt + 0][lane] = (uint32_t)ra.y;
    W.vals[kValExt + 1][lane] = (uint32_t)ra.z;
    W.vals[kValExt + 2][lane] = (uint32_t)ra.w;
    W.vals[kValExt + 3][lane] = (uint32_t)rb.y;
    W.vals[kValExt + 4][lane] = (uint32_t)rb.z;
    W.vals[kValExt + 5][lane] = (uint32_t)rb.w;
    if (n_new > 0) W.vals[kValNew + 0][lane] = mk_agent(a);
    if (n_new > 1) W.vals[kValNew + 1][lane] = mk_agent(b);
  }
  for (uint32_t j = 2; j < n_new; j++) {
    const uint32_t sl = take_agent(W, L, lane);
    if constexpr (WM::kHasTable) W.vals[kValNew + j][lane] = mk_agent(sl);
  }
  for (uint32_t f = 0; f < n_fresh; f++) {
    const uint32_t x = take_name<kTrack>(d, W, L, lane, net);
    if constexpr (WM::kHasTable) W.vals[kValFresh + f][lane] = mk_var(x);
  }
  for (uint32_t j = 0; j < n_new; j++) {
    const uint32_t w = T.agent[j];
    int4 rec;
    rec.x = (int32_t)((net << 8) | (w & 0xFFu));
    rec.y = port((w >> 8) & 0xFFu);
    rec.z = port((w >> 16) & 0xFFu);
    rec.w = port(w >> 24);
    st_node(d.node + idx_of(value(kValNew + j)), rec);
  }
  S.steps = 1;
  for (uint32_t k = 0; k < n_link; k++) {
    const uint32_t lk = T.link[k];
    put_equation(W, S, lane, value(lk & 0xFFu), value(lk >> 8));
  }
  if (n_new == 0) put_agent<kTrack>(d, W, L, lane, a);
  if (n_new < 2) put_agent<kTrack>(d, W, L, lane, b);
  L.live += (long long)n_new - 2;
}

template <bool kTrack, class Rules, int I, class WM>
__device__ __forceinline__ void spec_rule(const Dev& d, WM& W, Lane& L, int lane, uint32_t a, uint32_t b,
                                          const int4& ra, const int4& rb, uint32_t net, uint32_t lim,
                                          Step& S) {
  if constexpr (I < Rules::kN && I < kSpecialisedMaxRules) {
    if constexpr (chain_passes(Rules::kT[I], chain_info(Rules::kT[I])))
      pass_rule<kTrack, Rules, I>(d, W, L, lane, a, b, ra, rb, net, lim, S);
    else if constexpr (runs_along<Rules, I>()) run_rule<kTrack, Rules, I>(d, W, L, lane, a, b, ra, rb, net, lim, S);
    else one_step<kTrack, Rules, I>(d, W, L, lane, a, b, ra, rb, net, S);
  }
}
#define INET_SPEC_CASE(I)                                                             \
  case I:                                                                             \
    spec_rule<kTrack, Rules, I>(d, W, L, lane, a, b, ra, rb, net, lim, S);             \
    break;

// One step of each lane whose `valid` is set: an interaction, or a run of
// them (warp-collective).  The new active pairs are left in
// W.out[0..S.np)[lane]; a pair that cannot be reduced (no rule, corrupt
// state) is dropped.
template <bool kTrack, class Rules, class WM>
__device__ __forceinline__ void async_interact(const Dev& d, const PackedTpl* tmpl, const int16_t* tab,
                                               uint32_t* hist, WM& W, Lane& L, bool valid, uint32_t a,
                                               uint32_t b, bool pre, int4 ra, int4 rb, Step& S) {
  const int lane = threadIdx.x & 31;
  uint32_t net = 0, ti = 0;
  S.np = S.ne = S.steps = 0;
  S.fwd = S.have_b = false;
  S.fin = -1;
  if (valid && (a >= d.cap_agents || b >= d.cap_agents)) {
    report(d, INET_ERR_STATE, 2);
    valid = false;
  }
  if (valid) {
    if (!pre) {
      ra = ld_node(d.node + a);
      rb = ld_node(d.node + b);
    }
    const uint32_t la = (uint32_t)ra.x & 0xFFu, lb = (uint32_t)rb.x & 0xFFu;
    const int e = (la < d.n_labels && lb < d.n_labels) ? tab[la * d.n_labels + lb] : -1;
    net = (uint32_t)ra.x >> 8;
    if (net >= d.max_nets) {
      report(d, INET_ERR_STATE, 3);
      valid = false;
    } else if (e < 0) {
      valid = false;
      atomicCAS(d.netstat + net, 0, INET_ERR_NO_RULE);
      report(d, INET_ERR_NO_RULE, net);
      atomicAdd(d.netctr + net, (unsigned long long)(-(1ll << kNetPairShift)));
    } else {
      if (e & 1) {
        int4 t = ra; ra = rb; rb = t;
        uint32_t u = a; a = b; b = u;
      }
      ti = (uint32_t)e >> 1;
    }
  }
  const uint32_t hdr = valid ? tmpl[ti].hdr : 0u;
  const uint32_t n_new = hdr & 0xFFu, need_a = n_new > 2 ? n_new - 2 : 0u, need_v = (hdr >> 8) & 0xFFu;
  const unsigned lack = __ballot_sync(kFull, (uint32_t)L.na < need_a || (uint32_t)L.nv < need_v);
  if (lack) {
    bool runs = false;
    if constexpr (Rules::kN > 0) runs = (run_mask<Rules>() >> (ti & 31u)) & 1u;
    // In a warp with few pairs a lane may have its last one here, and what it
    // took for later would send the next lane to the pools (L-System(19) 0.30
    // ms, 0.32 with 4 or more always); a lane of a busy warp will be back (64
    // Fibonacci nets 41 ms, 43 with the bare need).
    const uint32_t more = __popc(__ballot_sync(kFull, valid)) >= 16 ? 4u : 0u;
    if (!refill(d, W, L, runs, more, need_a, need_v, lane)) return;  // fatal: the loop stops
  }
  // a run keeps the warp's other lanes waiting, and what waits for its output
  uint32_t lim = 1;
  if constexpr (Rules::kN > 0) {
    const bool one = valid && !(ti < 32 && ((run_mask<Rules>() >> (ti & 31u)) & 1u));
    const int all = __popc(__ballot_sync(kFull, valid)), ones = __popc(__ballot_sync(kFull, one));
    lim = all == 1 ? kRunLone : 2 * ones > all ? kRunMixed : kRunMany;
  }
  if (valid) {
    if constexpr (Rules::kN == 0) {
      interpret<kTrack>(d, W, L, lane, tmpl[ti], a, b, ra, rb, net, S);
    } else {
      switch (ti) {
        INET_SPEC_CASE(0) INET_SPEC_CASE(1) INET_SPEC_CASE(2) INET_SPEC_CASE(3) INET_SPEC_CASE(4) INET_SPEC_CASE(5)
        INET_SPEC_CASE(6) INET_SPEC_CASE(7) INET_SPEC_CASE(8) INET_SPEC_CASE(9) INET_SPEC_CASE(10) INET_SPEC_CASE(11)
        INET_SPEC_CASE(12) INET_SPEC_CASE(13) INET_SPEC_CASE(14) INET_SPEC_CASE(15) INET_SPEC_CASE(16)
        INET_SPEC_CASE(17) INET_SPEC_CASE(18) INET_SPEC_CASE(19) INET_SPEC_CASE(20) INET_SPEC_CASE(21)
        INET_SPEC_CASE(22) INET_SPEC_CASE(23) INET_SPEC_CASE(24) INET_SPEC_CASE(25) INET_SPEC_CASE(26)
        INET_SPEC_CASE(27) INET_SPEC_CASE(28) INET_SPEC_CASE(29) INET_SPEC_CASE(30) INET_SPEC_CASE(31)
        default:
          if constexpr (Rules::kN > kSpecialisedMaxRules)
            interpret<kTrack>(d, W, L, lane, tmpl[ti], a, b, ra, rb, net, S);
          break;
      }
      static_assert(kSpecialisedMaxRules == 32, "one case per rule with its own code");
    }
  }
  if (__any_sync(kFull, S.ne != 0)) {
    __threadfence();
    if (S.ne) link_lane<kTrack>(d, W, L, S, lane);
  }
  if (valid) {
    // per-net counters (interactions and the change of pending pairs) and
    // the rule histogram: one fire-and-forget atomic each; with kTrack the
    // net's live agents too (its quota is checked between launches)
    const uint32_t in = tmpl[ti].inside, n_in = in & 0xFFu;
    uint32_t ints = S.steps * (1 + n_in);
    long long dlive = ((long long)n_new - 2) * (long long)S.steps;
    atomicAdd(&hist[hdr >> 24], S.steps);
    if (n_in > 0) atomicAdd(&hist[(in >> 8) & 0xFFu], S.steps);
    if (n_in > 1) atomicAdd(&hist[(in >> 16) & 0xFFu], S.steps);
    if (Rules::kN > 0 && S.fin >= 0) {
      const uint32_t fh = tmpl[S.fin].hdr, fi = tmpl[S.fin].inside, f_in = fi & 0xFFu;
      ints += 1 + f_in;
      dlive += (long long)(fh & 0xFFu) - 2;
      atomicAdd(&hist[fh >> 24], 1u);
      if (f_in > 0) atomicAdd(&hist[(fi >> 8) & 0xFFu], 1u);
      if (f_in > 1) atomicAdd(&hist[(fi >> 16) & 0xFFu], 1u);
    }
    atomicAdd(d.netctr + net, (unsigned long long)ints + ((unsigned long long)((long long)S.np - 1) << kNetPairShift));
    if constexpr (kTrack) {
      if (dlive) atomicAdd(reinterpret_cast<unsigned long long*>(d.netlive + net), (unsigned long long)dlive);
    }
  }
  __syncwarp();
}
#undef INET_SPEC_CASE

// Writes a pair back to the exit frontier (other buffer).
__device__ __noinline__ void exit_pair(const Dev& d, Pair p) {
  const uint32_t k = atomicAdd(&d.ctrl->aexit, 1u);
  if (k < d.cap_pairs) {
    __stcg(reinterpret_cast<unsigned long long*>(d.front[d.qcur ^ 1u] + k), *reinterpret_cast<unsigned long long*>(&p));
  } else {
    set_error(d.ctrl, INET_ERR_ARENA_FULL, 5);
  }
}

// A lane that claimed a ticket takes its pair as soon as it is published
// and frees the cell for the next lap.  Every wait of the asynchronous loop
// does this too, so a producer waiting for a cell never waits on a lane
// that is itself waiting.
__device__ __forceinline__ void poll_ticket(const Dev& d, const Pair* Q, bool& have, unsigned long long& ticket,
                                            unsigned long long tslot, uint32_t& pa, uint32_t& pb) {
  if (!have && ticket != kNoTicket) {
    unsigned long long* sq = d.qseq + tslot;
    if (ld_acquire64(sq) == ticket + 1) {
      const unsigned long long v = __ldcg(reinterpret_cast<const unsigned long long*>(Q + tslot));
      st_release64(sq, ticket + d.cap_pairs);
      pa = (uint32_t)v;
      pb = (uint32_t)(v >> 32);
      have = true;
      ticket = kNoTicket;
    }
  }
}

// Bounded wait for ticket t's pair (when no producer runs any more);
// returns false on timeout.
__device__ __noinline__ bool wait_ticket(const Dev& d, const Pair* Q, unsigned long long t, Pair* out) {
  const unsigned long long s = t % d.cap_pairs;
  const unsigned long long t0 = globaltimer();
  for (uint32_t spin = 0;; spin++) {
    if (ld_acquire64(d.qseq + s) == t + 1) {
      const unsigned long long v = __ldcg(reinterpret_cast<const unsigned long long*>(Q + s));
      *out = Pair{(uint32_t)v, (uint32_t)(v >> 32)};
      return true;
    }
    __nanosleep(64);
    if ((spin & 63) == 63 && globaltimer() - t0 > d.timeout_ns) {
      set_error(d.ctrl, INET_ERR_TIMEOUT, 6);
      return false;
    }
  }
}

template <bool kTrack, class Rules = NoRules>
__global__ void __launch_bounds__(256, 2) k_async(Dev d) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  size_t off = 0;
  auto take = [&](size_t n) { off = (off + 15) / 16 * 16; unsigned char* p = smem_raw + off; off += n; return p; };
  PackedTpl* tmpl = reinterpret_cast<PackedTpl*>(take(sizeof(PackedTpl) * (d.n_tmpl ? d.n_tmpl : 1)));
  using WM = WarpMem<Rules::kN == 0>;
  WM* wm = reinterpret_cast<WM*>(take(sizeof(WM) * (blockDim.x / 32)));
  uint32_t* hist = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * INET_MAX_RULES));
  int16_t* tab = reinterpret_cast<int16_t*>(take(sizeof(int16_t) * d.n_labels * d.n_labels));
#pragma unroll 1
  for (uint32_t i = threadIdx.x; i < d.n_tmpl; i += blockDim.x) tmpl[i] = pack_template(d.tmpl[i]);
#pragma unroll 1
  for (uint32_t i = threadIdx.x; i < d.n_labels * d.n_labels; i += blockDim.x) tab[i] = d.table[i];
#pragma unroll 1
  for (uint32_t i = threadIdx.x; i < INET_MAX_RULES; i += blockDim.x) hist[i] = 0;
  if constexpr (Rules::kN > 0) {
    // a specialised kernel runs only on the rule set it was built for (the
    // check sits after the carve-up of shared memory: at the top of the
    // kernel it cost the loop 6 more registers)
    if (d.rules_key != Rules::kKey || d.n_tmpl != (uint32_t)Rules::kN) {
      if (threadIdx.x == 0 && blockIdx.x == 0) set_error(d.ctrl, INET_ERR_STATE, 10);
      return;
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  WM& W = wm[wid];
  if (lane == 0) W.an = W.vn = 0;
  Lane L{0, 0, 0};
  __syncthreads();
  if constexpr (Rules::kN > 0) {
    spec_templates<Rules>(tmpl);
    __syncthreads();
  }
  Ctrl* c = d.ctrl;
  Pair* Q = d.front[d.qcur];
  const unsigned long long cap = d.cap_pairs;
  const uint32_t total_warps = gridDim.x * (blockDim.x / 32);
  bool have = false;
  uint32_t pa = 0, pb = 0;
  unsigned long long ticket = kNoTicket, tslot = 0;
  uint32_t nap = 0, flag = 0;
  unsigned long long qh = 0, qt = 0;
  bool stop = false, finished = false, check_now = false;
  bool pre = false;
  int4 pra = make_int4(0, 0, 0, 0), prb = pra;
  unsigned long long t_start = 0;
  if (lane == 0) {
    const unsigned long long now = globaltimer();
    atomicCAS(&c->slice_t0, 0ull, now);
    t_start = ld_volatile64(&c->slice_t0);
  }
  for (uint32_t it = 0;; it++) {
    // stop / slice checks every 4 iterations (on flags loaded during the
    // iteration before; an iteration may hold a run, and with 16 a slice of 250
    // us took 2.2 ms on 64 Fibonacci nets instead of 0.56), and when a napping
    // warp's clock says the time slice is over
    if ((it & 3) == 3 || check_now) {
      if (check_now) {
        if (lane == 1) flag = ld_volatile(&c->astop);
        if (lane == 2) flag = ld_volatile((const uint32_t*)&c->fatal);
      }
      check_now = false;
      uint32_t st = __any_sync(kFull, flag != 0) ? 1u : 0u;
      if (lane == 0) {
        if (!st && globaltimer() - t_start > d.slice_ns) {
          c->astop = 1;
          c->hit_slice = 1;
          st = 1;
        }
      }
      if (__shfl_sync(kFull, st, 0)) {
        stop = true;
        break;
      }
    }
    // claim tickets for lanes without work when the queue has unclaimed
    // pairs.  While the queue holds fewer pairs than there are warps, only a
    // warp with no work claims, and one ticket at a time: each queued pair,
    // and the chain of interactions it starts, gets a warp of its own (with
    // idle lanes for the pairs it hands on) instead of sharing one with up
    // to 31 others, whose divergent work would slow every lane (2048 Mul
    // nets: 14.5 -> 12.9 ms with the grid at full occupancy).  A longer
    // queue is drained by every warp, busy ones looking every 8th iteration.
    const unsigned want = __ballot_sync(kFull, !have && ticket == kNoTicket);
    const unsigned busy = __ballot_sync(kFull, have);
    if (want && (!busy || (it & 7) == 0)) {
      unsigned long long base = 0;
      uint32_t k = 0;
      if (lane == 0) {
        // a busy warp looks at what it loaded during the iteration before
        if (!busy) asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(qh), "=l"(qt) : "l"(&c->q_head) : "memory");
        const unsigned long long backlog = qt > qh ? qt - qh : 0ull;
        const bool deep = backlog > total_warps;
        if (backlog && (!busy || deep)) {
          k = (uint32_t)min(min((unsigned long long)__popc(want), backlog), deep ? 32ull : 1ull);
          base = atomicAdd(&c->q_head, (unsigned long long)k);
        }
      }
      k = __shfl_sync(kFull, k, 0);
      if (k) {
        unsigned long long bm = 0;
        if (lane == 0) bm = base % cap;
        base = __shfl_sync(kFull, base, 0);
        bm = __shfl_sync(kFull, bm, 0);
        const unsigned rank = __popc(want & lanemask_lt());
        if (((want >> lane) & 1u) && rank < k) {
          ticket = base + rank;
          tslot = bm + rank;
          if (tslot >= cap) tslot %= cap;
        }
      }
    }
    poll_ticket(d, Q, have, ticket, tslot, pa, pb);
    const unsigned act = __ballot_sync(kFull, have);
    if (!act) {
      // idle: the loop is over when no pair is left anywhere
      uint32_t fin = 0;
      if (lane == 0) fin = ld_volatile_s64(&c->inflight) == 0 ? 1u : 0u;
      if (lane == 1) flag = ld_volatile(&c->astop);
      if (lane == 2) flag = ld_volatile((const uint32_t*)&c->fatal);
      if (__shfl_sync(kFull, fin, 0)) {
        finished = true;
        break;
      }
      // back off up to 16 us: with thousands of warps, most of them idle
      // in a narrow phase, shorter naps make their polling of the queue and
      // of the in-flight count contend with the warps doing the work (an
      // Ackermann batch 77 -> 63 ms, 2048 Mul nets 13.1 -> 12.7 ms).  The
      // slice's end is noticed from the clock, which needs no memory access.
      __nanosleep(nap);
      nap = nap < 16384 ? nap * 2 + 32 : 16384;
      {
        uint32_t late = 0;
        if (lane == 0) late = globaltimer() - t_start > d.slice_ns ? 1u : 0u;
        check_now = __any_sync(kFull, late != 0 || flag != 0);
      }
      continue;
    }
    nap = 0;
    if ((it & 3) == 2) {
      if (lane == 1) flag = ld_volatile(&c->astop);
      if (lane == 2) flag = ld_volatile((const uint32_t*)&c->fatal);
    }
    const bool look = (it & 7) == 7;
    if (look && lane == 0)
      asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(qh), "=l"(qt) : "l"(&c->q_head) : "memory");
    Step S;
    async_interact<kTrack, Rules>(d, tmpl, tab, hist, W, L, have, pa, pb, pre, pra, prb, S);
    const uint32_t np = S.np;
    // keep the first new pair; the records the step hands on in registers
    // need no load, the others are loaded below
    const bool had = have;
    have = np > 0;
    bool lda = have && !S.fwd, ldb = have && (!S.fwd || !S.have_b);
    pre = have;
    if (have) {
      const Pair p0 = W.out[0][lane];
      pa = p0.a;
      pb = p0.b;
      pra = S.ra;
      prb = S.rb;
    }
    const uint32_t extra = np > 1 ? np - 1 : 0u;
    // pairs in flight: each new pair beyond a lane's own next one joins
    // before it is published to another warp (lane 0 waits until the
    // increment is performed, so no consumer's decrement can overtake it);
    // each pair that produced nothing leaves afterwards.  When every new
    // pair stays in this warp the increment need not be waited for: only
    // this warp's lane 0 can later count those pairs out, and its atomics on
    // the counter are performed in program order, while the producing
    // lane's own next pair keeps the count above zero meanwhile.  At most
    // cap pairs may be in flight, the capacity of the frontier that a stop
    // drains them to; beyond it the arena is full (checked whenever pairs
    // go to the queue).  Under that bound the queue slot a producer needs
    // is held by a claimed ticket whenever it is still occupied: an
    // unclaimed one would put every later ticket, and so more than cap
    // pairs, in flight.
    const long long shrink = -(long long)__popc(__ballot_sync(kFull, had && np == 0));
    unsigned more = __ballot_sync(kFull, extra != 0);
    if (more) {
      // extra pairs go first to idle lanes of this warp (through shared
      // memory), the rest to the ticket queue
      // the lanes' first extra pairs, then their second ones, ...
      unsigned totx = 0;
#pragma unroll 1
      for (uint32_t j = 0; more; j++) {
        if (j < extra) W.xl[totx + __popc(more & lanemask_lt())] = W.out[1 + j][lane];
        totx += __popc(more);
        more = __ballot_sync(kFull, j + 1 < extra);
      }
      {
        const long long grow = (long long)totx;
        const unsigned idle = __ballot_sync(kFull, !have && ticket == kNoTicket);
        const unsigned nidle = __popc(idle);
        __syncwarp();
        const unsigned local = min(nidle, totx);
        if (lane == 0) {
          unsigned long long* ifl = reinterpret_cast<unsigned long long*>(&c->inflight);
          if (totx > local) {
            const long long r = (long long)atomicAdd(ifl, (unsigned long long)grow);
            if (r + grow > (long long)cap) set_error(c, INET_ERR_ARENA_FULL, 9);
          } else {
            atomicAdd(ifl, (unsigned long long)grow);
          }
        }
        __syncwarp();
        if ((idle >> lane) & 1u) {
          const unsigned r = __popc(idle & lanemask_lt());
          if (r < local) {
            const Pair p = W.xl[r];
            pa = p.a;
            pb = p.b;
            have = pre = lda = ldb = true;
          }
        }
        const unsigned toq = totx - local;
        if (toq) {
          // a step that left only agent-agent equations has not fenced: the
          // records of every pair are published before the pair is
          __threadfence();
          __syncwarp();
          unsigned long long qb = 0, qm = 0;
          if (lane == 0) {
            qb = atomicAdd(&c->q_tail, (unsigned long long)toq);
            qm = qb % cap;
          }
          qb = __shfl_sync(kFull, qb, 0);
          qm = __shfl_sync(kFull, qm, 0);
#pragma unroll 1
          for (unsigned j0 = 0; j0 < toq; j0 += 32) {
            const unsigned j = j0 + (unsigned)lane;
            bool pend = j < toq;
            const unsigned long long tk = qb + j;
            unsigned long long si = qm + j;
            if (si >= cap) si %= cap;
            const Pair p = pend ? W.xl[local + j] : Pair{0, 0};
            const unsigned long long t0 = globaltimer();
#pragma unroll 1
            for (uint32_t spin = 0;; spin++) {
              // written once the cell's previous pair (ticket tk - cap) is taken
              if (pend && ld_acquire64(d.qseq + si) == tk) {
                __stcg(reinterpret_cast<unsigned long long*>(Q + si),
                       (unsigned long long)p.a | ((unsigned long long)p.b << 32));
                st_release64(d.qseq + si, tk + 1);
                pend = false;
              }
              poll_ticket(d, Q, have, ticket, tslot, pa, pb);
              if (!__any_sync(kFull, pend)) break;
              __nanosleep(64);
              if ((spin & 15) == 15) {
                // after a fatal error (the arena is poisoned) or the time
                // limit, pairs not yet written are given up
                uint32_t give = 0;
                if (lane == 0) {
                  if (ld_volatile((const uint32_t*)&c->fatal)) {
                    give = 1;
                  } else if (globaltimer() - t0 > d.timeout_ns) {
                    set_error(c, INET_ERR_TIMEOUT, 7);
                    give = 1;
                  }
                }
                if (__shfl_sync(kFull, give, 0)) break;
              }
            }
          }
        }
        __syncwarp();
      }
    }
    if (lane == 0 && shrink) atomicAdd(reinterpret_cast<unsigned long long*>(&c->inflight), (unsigned long long)shrink);
    // one load for the lanes that keep a pair and the lanes handed one (two
    // loads of the same registers would wait for each other), in flight
    // during the next iteration's top
    if (pa >= d.cap_agents || pb >= d.cap_agents) pre = lda = ldb = false;
    if (lda) pra = ld_node(d.node + pa);
    if (ldb) prb = ld_node(d.node + pb);
    __syncwarp();
  }
  // leaving: publish live agents; a stop drains every pair to the other buffer
  {
    long long live = L.live;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) live += __shfl_xor_sync(kFull, live, o);
    if (lane == 0 && live) atomicAdd(reinterpret_cast<unsigned long long*>(&c->live), (unsigned long long)live);
  }
  if (finished && !stop) {
    if (lane == 0) {
      __threadfence();
      atomicAdd(&c->quiesce, 1u);
    }
  } else {
    uint32_t ok = 1;
    if (lane == 0) {
      __threadfence();
      atomicAdd(&c->quiesce, 1u);
    }
    __syncwarp();
    const unsigned long long t0 = globaltimer();
    for (;;) {
      poll_ticket(d, Q, have, ticket, tslot, pa, pb);  // producers still running may wait for this lane's slot
      uint32_t done = 0;
      if (lane == 0) {
        if (ld_volatile(&c->quiesce) >= total_warps) {
          done = 1;
        } else if (globaltimer() - t0 > d.timeout_ns) {
          set_error(c, INET_ERR_TIMEOUT, 8);
          ok = 0;
          done = 1;
        }
      }
      if (__shfl_sync(kFull, done, 0)) break;
      __nanosleep(256);
    }
    if (lane == 0) {
      __threadfence();
      if (ld_volatile((const uint32_t*)&c->fatal)) ok = 0;  // poisoned: nothing to keep
    }
    ok = __shfl_sync(kFull, ok, 0);
    if (ok) {
      const unsigned long long qt = ld_volatile64(&c->q_tail);
      if (!have && ticket != kNoTicket && ticket < qt) {
        Pair p;
        if (wait_ticket(d, Q, ticket, &p)) {
          pa = p.a;
          pb = p.b;
          have = true;
        }
      }
      if (have) exit_pair(d, Pair{pa, pb});
      // unclaimed tickets, shared among the warps
      const unsigned long long qh = ld_volatile64(&c->q_head);
      const uint32_t gw = blockIdx.x * (blockDim.x / 32) + (uint32_t)wid;
#pragma unroll 1
      for (unsigned long long tk = qh + (unsigned long long)gw * 32 + lane; tk < qt;
           tk += (unsigned long long)total_warps * 32) {
        Pair p;
        if (wait_ticket(d, Q, tk, &p)) exit_pair(d, p);
      }
    }
  }
  // free slots known only to this warp go back to the rings (when owners are
  // kept, marked free: some were fetched from the pools and never used, which
  // may come from the bump pointer with stale contents)
  __syncwarp();
  {
    const uint32_t ac = (uint32_t)min(W.an, WM::kAStack), vc = (uint32_t)min(W.vn, WM::kVStack);
    uint32_t inc = (uint32_t)L.na | ((uint32_t)L.nv << 16);
    const uint32_t own = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += t;
    }
    const uint32_t tot = __shfl_sync(kFull, inc, 31);
    const uint32_t ta = ac + (tot & 0xFFFFu), tv = vc + (tot >> 16);
    unsigned long long ab = 0, vb = 0;
    if (lane == 0) {
      if (ta) ab = atomicAdd(&c->a_tail, (unsigned long long)ta);
      if (tv) vb = atomicAdd(&c->v_tail, (unsigned long long)tv);
    }
    ab = __shfl_sync(kFull, ab, 0);
    vb = __shfl_sync(kFull, vb, 0);
    auto give_agent = [&](unsigned long long at, uint32_t sl) {
      if constexpr (kTrack) {
        if (sl < d.cap_agents) __stcg(&d.node[sl].head, kFreeHead);
      }
      __stcg(d.afree + at % d.cap_agents, sl);
    };
    auto give_name = [&](unsigned long long at, uint32_t x) {
      if constexpr (kTrack) {
        if (x < d.cap_vars) __stcg(d.vown + x, kNoNet);
      }
      __stcg(d.vfree + at % d.cap_vars, x);
    };
#pragma unroll 1
    for (uint32_t j = (uint32_t)lane; j < ac; j += 32) give_agent(ab + j, W.astk[j]);
#pragma unroll 1
    for (uint32_t j = (uint32_t)lane; j < vc; j += 32) give_name(vb + j, W.vstk[j]);
    const uint32_t ex = inc - own;
#pragma unroll 1
    for (int j = 0; j < L.na; j++) give_agent(ab + ac + (ex & 0xFFFFu) + (uint32_t)j, W.ares[j][lane]);
#pragma unroll 1
    for (int j = 0; j < L.nv; j++) give_name(vb + vc + (ex >> 16) + (uint32_t)j, W.vres[j][lane]);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < d.n_tmpl; i += blockDim.x)
    if (hist[i]) atomicAdd(&d.rule_hist[i], (unsigned long long)hist[i]);
}

// Before an asynchronous launch: the current frontier's pairs are tickets
// 0 .. n0-1, already written; every other cell waits for its first ticket.
// Only cells an earlier launch used are rewritten (all of them once after a
// reset), so a short launch does not pay, or flush L2 with, the whole ring.
__global__ void k_async_fill(Dev d) {
  const Ctrl* c = d.ctrl;
  const uint32_t n0 = min(c->fcount[d.qcur], d.cap_pairs);
  const unsigned long long lim =
      c->qinit ? max(min(c->qdirty, (unsigned long long)d.cap_pairs), (unsigned long long)n0) : d.cap_pairs;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < lim;
       i += (unsigned long long)gridDim.x * blockDim.x)
    d.qseq[i] = i < n0 ? i + 1 : i;
}

// Before an asynchronous launch (one thread): publish the rings, make the
// current frontier the ticket queue.
__global__ void k_async_prep(Dev d) {
  Ctrl* c = d.ctrl;
  const uint32_t n0 = min(c->fcount[d.qcur], d.cap_pairs);
  if (c->a_head > c->a_pub) c->a_head = c->a_pub;
  c->a_pub = c->a_tail;
  if (c->v_head > c->v_pub) c->v_head = c->v_pub;
  c->v_pub = c->v_tail;
  c->qinit = 1;  // the fill before this launch initialised the ring
  c->q_head = 0;
  c->q_tail = n0;
  c->inflight = n0;
  c->astop = 0;
  c->quiesce = 0;
  c->aexit = 0;
  c->slice_t0 = 0;
  c->hit_slice = 0;
  c->done = 0;
  __threadfence();
}

// After an asynchronous launch (one thread): the pairs written back become
// the frontier of the other buffer.
__global__ void k_async_post(Dev d) {
  Ctrl* c = d.ctrl;
  const uint32_t cur = d.qcur;
  const uint32_t n = min(c->aexit, d.cap_pairs);
  // pops that found the ring empty went to the bump pointer but advanced the head
  if (c->a_head > c->a_pub) c->a_head = c->a_pub;
  if (c->v_head > c->v_pub) c->v_head = c->v_pub;
  c->fcount[cur] = 0;
  c->fcount[cur ^ 1u] = n;
  // cells this launch wrote: tickets below the tail (any after a fatal error)
  c->qdirty = c->fatal ? (unsigned long long)d.cap_pairs : min(c->q_tail, (unsigned long long)d.cap_pairs);
  c->step = c->step + 1;
  c->done = n == 0 || c->fatal != 0 ? 1u : 0u;
  if (c->live > c->peak_live) c->peak_live = c->live;
  __threadfence();
}

}  // namespace inet
