// Batch evaluation of a window of the space: materialise every output, or
// filter and compact the survivors in index order.
//
// A "group" is the n_codes consecutive points that share (model, factorisation,
// activation variant, tensor-axis variant).  A warp owns a contiguous run of the
// window's groups.  Within a group a lane owns up to four (Theta, Omega, G)
// triples.  A triple's bytes, priced communication, unpriced communication and
// host bytes are small-integer multiples of four per-group scalars (elements per
// position E, largest shard s, reconstruction unit u, ring volume x), and the
// integer coefficients depend only on the triple's modes and the model's byte
// widths -- so they are computed once per model and a group costs a few
// multiply-adds per triple.  The activation digit then adds one of NM
// per-group values.  Codes of a group run digit-major, triple-minor, so for a
// fixed digit the lanes write consecutive elements.  Materialise stages one
// output array of a group in shared memory and stores it with one bulk copy
// (shared -> global, asynchronous), so the warp computes the next array while
// the previous one drains.
//
// Compaction is count -> write.  The count pass (k_compact_count) never forms a point's
// bytes or flags: a lane owns a factorisation, and a point is one compare of a triple's own
// bytes with a per-(variant, digit) bound, masked by the digits the required flags allow.
// It leaves each group's offset in its run of factorisations, appends the factorisations that have
// survivors to a list, and its last block turns the runs' totals into offsets.  The write
// pass (k_write) takes the listed factorisations a block each, evaluates their groups from a common
// table of triples and places their survivors with ballot/popc prefix sums.  Output order is the
// index order, so the result is unique.
#include "ps_device.cuh"
#include "ps_internal.h"
#include "ps_lane.cuh"

namespace {

// Launch shapes (blocks of four warps).  Materialise is fastest with about one group per warp:
// short-lived blocks keep the warps of an SM at different stages (set-up, staging, draining
// stores) and the running warps write neighbouring stretches of every output array.
#ifndef EVAL_BULK_EVICT_FIRST
#define EVAL_BULK_EVICT_FIRST 1
#endif
#ifndef EVAL_GRID_PER_SM_MATERIALISE
#define EVAL_GRID_PER_SM_MATERIALISE 128
#endif
// (the write pass's shape: see k_write)
#ifndef EVAL_MIN_BLOCKS_WRITE
#define EVAL_MIN_BLOCKS_WRITE 5
#endif
#ifndef EVAL_GRID_PER_SM_WRITE
#define EVAL_GRID_PER_SM_WRITE 32
#endif
constexpr int THREADS = EVAL_THREADS;
constexpr int WARPS = THREADS / 32;
static_assert(THREADS % 128 == 0, "k_write gives every variant of a unit a warp: one, two or four");

// the flags that a composition has or has not, whatever its placements
constexpr u32 CV_BITS = PS_F_CV | PS_F_T_DIV_HEADS | PS_F_K_DIV_LAYERS | PS_F_TP_LE_MAX | PS_F_AXIS_FORM;

// internal bits of a triple's static description (above the public flag bits)
enum : u32 {
  X_HOST3 = 1u << 16,     // one of Theta, Omega, G is offloaded
  X_MO3 = 1u << 17,       // one of them is materialised or offloaded
  X_EXT0 = 1u << 18       // the data axis moves nothing beyond Theorem 2's terms
};

// static description of a triple when the data axis has several shard positions (d1 = false)
// or a single device (d1 = true)
__device__ __forceinline__ u32 triple_static(u32 th, u32 om, u32 gr, bool d1) {
  const bool on_shard = in_set(SET_UPDATE_ON_SHARD, om);
  const bool omega_full = (om == PS_MODE_R) || (d1 && in_set(SET_SHARDLIKE, om));
  const bool theta_avail = in_set(SET_THETA_ALWAYS, th) || (th == PS_MODE_S && d1) ||
                           (th == PS_MODE_M && omega_full);
  const bool grad_cover = d1 || on_shard || in_set(SET_GRAD_FULL, gr);
  const u32 seen = (1u << th) | (1u << om) | (1u << gr);
  // with one replica nothing moves; otherwise the unpriced data-axis terms are
  // non-zero exactly when their mode conditions hold (ring volume >= 1 element)
  const bool ext0 = d1 || !((th == PS_MODE_O) || (th == PS_MODE_R && on_shard) ||
                            in_set((1u << PS_MODE_SG) | SET_M_OR_O, gr) || om == PS_MODE_SG);
  return (theta_avail ? PS_F_THETA_AVAIL : 0) | (grad_cover ? PS_F_GRAD_COVER : 0) |
         (om != PS_MODE_M ? PS_F_SC : 0) | (((seen >> PS_MODE_O) & 1u) ? X_HOST3 : 0) |
         ((seen & SET_M_OR_O) ? X_MO3 : 0) | (ext0 ? X_EXT0 : 0);
}

// the same for a factorisation whose shards are all held by every device (several copies,
// one shard position): a shard is the whole tensor as on a single device, the gathers move
// nothing, but the gradient modes Theorem 2 does not price still move data
__device__ __forceinline__ u32 triple_static_all_copies(u32 th, u32 om, u32 gr) {
  const u32 st = triple_static(th, om, gr, true) & ~X_EXT0;
  return st | (in_set((1u << PS_MODE_SG) | SET_M_OR_O, gr) ? 0u : X_EXT0);
}

// Staging for the materialise path.  A warp builds one output array of one
// group (NC elements) in shared memory and hands it to the copy engine as a
// single bulk store (cp.async.bulk, shared -> global), then goes on computing the
// next array while the store drains; two staging buffers per warp alternate.
// A bulk store needs both addresses 16-byte aligned and a size that is a
// multiple of 16 bytes, while an output array is only aligned to its element and
// a group starts anywhere in it.  So element c of the group is staged at slot
// c + skew, where skew = (destination address / element size) mod (16 / element
// size): the shared and global addresses of every element then agree modulo 16,
// the elements before the first 16-byte boundary and after the last one (at
// most 16 / element size - 1 each) are written with plain stores, and everything
// between goes out as one bulk store.  Of a group at an edge of the window the part
// inside goes out the same way with 625 codes a group: a loop of its own for such groups, with its
// code fetched where a window is short and nothing hides that, took a window of 700 points
// 4.9 us with predicated stores and 5.9 with branches around them; staged it takes 3.9, and 2^25
// points 171 us instead of 179 and 176.  With up to 256 codes such groups take the plain loop: short
// windows 3.3 us instead of 3.6 (one behind the other 4.2 instead of 5.0 to 6.2), 2^24 points 99
// instead of 109, since the staged path knows its bounds when it is compiled.
template <int NC>
struct Stage {
  static constexpr int SLOTS = NC + 4;                                   // u64 slots, room for the skew
  static constexpr int BYTES = ((SLOTS * 8 + 127) / 128) * 128;          // one buffer
};

__device__ __forceinline__ u32 smem_addr(const void* p) { return (u32)__cvta_generic_to_shared(p); }

// lane 0 owns the warp's bulk stores: wait until at most `pending` of them still read shared memory
template <int PENDING>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(PENDING) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// All lanes have written element c of a group to buf[c + skew]; store those from lo to hi to dst[lo .. hi).
template <typename T>
__device__ __forceinline__ void warp_bulk_store(T* __restrict__ dst, const T* buf, int skew, int lo, int hi, int lane) {
  constexpr int PER16 = 16 / (int)sizeof(T);
  // make the lanes' shared-memory writes visible to the copy engine
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  dst += lo;
  buf += lo + skew;
  const int n = hi - lo;
  const int head = min(-(lo + skew) & (PER16 - 1), n);                   // elements before the first boundary
  const int body = ((n - head) / PER16) * PER16;
  if (lane < head) dst[lane] = buf[lane];
  const int tail = n - head - body;
  if (lane < tail) dst[head + body + lane] = buf[head + body + lane];
  if (lane == 0 && body > 0) {
#if EVAL_BULK_EVICT_FIRST
    // The output is written once and not read back by this kernel: with the evict-first
    // policy the lines leave the L2 as whole lines.  (Without a policy the same stores
    // cost 12 % more DRAM write traffic than the bytes stored.)
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;"
                 ::"l"(dst + head), "r"(smem_addr(buf + head)), "r"(body * (int)sizeof(T)), "l"(policy)
                 : "memory");
#else
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 ::"l"(dst + head), "r"(smem_addr(buf + head)), "r"(body * (int)sizeof(T))
                 : "memory");
#endif
  }
  if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

__device__ __forceinline__ void load_record(const SpaceDev& sp, u32 model, ModelRec& rec) {
  const uint4* src = reinterpret_cast<const uint4*>(&sp.recs[model]);
  uint4* dst = reinterpret_cast<uint4*>(&rec);
#pragma unroll
  for (int k = 0; k < 6; ++k) dst[k] = __ldg(src + k);   // the 96-byte record, 16 bytes at a time
}

// POW2: every degree of the space is a power of two (no division is compiled in)
template <int NM, bool POW2>
__global__ void __launch_bounds__(THREADS, EVAL_MIN_BLOCKS) k_eval(SpaceDev sp, EvalArgs a) {
  constexpr int N2 = NM * NM, N3 = NM * NM * NM, NC = N3 * NM;
  constexpr int R = (N3 + 31) / 32;
  // two staging buffers per warp
  extern __shared__ __align__(128) unsigned char stage_all[];
  unsigned char* const stage_warp = stage_all + (threadIdx.x >> 5) * 2 * Stage<NC>::BYTES;
  u32 stage_turn = 0;                                                     // which buffer is next
  const int lane = threadIdx.x & 31;
  const u32 warp_global = blockIdx.x * WARPS + (threadIdx.x >> 5);
  const u32 n_warps = gridDim.x * WARPS;
  // the window's groups are dealt evenly, a contiguous stretch per warp
  const u32 per_warp = (a.n_tiles + n_warps - 1) / n_warps;
  const u32 it_begin = (u32)min((u64)warp_global * per_warp, (u64)a.n_tiles);
  const u32 it_end = min(it_begin + per_warp, a.n_tiles);
  const u32 groups_per_model = sp.n_facts * sp.nvt;

  // with all five modes allowed digit d is mode d, and the compiler knows every
  // per-digit property below
  const u32 modemap = (NM == 5) ? 0x43210u : sp.modemap;
  // the lane's triples: modes never change
  u32 th[R], om[R], gr[R];
  bool live[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const u32 t = lane + 32 * r;
    live[r] = t < (u32)N3;
    const u32 tt = live[r] ? t : 0;
    th[r] = digit_mode(modemap, tt % NM);
    om[r] = digit_mode(modemap, (tt / NM) % NM);
    gr[r] = digit_mode(modemap, tt / N2);
  }
  // classes of the activation digit (Theorem 3: a replica needs its own activations)
  u32 own = 0, is_o = 0, not_mo = 0;
#pragma unroll
  for (int d = 0; d < NM; ++d) {
    const u32 ac = digit_mode(modemap, d);
    if (in_set(SET_ACT_OWN, ac)) own |= 1u << d;
    if (ac == PS_MODE_O) is_o |= 1u << d;
    if (!in_set(SET_M_OR_O, ac)) not_mo |= 1u << d;
  }

  // per model: widths and the coefficients that follow from them
  u32 model_cur = 0xffffffffu;
  ModelRec rec;
  u32 ka[R], kb[R], kc[R], kp[R], ke[R], kh[R];   // bytes (E, s, u), priced / unpriced comm (x), host (s)
  u32 st_many[R], st_one[R];                      // static description of a triple by the class of the factorisation
  u32 st_copies[POW2 ? 1 : R];                    // (the third class needs several copies of a shard)

  for (u32 it = it_begin; it < it_end; ++it) {
    const u64 g = a.first_group + it;
    // (a 32-bit division where the group number allows it: it is done once per group by every lane)
    const u32 model = (g >> 32) == 0 ? (u32)g / groups_per_model : (u32)(g / groups_per_model);
    const u32 gl = (u32)(g - (u64)model * groups_per_model);
    const u32 unit = gl / sp.nvt, vt = gl - unit * sp.nvt;
    const u32 v = vt / sp.nt, tau = vt - v * sp.nt;
    if (model != model_cur) {
      model_cur = model;
      load_record(sp, model, rec);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const u32 modes[3] = {th[r], om[r], gr[r]};
        const u32 width[3] = {rec.wT, rec.wO, rec.wG};
        const bool on_shard = in_set(SET_UPDATE_ON_SHARD, om[r]);
        u32 ca = 0, cb = 0, cc = 0;
#pragma unroll
        for (int s = 0; s < 3; ++s) {        // Theorem 1: R holds E, S and S* a shard, S* and M a unit
          if (modes[s] == PS_MODE_R) ca += width[s];
          if (in_set(SET_SHARDLIKE, modes[s])) cb += width[s];
          if (modes[s] == PS_MODE_SG) cc += width[s] * sp.sstar_units;   // one or two unit buffers
          if (modes[s] == PS_MODE_M) cc += width[s];
        }
        ka[r] = ca; kb[r] = cb; kc[r] = cc;
        // Theorem 2: all-reduce (2x) or reduce-scatter (1x) of G, two all-gathers of gathered
        // Theta for every micro-batch
        kp[r] = (th[r] == PS_MODE_SG ? 2 * sp.accum * rec.wT : 0) +
                (gr[r] == PS_MODE_R ? 2 * rec.wG : (gr[r] == PS_MODE_S ? rec.wG : 0));
        // what the execution model moves beyond that
        u32 e = 0;
        if (th[r] == PS_MODE_O) e += 2 * sp.accum * rec.wT;
        if (th[r] == PS_MODE_R && on_shard) e += rec.wT;
        if (om[r] == PS_MODE_SG) e += rec.wO;
        if (gr[r] == PS_MODE_SG) e += 2 * rec.wG;
        if (gr[r] == PS_MODE_M) e += (on_shard ? 1 : 2) * rec.wG;
        if (gr[r] == PS_MODE_O) e += rec.wG;
        ke[r] = e;
        kh[r] = (th[r] == PS_MODE_O ? (2 * sp.accum + 1) * rec.wT : 0) + (om[r] == PS_MODE_O ? 2 * rec.wO : 0) +
                (gr[r] == PS_MODE_O ? 2 * rec.wG : 0);
        st_many[r] = triple_static(th[r], om[r], gr[r], false);
        st_one[r] = triple_static(th[r], om[r], gr[r], true);
        if (!POW2) st_copies[r] = triple_static_all_copies(th[r], om[r], gr[r]);
      }
    }

    // ---- per group: shard quantities (all divisions), activation bytes per digit
    const Fact f = sp.facts[unit];
    const u32 repl = POW2 ? 1u : sp.repl;        // the power-of-two case is compiled for one copy of every shard
    const Pow2 p2 = POW2 ? pow2_of(f) : pow2_of(f, repl);
    const UnitBase ub = POW2 ? unit_base_pow2_one_copy(rec, f, p2, sp.tp_max_valid, true)
                        : p2.all ? unit_base_pow2(rec, f, p2, sp.tp_max_valid, true)
                                 : unit_base(rec, f, sp.tp_max_valid, true, repl);
    ModelRec variant = rec;                      // (an index into the record would put all of it into local memory)
    variant.A[0] = __ldg(&sp.recs[model].A[v]); variant.UA[0] = __ldg(&sp.recs[model].UA[v]);
    const ActBase ab = POW2 ? act_base_pow2_one_copy(variant, p2, 0, tau)
                       : p2.all ? act_base_pow2(variant, p2, 0, tau) : act_base(variant, f, 0, tau, ub.G);
    const u64 c_axis = model_axis_traffic(rec, f, ub, tau, sp.tp_coll, sp.accum);
    u64 act[NM];
#pragma unroll
    for (int d = 0; d < NM; ++d) act[d] = mu_elems(digit_mode(modemap, d), ab.EA, ab.shA, ab.uA, sp.sstar_units);
    const u64 act_host = 2 * ab.EA * sp.accum;
    const u32 avail = ub.d1 ? ((1u << NM) - 1u) : own;     // digits with PS_F_ACT_AVAIL

    u64 mem3[R], paper3[R], ext3[R], host3[R];
    u32 st[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      mem3[r] = mad_small(ub.E2, ka[r], mad_small(ub.sh, kb[r], mad_small(ub.u, kc[r], 0)));
      paper3[r] = mad_small(ub.x, kp[r], 0);
      ext3[r] = mad_small(ub.x, ke[r], 0);
      if (repl > 1) {
        // several copies of every shard: reducing gradients to shards costs x2 more, an
        // all-reduce over all devices x3 more (both zero with one copy)
        const bool on_shard = in_set(SET_UPDATE_ON_SHARD, om[r]);
        paper3[r] += (u64)rec.wG * ((gr[r] == PS_MODE_S ? ub.x2 : 0) + (gr[r] == PS_MODE_R ? ub.x3 : 0));
        ext3[r] += (u64)rec.wG * (((gr[r] == PS_MODE_SG || gr[r] == PS_MODE_O || (gr[r] == PS_MODE_M && on_shard)) ? ub.x2 : 0) +
                                  ((gr[r] == PS_MODE_M && !on_shard) ? ub.x3 : 0));
      }
      host3[r] = mad_small(ub.sh, kh[r], 0);
      // (with one copy of every shard a factorisation is sharded or a single device)
      if (POW2) st[r] = ub.d1 ? st_one[r] : st_many[r];
      else st[r] = ub.cls == CLS_SHARDED ? st_many[r] : (ub.cls == CLS_ONE_DEVICE ? st_one[r] : st_copies[POW2 ? 0 : r]);
    }

    // ---- the group's points inside the window
    const u64 group_first = g * NC;
    const u32 code_lo = a.first > group_first ? (u32)(a.first - group_first) : 0u;
    const u64 window_end = a.first + a.count;
    const u32 code_hi = window_end < group_first + NC ? (u32)(window_end - group_first) : (u32)NC;
    const u64 out_base = group_first - a.first;          // (wraps when the group starts before the window; only used with code >= code_lo)

    // flags of a point = what the triple fixes | what the digit fixes | what needs both:
    //   gradient integrity needs the triple's two availability bits and the digit's,
    //   "paper priced" needs a triple without M/O and unpriced traffic and a digit without M/O
    u32 fl_base[R], fl_gi[R], fl_priced[R];
    constexpr u32 both = PS_F_THETA_AVAIL | PS_F_GRAD_COVER;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      fl_base[r] = ub.cv | (st[r] & (both | PS_F_SC)) | ((st[r] & X_HOST3) ? PS_F_USES_HOST : 0);
      fl_gi[r] = ((st[r] & both) == both) ? PS_F_GI : 0;
      fl_priced[r] = ((st[r] & (X_EXT0 | X_MO3)) == X_EXT0) ? PS_F_PAPER_PRICED : 0;
    }
    const bool all_out = a.out.mem && a.out.comm_paper && a.out.comm_ext && a.out.host && a.out.flags;

    if (all_out && (NM == 5 || (code_lo == 0 && code_hi == (u32)NC))) {
      // one output array at a time: stage the group's NC values, hand them to the copy engine
#pragma unroll
      for (int which = 0; which < 5; ++which) {
        u64* const stage = reinterpret_cast<u64*>(stage_warp + (stage_turn & 1u) * Stage<NC>::BYTES);
        u32* const stage32 = reinterpret_cast<u32*>(stage);
        ++stage_turn;
        u64* const dst64 = (which == 0 ? a.out.mem : which == 1 ? a.out.comm_paper
                            : which == 2 ? a.out.comm_ext : a.out.host) + out_base;
        u32* const dst32 = a.out.flags + out_base;
        const int skew = which < 4 ? (int)((reinterpret_cast<uintptr_t>(dst64) >> 3) & 1)
                                   : (int)((reinterpret_cast<uintptr_t>(dst32) >> 2) & 3);
        // the store that used this buffer two arrays ago must have read it completely
        if (lane == 0) bulk_wait_read<1>();
        __syncwarp();
#pragma unroll
        for (int d = 0; d < NM; ++d) {
          const bool d_avail = (avail >> d) & 1u, d_off = (is_o >> d) & 1u, d_notmo = (not_mo >> d) & 1u;
          const u32 fl_digit = (d_avail ? PS_F_ACT_AVAIL : 0) | (d_off ? PS_F_USES_HOST : 0);
          const u32 gi_mask = d_avail ? ~0u : 0u, priced_mask = d_notmo ? ~0u : 0u;
          const u64 host_add = d_off ? act_host : 0;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (!live[r]) continue;
            const u32 slot = lane + 32 * r + d * N3 + skew;
            if (which == 0) stage[slot] = mem3[r] + act[d];
            else if (which == 1) stage[slot] = paper3[r];
            else if (which == 2) stage[slot] = ext3[r] + c_axis;
            else if (which == 3) stage[slot] = host3[r] + host_add;
            else stage32[slot] = fl_base[r] | fl_digit | (fl_gi[r] & gi_mask) | (fl_priced[r] & priced_mask);
          }
        }
        if (which < 4) warp_bulk_store(dst64, stage, skew, code_lo, code_hi, lane);
        else warp_bulk_store(dst32, stage32, skew, code_lo, code_hi, lane);
      }
      continue;
    }

    // (some of the outputs only; with up to four modes the groups at the window's edges)
#pragma unroll 1
    for (int d = 0; d < NM; ++d) {
      const u64 act_d = mu_elems(digit_mode(modemap, d), ab.EA, ab.shA, ab.uA, sp.sstar_units);
      const bool d_avail = (avail >> d) & 1u, d_off = (is_o >> d) & 1u, d_notmo = (not_mo >> d) & 1u;
      const u32 fl_digit = (d_avail ? PS_F_ACT_AVAIL : 0) | (d_off ? PS_F_USES_HOST : 0);
      const u32 gi_mask = d_avail ? ~0u : 0u, priced_mask = d_notmo ? ~0u : 0u;
      const u64 host_add = d_off ? act_host : 0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const u32 code = lane + 32 * r + d * N3;
        if (!(live[r] && code >= code_lo && code < code_hi)) continue;
        const u64 o = out_base + code;
        if (a.out.mem) a.out.mem[o] = mem3[r] + act_d;
        if (a.out.comm_paper) a.out.comm_paper[o] = paper3[r];
        if (a.out.comm_ext) a.out.comm_ext[o] = ext3[r] + c_axis;
        if (a.out.host) a.out.host[o] = host3[r] + host_add;
        if (a.out.flags) a.out.flags[o] = fl_base[r] | fl_digit | (fl_gi[r] & gi_mask) | (fl_priced[r] & priced_mask);
      }
    }
  }
  // the staging buffers must outlive the bulk stores that read them
  if (lane == 0) bulk_wait_all();
}

// ------------------------------------------------------------------ compaction: write
// A unit's triples as its groups share them: bytes, traffic on the data axis, host bytes and flags.
template <int NM>
struct UnitTable {
  static constexpr int N3 = NM * NM * NM;
  u64 mem[N3], paper[N3], ext[N3], host[N3];
  u32 flags[N3];              // high half: the bits that need the triple and the digit
};

// A block takes the listed units in turns of as many as give each of its warps a group: the warps
// of a unit make its table of triples together, a thread a triple, and then each evaluates its
// group (activation and tensor-axis variant) from that table and places its survivors by ballot and
// popc.  What bounds it: the set-up of a group and its stores.  With the triples' coefficients and
// figures formed by every warp for itself, four triples a lane, 2^23 points with half of them
// surviving took 74 us and 2^25 with one in two thousand 32, with the count pass; like this 68 and 28,
// launched before the count pass has ended 67 and 26.5.  Five blocks are resident: with four 2^25 points that
// all survive take 305 us instead of 316, half of 2^23 67.7 instead of 61.2 (256 codes a group) and 48.4 instead of
// 45.1 (625).  The grid: see launch_write_p.
template <int NM, bool POW2>
__global__ void __launch_bounds__(THREADS, EVAL_MIN_BLOCKS_WRITE) k_write(const __grid_constant__ SpaceDev sp,
                                                                         const __grid_constant__ EvalArgs a) {
  constexpr int N2 = NM * NM, N3 = NM * NM * NM, NC = N3 * NM, R = (N3 + 31) / 32;
  __shared__ UnitTable<NM> tables[WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 nvt = sp.nvt, teams = WARPS / nvt, team = warp / nvt, vt = warp - team * nvt;   // nvt: 1, 2 or 4
  const u32 v = vt / sp.nt, tau = vt - v * sp.nt;
  UnitTable<NM>& table = tables[team];
  const u32 modemap = (NM == 5) ? 0x43210u : sp.modemap;
  u32 own = 0;                                             // Theorem 3: a replica needs its own activations
#pragma unroll
  for (int d = 0; d < NM; ++d)
    if (in_set(SET_ACT_OWN, digit_mode(modemap, d))) own |= 1u << d;
  asm volatile("griddepcontrol.wait;" ::: "memory");      // the count pass has ended, nothing of it is read before
  const u32 n_listed = *a.n_listed;
  for (u64 first = (u64)blockIdx.x * teams; first < n_listed; first += (u64)gridDim.x * teams) {
    const bool have = first + team < n_listed;
    const u32 place = a.nonempty[have ? first + team : first];
    const u64 ug = a.first_unit + place;
    const u32 model = (ug >> 32) == 0 ? (u32)ug / sp.n_facts : (u32)(ug / sp.n_facts);
    ModelRec rec;
    load_record(sp, model, rec);
    if (v) { rec.A[0] = rec.A[1]; rec.UA[0] = rec.UA[1]; }  // (the warp's variant; an index known here keeps the record in registers)
    const Fact f = sp.facts[(u32)(ug - (u64)model * sp.n_facts)];
    const u32 repl = POW2 ? 1u : sp.repl;
    const Pow2 p2 = POW2 ? pow2_of(f) : pow2_of(f, repl);
    const UnitBase ub = POW2 ? unit_base_pow2_one_copy(rec, f, p2, sp.tp_max_valid, true)
                        : p2.all ? unit_base_pow2(rec, f, p2, sp.tp_max_valid, true)
                                 : unit_base(rec, f, sp.tp_max_valid, true, repl);
    __syncthreads();                                       // (the tables of the turn before have been read)
    for (u32 t = tid - team * 32 * nvt; t < (u32)N3; t += 32 * nvt) {
      const u32 th = digit_mode(modemap, t % NM), om = digit_mode(modemap, (t / NM) % NM), gr = digit_mode(modemap, t / N2);
      const u32 modes[3] = {th, om, gr}, width[3] = {rec.wT, rec.wO, rec.wG};
      const bool on_shard = in_set(SET_UPDATE_ON_SHARD, om);
      u32 ca = 0, cb = 0, cc = 0;
#pragma unroll
      for (int st = 0; st < 3; ++st) {        // Theorem 1: R holds E, S and S* a shard, S* and M a unit
        if (modes[st] == PS_MODE_R) ca += width[st];
        if (in_set(SET_SHARDLIKE, modes[st])) cb += width[st];
        if (modes[st] == PS_MODE_SG) cc += width[st] * sp.sstar_units;
        if (modes[st] == PS_MODE_M) cc += width[st];
      }
      // Theorem 2, and what the execution model moves beyond it (as in k_eval)
      const u32 kp = (th == PS_MODE_SG ? 2 * sp.accum * rec.wT : 0) +
                     (gr == PS_MODE_R ? 2 * rec.wG : (gr == PS_MODE_S ? rec.wG : 0));
      u32 ke = 0;
      if (th == PS_MODE_O) ke += 2 * sp.accum * rec.wT;
      if (th == PS_MODE_R && on_shard) ke += rec.wT;
      if (om == PS_MODE_SG) ke += rec.wO;
      if (gr == PS_MODE_SG) ke += 2 * rec.wG;
      if (gr == PS_MODE_M) ke += (on_shard ? 1 : 2) * rec.wG;
      if (gr == PS_MODE_O) ke += rec.wG;
      const u32 kh = (th == PS_MODE_O ? (2 * sp.accum + 1) * rec.wT : 0) + (om == PS_MODE_O ? 2 * rec.wO : 0) +
                     (gr == PS_MODE_O ? 2 * rec.wG : 0);
      u64 paper = mad_small(ub.x, kp, 0), ext = mad_small(ub.x, ke, 0);
      if (repl > 1) {
        paper += (u64)rec.wG * ((gr == PS_MODE_S ? ub.x2 : 0) + (gr == PS_MODE_R ? ub.x3 : 0));
        ext += (u64)rec.wG * (((gr == PS_MODE_SG || gr == PS_MODE_O || (gr == PS_MODE_M && on_shard)) ? ub.x2 : 0) +
                              ((gr == PS_MODE_M && !on_shard) ? ub.x3 : 0));
      }
      table.mem[t] = mad_small(ub.E2, ca, mad_small(ub.sh, cb, mad_small(ub.u, cc, 0)));
      table.paper[t] = paper;
      table.ext[t] = ext;
      table.host[t] = mad_small(ub.sh, kh, 0);
      const u32 st = !POW2 && ub.cls == CLS_ALL_COPIES ? triple_static_all_copies(th, om, gr) : triple_static(th, om, gr, ub.d1);
      constexpr u32 both = PS_F_THETA_AVAIL | PS_F_GRAD_COVER;
      table.flags[t] = ub.cv | PS_F_FEASIBLE | (st & (both | PS_F_SC)) | ((st & X_HOST3) ? PS_F_USES_HOST : 0) |
                       ((st & both) == both ? PS_F_GI << 16 : 0) |
                       ((st & (X_EXT0 | X_MO3)) == X_EXT0 ? PS_F_PAPER_PRICED << 16 : 0);
    }
    __syncthreads();
    const u64 g = ug * nvt + vt, tile = g - a.first_group;               // (wraps before the window)
    if (!have || tile >= a.n_tiles) continue;
    // ---- the warp's group: what its variant and the digits add
    const ActBase ab = POW2 ? act_base_pow2_one_copy(rec, p2, 0, tau)
                       : p2.all ? act_base_pow2(rec, p2, 0, tau) : act_base(rec, f, 0, tau, ub.G);
    const u64 c_axis = model_axis_traffic(rec, f, ub, tau, sp.tp_coll, sp.accum);
    const u64 act_host = 2 * ab.EA * sp.accum;
    const u32 avail = ub.d1 ? ((1u << NM) - 1u) : own;                    // digits with PS_F_ACT_AVAIL
    const u64 group_first = g * NC, window_end = a.first + a.count;
    const u32 code_lo = a.first > group_first ? (u32)(a.first - group_first) : 0u;
    const u32 code_hi = window_end < group_first + NC ? (u32)(window_end - group_first) : (u32)NC;
    // survivors before this group: those of the runs before its run, and of the run's earlier groups
    u64 at = a.run_offset[place / EVAL_RUN_UNITS] + a.group_offset[tile];
    u64 mem3[R], host3[R];
    u32 flags3[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int t = min(lane + 32 * r, N3 - 1);
      mem3[r] = table.mem[t]; host3[r] = table.host[t]; flags3[r] = table.flags[t];
    }
#pragma unroll
    for (int d = 0; d < NM; ++d) {
      const u32 mode = digit_mode(modemap, d);
      const u64 act = mu_elems(mode, ab.EA, ab.shA, ab.uA, sp.sstar_units), host_add = mode == PS_MODE_O ? act_host : 0;
      const u32 with = (((avail >> d) & 1u) ? PS_F_GI : 0) | (!in_set(SET_M_OR_O, mode) ? PS_F_PAPER_PRICED : 0);
      const u32 alone = (((avail >> d) & 1u) ? PS_F_ACT_AVAIL : 0) | (mode == PS_MODE_O ? PS_F_USES_HOST : 0);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const u32 t = lane + 32 * r, code = t + d * N3;
        const u64 mem = mem3[r] + act, host = host3[r] + host_add;
        const u32 fl = (flags3[r] & 0xffffu) | alone | ((flags3[r] >> 16) & with);
        const bool pass = t < (u32)N3 && code >= code_lo && code < code_hi && mem <= a.cap_bytes && host <= a.host_cap &&
                          (fl & a.require_flags) == a.require_flags;
        const u32 votes = __ballot_sync(0xffffffffu, pass);
        if (pass) {
          const u64 o = at + __popc(votes & ((1u << lane) - 1u));
          if (a.idx_out) a.idx_out[o] = group_first + code;
          if (a.out.mem) a.out.mem[o] = mem;
          if (a.out.comm_paper) a.out.comm_paper[o] = table.paper[t];
          if (a.out.comm_ext) a.out.comm_ext[o] = table.ext[t] + c_axis;
          if (a.out.host) a.out.host[o] = host;
          if (a.out.flags) a.out.flags[o] = fl;
        }
        at += __popc(votes);
      }
    }
  }
}

// ------------------------------------------------------------------ compaction: count
// bytes of a state under a mode (the same for every lane) in the lane's unit
template <int NM, typename T, bool HOST_LIMITED>
__device__ __forceinline__ double state_bytes(const LaneUnit<NM, T, HOST_LIMITED>& lu, u32 mode, double width, u32 sstar_units) {
  if (mode == PS_MODE_R) return width * lu.E;
  if (mode == PS_MODE_S) return width * lu.s;
  if (mode == PS_MODE_SG) return width * (lu.s + sstar_units * lu.u);
  if (mode == PS_MODE_M) return width * lu.u;
  return 0.0;
}

// One block per run of 32 consecutive units; a lane owns a unit, the warps share the
// (Theta, Omega) pairs.  What bounds it: the fp64 pipe (a compare per point), and for small
// windows the chain of a unit's set-up.  As one warp per run of groups, its lanes the
// triples, it took 21 us for 2^25 points and was followed by a scan kernel of 3 us; like
// this it takes 12.
constexpr int COUNT_WARPS = 8;
template <int NM, typename T, bool HOST_LIMITED>
__global__ void __launch_bounds__(COUNT_WARPS * 32, 2) k_compact_count(SpaceDev sp, EvalArgs a) {
  constexpr int N2 = NM * NM, N3 = NM * NM * NM, NC = N3 * NM;
  __shared__ unsigned char allowed_of[3][N3];
  __shared__ u32 cnt[4][32];
  __shared__ u64 warp_sum[COUNT_WARPS];
  __shared__ u64 carry;
  __shared__ u32 last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;");     // the write pass waits for this grid's end itself
  const u32 modemap = (NM == 5) ? 0x43210u : sp.modemap;
  const u32 req = a.require_flags;
  const u32 req_cv = req & CV_BITS;
  // capacities as exclusive bounds (memory stays below 2^61)
  const u64 cap_x = min(a.cap_bytes, (u64)1 << 62) + 1;
  const u64 host_x = min(a.host_cap, HOST_BYTES_END) + 1;
  constexpr u32 all = (1u << NM) - 1u;
  u32 own = 0, is_o = 0, not_mo = 0;
#pragma unroll
  for (int d = 0; d < NM; ++d) {
    const u32 ac = digit_mode(modemap, d);
    if (in_set(SET_ACT_OWN, ac)) own |= 1u << d;
    if (ac == PS_MODE_O) is_o |= 1u << d;
    if (!in_set(SET_M_OR_O, ac)) not_mo |= 1u << d;
  }
  if (tid < 128) cnt[warp][lane] = 0;
  for (int t = tid; t < N3; t += COUNT_WARPS * 32) {
    const u32 th = digit_mode(modemap, t % NM), om = digit_mode(modemap, (t / NM) % NM), gr = digit_mode(modemap, t / N2);
    allowed_of[CLS_SHARDED][t] = (unsigned char)allowed_act_digits(triple_bits(th, om, gr, CLS_SHARDED), req, all, own, is_o, not_mo);
    allowed_of[CLS_ONE_DEVICE][t] = (unsigned char)allowed_act_digits(triple_bits(th, om, gr, CLS_ONE_DEVICE), req, all, all, is_o, not_mo);
    allowed_of[CLS_ALL_COPIES][t] = (unsigned char)allowed_act_digits(triple_bits(th, om, gr, CLS_ALL_COPIES), req, all, all, is_o, not_mo);
  }
  // ---- the lane's unit
  const u32 k = blockIdx.x * EVAL_RUN_UNITS + lane;
  const bool have = k < a.n_units;
  const u64 unit_global = a.first_unit + min(k, a.n_units - 1);
  const u32 model = (u32)(unit_global / sp.n_facts);
  ModelRec rec;
  load_record(sp, model, rec);
  const Fact f = sp.facts[(u32)(unit_global - (u64)model * sp.n_facts)];
  const UnitBase ub = unit_of(sp, rec, f);
  LaneUnit<NM, T, HOST_LIMITED> lu;
  lu.load(sp, rec, f, ub, modemap, cap_x, host_x, have && (ub.cv & req_cv) == req_cv);
  const T host_room = as<T>(host_x);
  const double wT = rec.wT, wO = rec.wO, wG = rec.wG;
  const T host_T = as<T>((2 * sp.accum + 1) * rec.wT), host_O = as<T>(2 * rec.wO);
  const unsigned char* const allowed_here = allowed_of[lu.shift >> 3];
  __syncthreads();
  float n[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const u32 pairs = __any_sync(0xffffffffu, lu.allowed != 0) ? N2 : 0;     // (a run without a unit that can pass is not walked)
#pragma unroll 1
  for (u32 p = warp * pairs / COUNT_WARPS; p < (warp + 1) * pairs / COUNT_WARPS; ++p) {
    const u32 th = p / NM, om = p - th * NM, th_mode = digit_mode(modemap, th), om_mode = digit_mode(modemap, om);
    const double to_mem = state_bytes(lu, th_mode, wT, sp.sstar_units) + state_bytes(lu, om_mode, wO, sp.sstar_units);
    const T to_host = (th_mode == PS_MODE_O ? host_T * lu.shard : T(0)) + (om_mode == PS_MODE_O ? host_O * lu.shard : T(0));
#pragma unroll
    for (int gr = 0; gr < NM; ++gr) {
      const double m = to_mem + lu.gr_mem[gr];
      u32 allowed = allowed_here[th + NM * om + N2 * gr] & lu.allowed;
      T h = to_host;
      if (HOST_LIMITED) {
        if (digit_mode(modemap, gr) == PS_MODE_O) h += lu.gr_host;
        if (!(h < host_room)) allowed = 0;
      }
#pragma unroll
      for (int d = 0; d < NM; ++d) {
        if (HOST_LIMITED && digit_mode(modemap, d) == PS_MODE_O) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            n[q] += ((allowed >> d) & 1u) && m < lu.bounds(d)[q] && h < lu.host_bound[q] ? 1.0f : 0.0f;
        } else {
          count_variants(n, m, lu.bounds(d), allowed & (1u << d));
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (n[q] != 0.0f) atomicAdd(&cnt[q][lane], (u32)n[q]);
  __syncthreads();

  // ---- the groups at the window's edges again, code by code: a warp each, from the figures
  // that the lane owning the unit holds
  if (warp < 2) {
    const u64 window_end = a.first + a.count;
    const u64 g = warp == 0 ? a.first / NC : (window_end - 1) / NC;
    const u64 ug = g / sp.nvt, u = ug - a.first_unit;
    const u64 group_first = g * NC;
    const u32 code_lo = a.first > group_first ? (u32)(a.first - group_first) : 0u;
    const u32 code_hi = window_end < group_first + NC ? (u32)(window_end - group_first) : (u32)NC;
    if (u / EVAL_RUN_UNITS == blockIdx.x && !(warp == 1 && g == a.first / NC) && (code_lo != 0 || code_hi != (u32)NC)) {
      const int src = (int)(u % EVAL_RUN_UNITS);
      const u32 vt = (u32)(g - ug * sp.nvt), v = vt / sp.nt, tau = vt - v * sp.nt, slot = 2 * v + tau;
      const double E = __shfl_sync(0xffffffffu, lu.E, src), S = __shfl_sync(0xffffffffu, lu.s, src), U = __shfl_sync(0xffffffffu, lu.u, src);
      const double W[3] = {__shfl_sync(0xffffffffu, wT, src), __shfl_sync(0xffffffffu, wO, src),
                           __shfl_sync(0xffffffffu, wG, src)};
      const T shard = __shfl_sync(0xffffffffu, lu.shard, src);
      const u32 shift = __shfl_sync(0xffffffffu, lu.shift, src), counted = __shfl_sync(0xffffffffu, lu.allowed, src);
      double bound[NM];
      T host_bound = T(0);
#pragma unroll
      for (u32 q = 0; q < 4; ++q)
        if (q == slot) {
#pragma unroll
          for (int d = 0; d < NM; ++d) bound[d] = __shfl_sync(0xffffffffu, lu.bounds(d)[q], src);
          if (HOST_LIMITED) host_bound = __shfl_sync(0xffffffffu, lu.host_bound[q], src);
        }
      u32 survivors = 0;
      for (u32 code = code_lo + lane; code < code_hi; code += 32) {
        const u32 t = code % N3, digit = code / N3;
        const u32 modes[3] = {digit_mode(modemap, t % NM), digit_mode(modemap, (t / NM) % NM), digit_mode(modemap, t / N2)};
        double m = 0.0;
        T h = T(0);
#pragma unroll
        for (int st = 0; st < 3; ++st) {
          const double held = (modes[st] == PS_MODE_R ? E : in_set(SET_SHARDLIKE, modes[st]) ? S : 0.0) +
                              (modes[st] == PS_MODE_SG ? sp.sstar_units * U : modes[st] == PS_MODE_M ? U : 0.0);
          m += W[st] * held;
          if (modes[st] == PS_MODE_O) h += as<T>((st == 0 ? 2 * sp.accum + 1 : 2) * (u32)W[st]) * shard;
        }
        bool fits = false;
#pragma unroll
        for (int d = 0; d < NM; ++d)
          if (digit == (u32)d) fits = m < bound[d];
        if (HOST_LIMITED) fits = fits && h < host_room && (digit_mode(modemap, digit) != PS_MODE_O || h < host_bound);
        if (fits && ((allowed_of[shift >> 3][t] & counted) >> digit) & 1u) ++survivors;
      }
      survivors = __reduce_add_sync(0xffffffffu, survivors);
      if (lane == 0) cnt[slot][src] = survivors;
    }
  }
  __syncthreads();
  if (warp == 0) {
    // ---- offsets inside the run, and the list of units with survivors
    u32 mine = 0, filled = 0, c[4];
    bool inside[4];
    u64 at[4];
#pragma unroll
    for (u32 q = 0; q < 4; ++q) {
      const u32 v = q >> 1, tau = q & 1;
      at[q] = unit_global * sp.nvt + v * sp.nt + tau - a.first_group;      // (wraps before the window)
      inside[q] = have && v < sp.nv && tau < sp.nt && at[q] < a.n_tiles;
      c[q] = inside[q] ? cnt[q][lane] : 0;
      mine += c[q];
    }
    filled = mine ? 1u : 0u;
    u32 incl = mine, listed = filled;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 up = __shfl_up_sync(0xffffffffu, incl, o), up2 = __shfl_up_sync(0xffffffffu, listed, o);
      if (lane >= o) { incl += up; listed += up2; }
    }
    u32 base = 0;
    if (lane == 31 && listed) base = atomicAdd(a.n_nonempty, listed);
    base = __shfl_sync(0xffffffffu, base, 31) + listed - filled;
    u32 before = incl - mine;
#pragma unroll
    for (u32 q = 0; q < 4; ++q) {
      if (inside[q]) a.group_offset[at[q]] = before;
      before += c[q];
    }
    if (filled) a.nonempty[base] = k;
    if (lane == 31) a.run_offset[blockIdx.x] = incl;
    // ---- the block that finishes last turns the runs' totals into offsets
    __threadfence();
    __syncwarp();
    if (lane == 0) last = atomicAdd(a.blocks_done, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) carry = 0;
  constexpr int SCAN_ITEMS = 4;
  volatile u64* const runs = a.run_offset;
  for (u64 tile = 0; tile < a.n_runs; tile += COUNT_WARPS * 32 * SCAN_ITEMS) {
    __syncthreads();
    const u64 i0 = tile + SCAN_ITEMS * tid;
    u64 c[SCAN_ITEMS], mine = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) { c[j] = i0 + j < a.n_runs ? runs[i0 + j] : 0; mine += c[j]; }
    u64 incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    u64 before = carry;                          // everything before this warp
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
    u64 run = before + incl - mine;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
      if (i0 + j < a.n_runs) runs[i0 + j] = run;
      run += c[j];
    }
    __syncthreads();
    if (tid == COUNT_WARPS * 32 - 1) carry = before + incl;
  }
  __syncthreads();
  if (tid == 0) {
    *a.n_out = carry;
    *a.n_listed = *static_cast<volatile u32*>(a.n_nonempty);
    *a.n_nonempty = 0;            // the next compaction's list starts empty
    *a.blocks_done = 0;
  }
}

int multiprocessors() {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <int NM, bool POW2>
cudaError_t launch_eval_p(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  // one warp per run of groups; enough blocks to fill the GPU, no more than groups
  const unsigned needed = (a.n_tiles + WARPS - 1) / WARPS;
  const unsigned most = (unsigned)multiprocessors() * EVAL_GRID_PER_SM_MATERIALISE;
  const unsigned blocks = needed < most ? needed : most;
  const size_t smem = (size_t)WARPS * 2 * Stage<NM * NM * NM * NM>::BYTES;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_eval<NM, POW2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  k_eval<NM, POW2><<<blocks, THREADS, smem, stream>>>(sp, a);
  return cudaGetLastError();
}

template <int NM, bool POW2>
cudaError_t launch_write_p(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  // 32 blocks an SM, not more than there are units; 64 where there are more units than that and the filter requires
  // nothing of the composition, so that most of them may be listed.  Short blocks keep the warps at
  // different stages, but those that find nothing left to do cost a launch.  With 16, 32 and 64: 2^25 points that all
  // survive 337, 324 and 316 us (five modes; 2^24 in four modes 196, 184 and 177), half of 2^23 59.9, 58.4 and
  // 61.2, one of 2^25 in two thousand (valid placements) 25.1, 25.1 and 27.1.
  const unsigned teams = WARPS / sp.nvt, needed = (a.n_units + teams - 1) / teams;
  const unsigned per_sm = (unsigned)multiprocessors() * EVAL_GRID_PER_SM_WRITE;
  const unsigned most = needed > 2 * per_sm && (a.require_flags & CV_BITS) == 0 ? 2 * per_sm : per_sm;
  // enqueued so that its blocks are there when the count pass's last ones end
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t config = {};
  config.gridDim = dim3(needed < most ? needed : most);
  config.blockDim = dim3(THREADS);
  config.stream = stream;
  config.attrs = &early;
  config.numAttrs = 1;
  return cudaLaunchKernelEx(&config, k_write<NM, POW2>, sp, a);
}

template <int NM>
cudaError_t launch_materialise_t(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  return (sp.all_pow2 && sp.repl == 1) ? launch_eval_p<NM, true>(sp, a, stream) : launch_eval_p<NM, false>(sp, a, stream);
}
template <int NM>
cudaError_t launch_write_t(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  return (sp.all_pow2 && sp.repl == 1) ? launch_write_p<NM, true>(sp, a, stream) : launch_write_p<NM, false>(sp, a, stream);
}

}  // namespace

void eval_plan_runs(const SpaceDev& sp, EvalArgs& a) {
  a.first_unit = a.first_group / sp.nvt;
  a.n_units = (u32)((a.first_group + a.n_tiles - 1) / sp.nvt - a.first_unit + 1);
  a.n_runs = (a.n_units + EVAL_RUN_UNITS - 1) / EVAL_RUN_UNITS;
}

cudaError_t launch_eval_materialise(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  switch (sp.nm) {
    case 1: return launch_materialise_t<1>(sp, a, stream);
    case 2: return launch_materialise_t<2>(sp, a, stream);
    case 3: return launch_materialise_t<3>(sp, a, stream);
    case 4: return launch_materialise_t<4>(sp, a, stream);
    default: return launch_materialise_t<5>(sp, a, stream);
  }
}
template <int NM>
static cudaError_t launch_count_t(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  // every byte count exact in a double
  if (sp.all_small && a.cap_bytes < ((u64)1 << 53) - 1) {
    if (NM < 4 || a.host_cap < HOST_BYTES_END) k_compact_count<NM, double, true><<<a.n_runs, COUNT_WARPS * 32, 0, stream>>>(sp, a);
    else k_compact_count<NM, double, NM < 4><<<a.n_runs, COUNT_WARPS * 32, 0, stream>>>(sp, a);
  } else {
    k_compact_count<NM, u64, true><<<a.n_runs, COUNT_WARPS * 32, 0, stream>>>(sp, a);
  }
  return cudaGetLastError();
}
cudaError_t launch_eval_count(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  switch (sp.nm) {
    case 1: return launch_count_t<1>(sp, a, stream);
    case 2: return launch_count_t<2>(sp, a, stream);
    case 3: return launch_count_t<3>(sp, a, stream);
    case 4: return launch_count_t<4>(sp, a, stream);
    default: return launch_count_t<5>(sp, a, stream);
  }
}
cudaError_t launch_eval_write(const SpaceDev& sp, const EvalArgs& a, cudaStream_t stream) {
  switch (sp.nm) {
    case 1: return launch_write_t<1>(sp, a, stream);
    case 2: return launch_write_t<2>(sp, a, stream);
    case 3: return launch_write_t<3>(sp, a, stream);
    case 4: return launch_write_t<4>(sp, a, stream);
    default: return launch_write_t<5>(sp, a, stream);
  }
}
