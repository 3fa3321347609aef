// Batched brute-force verifier: the paper's verification protocol (Section 7.1)
// as a data-parallel workload.  One block runs one case: a tiny layered network
// trained with Adam in fp64 on D logical devices that hold every state exactly
// as its placement mode says (Definition 1), with ring collectives whose bytes are
// counted per device (Section 2.3), next to the single-device run
// on the global batch (Definition 4's yardstick).  Whatever a placement leaves
// unavailable when it is needed reads as zeros, so a placement that breaks
// gradient integrity (Theorem 3) or state consistency (Theorem 4) really leaves
// the single-device trajectory (Theorem 5).  Per case the kernel reports whether
// every step's reassembled Theta and Omega equal the single-device run, and the
// bytes held, sent and moved over the host link in the last step.
//
// The kernel knows none of the closed-form rules; it executes the mechanism:
//   (1) make Theta available, forward      (2) keep, shard, offload or drop A
//   (3) make Theta available, backward     (4) synchronise and deliver G
//   (5) update on the range this device commits (all of it if Omega is
//       replicated, its shard if Omega's home is a shard)
//   (6) put Theta back into its home.
//
// Layout.  A case's states live in the block's shared memory.  The network is a
// stack of elementwise layers, so a column (device, sample, j) is a chain of its own
// through the layers: forward and backward take one thread per column, of the placed
// run and of the single-device run at once (two independent chains hide each other's
// latency); the update takes one thread per (device, element).  Sums over samples and
// around the ring are taken in the order in which a device and a ring take them.
// What bounds it: the chain of tanh, divisions and square roots of a step (fp64
// latency), then the fp64 pipe.  2500 cases of 64 parameters, three steps: 13.8 ms as
// one thread per case with its arrays in global memory (20 blocks on 148 SMs), 0.22 ms
// like this (0.26 with divisions of the indices; blocks of 64 threads 0.28).
#include "ps_device.cuh"
#include "ps_internal.h"

namespace {

constexpr int MAX_D = 4;
constexpr int MAX_STEPS = 16;
constexpr int MAX_P = 8 * 32, MAX_EA = 8 * 4 * 32;   // the shape's ranges: units * h, units * b * h

struct Dims {
  int units, h, b, P, EA, accum, steps, nbuf;
  int wT, wO, wG;
  double lr, beta1, beta2, eps, rtol, atol;
};

// offsets (in doubles) of a case's arrays in shared memory
struct Layout {
  int th_home, om_home, th_use, local, acts, dz, ref_acts, ref_dz, gsum, ref_th, ref_om, ref_g, debias, total;
};
__host__ __device__ inline Layout make_layout(int P, int EA) {
  Layout l;
  int o = 0;
  l.th_home = o; o += MAX_D * P;        // Theta at home (device or host arena), at global positions
  l.om_home = o; o += MAX_D * 3 * P;    // Omega at home: master, first and second moment
  l.th_use = o; o += MAX_D * P;         // Theta as forward / backward see it
  l.local = o; o += MAX_D * P;          // un-reduced local gradients (not a placed state)
  l.acts = o; o += MAX_D * EA;          // activations written by forward, e = (l * b + s) * h + j
  l.dz = o; o += MAX_D * EA;            // gradients at the layers' pre-activations, the same index
  l.ref_acts = o; o += MAX_D * EA;      // the same of the single-device run (its samples by device)
  l.ref_dz = o; o += MAX_D * EA;
  l.gsum = o; o += P;                   // gradients summed around the ring
  l.ref_th = o; o += P;                 // the single-device run
  l.ref_om = o; o += 3 * P;
  l.ref_g = o; o += P;
  l.debias = o; o += 2 * MAX_STEPS;     // 1 - beta1^t, 1 - beta2^t
  l.total = o;
  return l;
}

// eq. (2): shard i of E elements over D devices is [floor(i E / D), floor((i+1) E / D))
__device__ __forceinline__ int cut_of(int E, int D, int i) { return (int)(((long long)i * E) / D); }

// k / d for the kernel's small indices: with m = ceil(2^20 / d) the product is exact while
// k * d < 2^20 (indices stay below 1280, divisors below 257)
struct Divisor {
  u32 d, m;
  __device__ __forceinline__ explicit Divisor(int divisor) : d((u32)divisor), m(((1u << 20) + (u32)divisor - 1u) / (u32)divisor) {}
  __device__ __forceinline__ int of(int k) const { return (int)(((u32)k * m) >> 20); }
};

struct Books {
  long long mem, comm, host;
};

// The bytes of one step, counted by the lanes of a warp that stand for the devices
// (lane i < D = device i; all 32 lanes take part).  A collective that repeats within the
// step is counted once and taken as often as it runs.
__device__ Books keep_books(const Dims& dm, int D, int pT, int pO, int pG, int pA, int lane) {
  const int P = dm.P, h = dm.h, units = dm.units, i = lane < D ? lane : 0;
  const bool here = lane < D;
  const bool on_shard = (pO == PS_MODE_S || pO == PS_MODE_SG || pO == PS_MODE_O);
  const int nbuf = dm.nbuf < units ? dm.nbuf : units;     // a second unit buffer needs a second unit
  // elements of [a, z) that device p holds
  auto piece = [&](int a, int z, int p) {
    const int s0 = max(a, cut_of(P, D, p)), s1 = min(z, cut_of(P, D, p + 1));
    return (long long)(s1 > s0 ? s1 - s0 : 0);
  };
  // elements this device sends in a ring all-gather of [a, z): in step s it passes on the
  // piece that started at device (i - s) mod D
  auto gather = [&](int a, int z) {
    long long sent = 0;
    for (int s = 0; s + 1 < D; ++s) sent += piece(a, z, (i - s + D) % D);
    return sent;
  };
  // and in a ring reduce-scatter: in step s its partial sum of chunk (i - 1 - s) mod D
  auto reduce_scatter = [&](int a, int z) {
    long long sent = 0;
    for (int s = 0; s + 1 < D; ++s) sent += piece(a, z, (i - 1 - s + 2 * D) % D);
    return sent;
  };
  auto by_units = [&](auto&& count) {
    long long sent = 0;
    for (int l = 0; l < units; ++l) sent += count(l * h, (l + 1) * h);
    return sent;
  };
  auto busiest = [&](long long mine) {                     // over the devices
    long long m = here ? mine : 0;
    for (int o = MAX_D / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    return __shfl_sync(0xffffffffu, m, 0);
  };
  const long long shard = piece(0, P, i);
  const long long shard_a = cut_of(dm.EA, D, i + 1) - cut_of(dm.EA, D, i);
  const long long passes = 2LL * dm.accum;                 // forward and backward of every micro-batch
  long long host = 0;
  Books k;
  k.comm = 0;
  // Theta for forward and backward, gathered one reconstruction unit (layer) at a time
  if (pT == PS_MODE_SG || pT == PS_MODE_O) k.comm += passes * busiest(by_units(gather) * dm.wT);
  if (pT == PS_MODE_O) host += (passes + 1) * shard * dm.wT;       // host -> device each time, device -> host at the end
  if (pA == PS_MODE_O) host += 2LL * dm.EA * dm.accum;             // device -> host, host -> device
  // gradients
  if (pG == PS_MODE_M) {                                           // reduced unit by unit as produced
    k.comm += busiest(by_units(reduce_scatter) * dm.wG);
    if (!on_shard) k.comm += busiest(by_units(gather) * dm.wG);
  } else {
    k.comm += busiest(reduce_scatter(0, P) * dm.wG);
    if (pG == PS_MODE_R) k.comm += busiest(gather(0, P) * dm.wG);
    if (pG == PS_MODE_SG) k.comm += busiest(by_units(gather) * dm.wG);
    if (pG == PS_MODE_O) host += 2 * shard * dm.wG;                // offload, reload at the update
  }
  // update: a gathered Omega unit by unit, three rows of w_O / 3 bytes
  if (pO == PS_MODE_SG) k.comm += busiest(by_units(gather) * 3 * (dm.wO / 3));
  if (pO == PS_MODE_O) host += 2 * shard * dm.wO;                  // load, store
  // re-replicate the updated shards
  if (pT == PS_MODE_R && on_shard) k.comm += busiest(gather(0, P) * dm.wT);
  // bytes held: per state what the fullest device keeps, plus its unit buffer
  auto held = [&](int mode, long long whole, long long part, long long unit, bool buffer_of_m) {
    long long m = 0;
    if (mode == PS_MODE_R) m = whole;
    if (mode == PS_MODE_S || mode == PS_MODE_SG) m = busiest(part);
    if (mode == PS_MODE_SG) m += nbuf * unit;
    if (mode == PS_MODE_M && buffer_of_m) m += unit;
    return m;
  };
  k.mem = held(pT, (long long)P * dm.wT, shard * dm.wT, (long long)h * dm.wT, true) +
          held(pO, (long long)P * dm.wO, shard * dm.wO, (long long)h * dm.wO, false) +
          held(pG, (long long)P * dm.wG, shard * dm.wG, (long long)h * dm.wG, true) +
          held(pA, dm.EA, shard_a, (long long)dm.b * h, true);
  k.host = busiest(host);
  return k;
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_verify(Dims dm, const ps_verify_case* __restrict__ cases, u64 n_cases,
                                                    const double* __restrict__ data, u64 data_len,
                                                    double* theta_out, ps_verify_result* __restrict__ out, volatile u32* status) {
  extern __shared__ __align__(16) double mem[];
  const int tid = threadIdx.x;
  const int P = dm.P, h = dm.h, b = dm.b, units = dm.units, EA = dm.EA;
  const Layout L = make_layout(P, EA);
  double* const th_home = mem + L.th_home;
  double* const om_home = mem + L.om_home;
  double* const th_use = mem + L.th_use;
  double* const local = mem + L.local;
  double* const acts = mem + L.acts;
  double* const dzs = mem + L.dz;
  double* const ref_acts = mem + L.ref_acts;
  double* const ref_dz = mem + L.ref_dz;
  double* const gsum = mem + L.gsum;
  double* const ref_th = mem + L.ref_th;
  double* const ref_om = mem + L.ref_om;
  double* const ref_g = mem + L.ref_g;
  double* const debias = mem + L.debias;
  const Divisor by_p(P), by_h(h), by_bh(b * h);
  for (int t = tid; t < 2 * dm.steps; t += THREADS)
    debias[t] = 1.0 - pow(t & 1 ? dm.beta2 : dm.beta1, (double)(t / 2 + 1));

  for (u64 idx = blockIdx.x; idx < n_cases; idx += gridDim.x) {
    const ps_verify_case cs = cases[idx];
    {
      // a case that names more devices than supported, no placement, or data outside the
      // given array is reported, not run
      const u64 need = (u64)P + 2ull * dm.accum * cs.D * b * h;
      if (cs.D < 1 || cs.D > MAX_D || cs.code > 624 || cs.data_offset > data_len || need > data_len - cs.data_offset) {
        if (tid == 0) {
          ps_verify_result r;
          r.mem = 0; r.comm = 0; r.host = 0; r.match = 0; r.pad = 0; r.max_rel_err = 0.0;
          out[idx] = r;
          report(status, ST_BAD_CASE);
        }
        if (theta_out) for (int e = tid; e < P; e += THREADS) theta_out[idx * (u64)P + e] = 0.0;
        continue;                                          // the same for every thread of the block
      }
    }
    const int D = (int)cs.D;
    const int pT = cs.code % 5, pO = (cs.code / 5) % 5, pG = (cs.code / 25) % 5, pA = (cs.code / 125) % 5;
    // problem data: theta0[P], xs[accum][D][b][h], ys[accum][D][b][h]
    const double* theta0 = data + cs.data_offset;
    const double* xs = theta0 + P;
    const double* ys = xs + (size_t)dm.accum * D * b * h;
    const bool on_shard = (pO == PS_MODE_S || pO == PS_MODE_SG || pO == PS_MODE_O);
    const bool th_shard = (pT == PS_MODE_S || pT == PS_MODE_SG || pT == PS_MODE_O);
    int cut[MAX_D + 1], cut_a[MAX_D + 1];
#pragma unroll
    for (int i = 0; i <= MAX_D; ++i) { cut[i] = cut_of(P, D, min(i, D)); cut_a[i] = cut_of(EA, D, min(i, D)); }
    // the device whose shard an element lies in
    auto owner_of = [&](const int* c, int e) {
      int o = 0;
#pragma unroll
      for (int i = 1; i < MAX_D; ++i) o += (i < D && e >= c[i]) ? 1 : 0;
      return o;
    };

    __syncthreads();                                       // the previous case is done with shared memory
    // ---- homes (Definition 1): what each device holds of Theta and Omega
    for (int k = tid; k < D * P; k += THREADS) {
      const int i = by_p.of(k), e = k - i * P;
      const bool mine = owner_of(cut, e) == i;
      const double t0 = theta0[e];
      th_home[k] = (pT == PS_MODE_R || (th_shard && mine)) ? t0 : 0.0;
      double* om = om_home + (size_t)i * 3 * P + e;
      om[0] = (pO == PS_MODE_R || (on_shard && mine)) ? t0 : 0.0;      // the master copy lives inside Omega
      om[P] = 0.0;
      om[2 * P] = 0.0;
    }
    // ---- the single-device run starts from the same point
    for (int e = tid; e < P; e += THREADS) {
      const double t0 = theta0[e];
      ref_th[e] = t0;
      ref_om[e] = t0;
      ref_om[P + e] = 0.0;
      ref_om[2 * P + e] = 0.0;
    }
    bool match = pO != PS_MODE_M;                          // (mode M: Omega is held nowhere)
    double worst = 0.0;
    __syncthreads();

    for (int t = 1; t <= dm.steps; ++t) {
      const double debias1 = debias[2 * (t - 1)], debias2 = debias[2 * (t - 1) + 1];
      auto adam_elem = [&](double& master, double& m, double& v, double g) {
        m = dm.beta1 * m + (1.0 - dm.beta1) * g;
        v = dm.beta2 * v + (1.0 - dm.beta2) * g * g;
        const double mh = m / debias1;
        const double vh = v / debias2;
        master = master - dm.lr * mh / (sqrt(vh) + dm.eps);
      };
      // Theta as forward and backward see it on every device (steps (1) and (3); its home
      // does not change before the update)
      for (int k = tid; k < D * P; k += THREADS) {
        const int i = by_p.of(k), e = k - i * P, o = owner_of(cut, e);
        double v = 0.0;
        if (pT == PS_MODE_R || (pT == PS_MODE_S && o == i)) v = th_home[k];
        else if (pT == PS_MODE_SG || pT == PS_MODE_O) v = th_home[o * P + e];       // gathered
        else if (pT == PS_MODE_M && (pO == PS_MODE_R || ((pO == PS_MODE_S || pO == PS_MODE_SG) && o == i)))
          v = om_home[(size_t)i * 3 * P + e];              // cast from the master copy, where Omega is resident
        th_use[k] = v;
      }
      const int n_all = dm.accum * D * b;
      for (int j = 0; j < dm.accum; ++j) {
        __syncthreads();
        // (1) forward, every layer's input stored; device i's samples in the placed run and
        // the same samples in the single-device run
        for (int c = tid; c < D * b * h; c += THREADS) {
          const int i = by_bh.of(c), sj = c - i * b * h, s = by_h.of(sj), jj = sj - s * h;
          double cur = xs[(size_t)j * D * b * h + c], rcur = cur;
          for (int l = 0; l < units; ++l) {
            const int at = i * EA + (l * b + s) * h + jj;
            acts[at] = cur;
            ref_acts[at] = rcur;
            cur = tanh(th_use[i * P + l * h + jj] * cur);
            rcur = tanh(ref_th[l * h + jj] * rcur);
          }
          // (where backward reads other activations than forward wrote, its outputs are
          // formed again from those; else the layers' outputs are the next layers' inputs)
          dzs[i * EA + ((units - 1) * b + s) * h + jj] = cur;
          ref_dz[i * EA + ((units - 1) * b + s) * h + jj] = rcur;
        }
        __syncthreads();
        // (2) activations between forward and backward, (3) backward of 0.5 ||out - y||^2, mean over samples
        for (int c = tid; c < D * b * h; c += THREADS) {
          const int i = by_bh.of(c), sj = c - i * b * h, s = by_h.of(sj), jj = sj - s * h;
          const double y = ys[(size_t)j * D * b * h + c];
          const int top = i * EA + ((units - 1) * b + s) * h + jj;
          if (pA == PS_MODE_S || pA == PS_MODE_SG) {
            double dh = 0.0;
            for (int l = units - 1; l >= 0; --l) {
              const int e = (l * b + s) * h + jj, o = owner_of(cut_a, e);
              // sharded: only the own slice is left; gathered: from the peers, whose slices
              // belong to other samples
              const double a = pA == PS_MODE_SG ? acts[o * EA + e] : (o == i ? acts[i * EA + e] : 0.0);
              const double th = th_use[i * P + l * h + jj];
              const double out_l = tanh(th * a);
              if (l == units - 1) dh = (out_l - y) / b;
              const double dz = dh * (1.0 - out_l * out_l);
              dzs[i * EA + e] = dz;
              dh = dz * th;
            }
          } else {
            double out_l = dzs[top];
            if (pA == PS_MODE_M) {                         // recomputed
              double cur = xs[(size_t)j * D * b * h + c];
              for (int l = 0; l < units; ++l) {
                acts[i * EA + (l * b + s) * h + jj] = cur;
                cur = tanh(th_use[i * P + l * h + jj] * cur);
              }
              out_l = cur;
            }
            double dh = (out_l - y) / b;
            for (int l = units - 1; l >= 0; --l) {
              const int at = i * EA + (l * b + s) * h + jj;
              const double th = th_use[i * P + l * h + jj];
              const double dz = dh * (1.0 - out_l * out_l);
              dzs[at] = dz;
              dh = dz * th;
              out_l = acts[at];
            }
          }
          {
            double out_l = ref_dz[top];
            double dh = (out_l - y) / n_all;
            for (int l = units - 1; l >= 0; --l) {
              const int at = i * EA + (l * b + s) * h + jj;
              const double dz = dh * (1.0 - out_l * out_l);
              ref_dz[at] = dz;
              dh = dz * ref_th[l * h + jj];
              out_l = ref_acts[at];
            }
          }
        }
        __syncthreads();
        // parameter gradients: a device's sum over its samples, added with weight 1 / accum
        // to its local sum; the single-device run's sum over all samples in order
        for (int k = tid; k < (D + 1) * P; k += THREADS) {
          const int i = by_p.of(k), e = k - i * P, l = by_h.of(e), jj = e - l * h;
          if (i < D) {
            double g = 0.0;
            for (int s = 0; s < b; ++s) {
              const int f = (l * b + s) * h + jj;
              double a = acts[i * EA + f];
              if (pA == PS_MODE_S || pA == PS_MODE_SG) {
                const int o = owner_of(cut_a, f);
                a = pA == PS_MODE_SG ? acts[o * EA + f] : (o == i ? a : 0.0);
              }
              g += dzs[i * EA + f] * a;
            }
            local[k] = (j == 0 ? 0.0 : local[k]) + g / dm.accum;
          } else {
            double g = j == 0 ? 0.0 : ref_g[e];
            for (int d = 0; d < D; ++d)
              for (int s = 0; s < b; ++s) {
                const int f = d * EA + (l * b + s) * h + jj;
                g += ref_dz[f] * ref_acts[f];
              }
            ref_g[e] = g;
          }
        }
      }
      __syncthreads();
      // (4) synchronise gradients: the travelling partial sum of an element's chunk ch starts
      // at device ch + 1 and ends, after D - 1 steps, at device ch; in a unit-by-unit
      // reduction (mode M) an element takes the same way.  And the single-device update.
      for (int k = tid; k < 2 * P; k += THREADS) {
        if (k < P) {
          const int ch = owner_of(cut, k);
          double sum = local[(ch + 1) % D * P + k];
          for (int s = 2; s <= D; ++s) sum = local[(ch + s) % D * P + k] + sum;
          gsum[k] = sum;
        } else {
          const int e = k - P;
          adam_elem(ref_om[e], ref_om[P + e], ref_om[2 * P + e], ref_g[e]);
          ref_th[e] = ref_om[e];
        }
      }
      __syncthreads();
      // deliver gradients, (5) update on the range whose update this device commits, (6) Theta
      // back to its home; then Definition 4: every holder's view of Theta and Omega against
      // the single-device state
      const bool whole_g = pG == PS_MODE_R || pG == PS_MODE_SG || (pG == PS_MODE_M && !on_shard);
      auto compare = [&](double got, double want) {
        const double d = fabs(got - want);
        if (d > dm.atol) {
          const double rel = d / (fabs(want) > 1e-300 ? fabs(want) : 1e-300);
          if (rel > worst) worst = rel;
        }
        if (!(d <= dm.atol + dm.rtol * fabs(want))) match = false;
      };
      for (int k = tid; k < D * P; k += THREADS) {
        const int i = by_p.of(k), e = k - i * P;
        const bool mine = owner_of(cut, e) == i;
        const double g = (whole_g || mine) ? gsum[e] / D : 0.0;      // mean over the D replicas
        double* om = om_home + (size_t)i * 3 * P + e;
        double newth = 0.0;
        if (pO == PS_MODE_R || (on_shard && mine)) {
          double master = om[0], m = om[P], v = om[2 * P];
          adam_elem(master, m, v, g);
          om[0] = master; om[P] = m; om[2 * P] = v;
          newth = master;
          compare(master, ref_om[e]);
          compare(m, ref_om[P + e]);
          compare(v, ref_om[2 * P + e]);
        } else if (pO == PS_MODE_M) {                      // nothing was kept, the update starts from nothing
          double m = 0.0, v = 0.0;
          adam_elem(newth, m, v, g);
        }
        if (pT == PS_MODE_R && on_shard) {
          if (mine) {
            for (int d = 0; d < D; ++d) { th_home[d * P + e] = newth; compare(newth, ref_th[e]); }
          }
        } else if (pT == PS_MODE_R || (th_shard && mine)) {
          th_home[k] = newth;
          compare(newth, ref_th[e]);
        }
        // (Theta in mode M exists only as the master copy, compared above)
      }
      __syncthreads();
    }

    // ---- the case's record
    match = __syncthreads_and(match) != 0;
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if ((tid & 31) == 0) gsum[tid >> 5] = worst;           // (at most 8 warps; gsum has P >= 1 elements and ref_th follows)
    __syncthreads();
    if (tid < 32) {
      double w = gsum[0];
      for (int k = 1; k < THREADS / 32; ++k) w = fmax(w, gsum[k]);
      const Books k = keep_books(dm, D, pT, pO, pG, pA, tid);
      if (tid == 0) {
        ps_verify_result r;
        r.mem = (u64)k.mem;
        r.comm = (u64)k.comm;
        r.host = (u64)k.host;
        r.match = match ? 1u : 0u;
        r.pad = 0;
        r.max_rel_err = w;
        out[idx] = r;
      }
    }
    if (theta_out) {
      // the parameters the job holds after the last step (first holder's view)
      for (int e = tid; e < P; e += THREADS) {
        const int o = owner_of(cut, e);
        double v;
        if (pT == PS_MODE_R) v = th_home[e];
        else if (pT == PS_MODE_M) v = pO == PS_MODE_M ? 0.0 : om_home[(size_t)(pO == PS_MODE_R ? 0 : o) * 3 * P + e];
        else v = th_home[o * P + e];
        theta_out[idx * (u64)P + e] = v;
      }
    }
  }
}

template <int THREADS>
cudaError_t launch_verify_t(const Dims& dm, const ps_verify_case* d_cases, u64 n, const double* d_data, u64 data_len,
                            double* d_theta_out, ps_verify_result* d_out, volatile u32* status, cudaStream_t stream) {
  const int smem = make_layout(dm.P, dm.EA).total * (int)sizeof(double);
  // (the limit belongs to the kernel, not to a launch: the same for every call, so that a small
  // shape's call on another thread does not lower it between this one's two statements)
  const int most = make_layout(MAX_P, MAX_EA).total * (int)sizeof(double);    // 188 KB
  cudaError_t e = cudaFuncSetAttribute(k_verify<THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)(n < (1u << 20) ? n : (1u << 20));
  k_verify<THREADS><<<blocks, THREADS, smem, stream>>>(dm, d_cases, n, d_data, data_len, d_theta_out, d_out, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_verify(const ps_verify_shape& s, const ps_verify_case* d_cases, u64 n, const double* d_data,
                          u64 data_len, double* d_theta_out, ps_verify_result* d_out, volatile u32* status,
                          cudaStream_t stream) {
  Dims dm;
  dm.units = (int)s.units; dm.h = (int)s.h; dm.b = (int)s.b;
  dm.P = dm.units * dm.h; dm.EA = dm.units * dm.b * dm.h;
  dm.accum = (int)s.accum; dm.steps = (int)s.steps; dm.nbuf = (int)s.gather_buffers;
  dm.wT = (int)s.w_theta; dm.wO = (int)s.w_omega; dm.wG = (int)s.w_grad;
  dm.lr = s.lr; dm.beta1 = s.beta1; dm.beta2 = s.beta2; dm.eps = s.eps; dm.rtol = s.rtol; dm.atol = s.atol;
  // a thread per column of the largest case, within what one block may usefully hold
  const int columns = MAX_D * dm.b * dm.h;
  if (columns <= 64) return launch_verify_t<64>(dm, d_cases, n, d_data, data_len, d_theta_out, d_out, status, stream);
  if (columns <= 256) return launch_verify_t<128>(dm, d_cases, n, d_data, data_len, d_theta_out, d_out, status, stream);
  return launch_verify_t<256>(dm, d_cases, n, d_data, data_len, d_theta_out, d_out, status, stream);
}
