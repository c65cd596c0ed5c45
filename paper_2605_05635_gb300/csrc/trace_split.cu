// trace_split.cu -- persistent per-ray kernel of the image path in split
// arithmetic (step_split.cuh): the rays of an FP64 image, and the promoted
// pass of the mixed path.  Method, scheduling, events and hand-offs as in
// trace.cu; the launch is FP64, the crossing events two-float too.
//
// The FP64 kernel it replaces there is bound by the FP64 pipe (about 1,100
// FP64 instructions per warp and step at 16 cycles each).  This one is bound
// by the FP32 pipes as long as its loop fits the instruction cache (32 KB)
// and little of it runs with few lanes, so
//   - the loop holds one copy of the right-hand side: f(y) of a ray that has
//     just started is an extra pass (s = -1) of the stage loop, and for a
//     launch one more (s = 0) gives the starting step;
//   - promoted rays are put back on their constants of motion by a kernel of
//     their own (promote_kernel) in which every lane has a ray, and hand-off
//     records carry float pairs, so starting or leaving the pass converts
//     nothing;
//   - crossings are parked as floats and evaluated (cross_split) for several lanes
//     together; a ray that ends with a parked crossing waits for the others.
// Measured (GB300): the promoted passes of three mixed 512^2 images (one a
// metric, 3 refinement levels) 676 -> 100 ms, a cored-NFW FP64 image of 96 x 75
// pixels with 2 levels 191 -> 42 ms; a lone ray 64,000 -> 13,000 cycles a step, which is
// what is left where a pass waits for its longest rays.
#include <cuda_runtime.h>

#include "step_split.cuh"

namespace bhrt {

// Lanes that exchange rays together: groups of 4, 6, 8 and 12 took 101, 100, 100
// and 101 ms of those passes.
constexpr int kRefillLanes = 6;

// Promoted rays back on their constants of motion (project_invariants), one
// record per thread.
__global__ void __launch_bounds__(128) promote_kernel(TraceArgs a) {
  const int64_t n = pass_items(a);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    SpillRec& s = const_cast<SpillRec*>(a.spill_in)[i];
    const ImgParams& ip = a.ip[s.img];
    double X, Y, y[6];
    int64_t pix;
    uint32_t im;
    resolve_item(a, s.item, im, pix, X, Y);
    float2* q = split_pairs(s);
#pragma unroll
    for (int c = 0; c < 6; ++c) y[c] = (double)q[c].x + (double)q[c].y;
    project_invariants(ip.md, s.E, s.ell, launch_carter(ip, X, Y), y);
    const F2 pR = f2_of(y[4]), pth = f2_of(y[5]);
    q[4] = make_float2(pR.h, pR.l);
    q[5] = make_float2(pth.h, pth.l);
    put_split_pair(s.E, f2_of(s.E));
    put_split_pair(s.ell, f2_of(s.ell));
  }
}

template <int MinBlocks, bool Vol>
__global__ void __launch_bounds__(kSplitThreads, MinBlocks) trace_split_kernel(TraceArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t n_items = pass_items(a);
  const unsigned long long budget = a.hdr->budget_ns;
  const unsigned long long t0 = a.hdr->t_start;

  __shared__ float4 stage[kStageSlots * kSplitThreads];
  const Stages st{&stage[threadIdx.x]};
  XPark xp;
  RaySplit r;
  const ImgParams* ip = a.ip;
  int64_t item = -1;
  uint32_t img = 0;
  bool active = false, drained = false;
  int wait = 0;            // term code (or kSpill) of a ray that waits for its crossing
  constexpr int kSpill = 16;
  r.xpend = false;
  r.fresh = 0;
  unsigned iter = 0, w_iters = 0, w_max = 0, w_acc = 0, w_rej = 0, w_rays = 0, w_full = 0;
  unsigned long long w_lanes = 0;

  const int pass = a.source;
  if (lane == 0) mark_first(&a.hdr->t_pass[0][pass][a.level]);
  while (true) {
    // ---- rays that have ended leave and new ones start, for kRefillLanes
    // lanes together (or when none steps); parked crossings of every lane are
    // evaluated first
    {
      const unsigned bm = __ballot_sync(kFull, active);
      const unsigned fm = __ballot_sync(kFull, wait != 0 || (!active && !drained));
      if (__popc(fm) >= kRefillLanes || bm == 0u) {
        if (r.xpend) {
          CrossState cs = r.cs;
          cross_split(*ip, r.k.E, r.k.ell, xp, cs, cross_out(a, item, img));
          r.cs = cs;
          r.xpend = false;
        }
        if (wait) {
          if (wait != kSpill) {
            finish_ray(a, item, img, wait - 1, r.cs, r.hdrift, r.nacc, r.nrej, 0.0, 0.0, r.lam);
            w_rays += 1;
            w_max = (unsigned)r.steps > w_max ? (unsigned)r.steps : w_max;
          } else {
            unsigned long long slot = atomicAdd(a.spill_out_count, 1ull);
            if (slot < (unsigned long long)a.spill_cap) {
              spill_from_split(r, item, img, a.spill_out[slot]);
            } else {
              w_full += 1;
              active = true;
            }
          }
          wait = 0;
        }
        const bool need = !active && !drained;
        int64_t idx = claim(a.head, need, lane);
        if (need) {
          if (idx < n_items) {
            if (a.source == 1) {
              const SpillRec& s = a.spill_in[idx];
              item = s.item;
              img = s.img;
              ip = &a.ip[img];
              resume_split(*ip, s, r);
            } else {
              item = idx;
              launch_item(a, idx, img, &xp);
              ip = &a.ip[img];
              take_launch(*ip, xp, r);
            }
            active = true;
          } else {
            drained = true;
            mark_first(&a.hdr->t_pass[1][pass][a.level]);
          }
        }
      }
    }
    const unsigned am = __ballot_sync(kFull, active);
    if (am == 0) break;  // nothing steps, waits or is left in the queue
    w_iters += 1;
    w_lanes += (unsigned long long)__popc(am);

    // ---- one attempted step of every active lane
    const SplitStep o = split_attempt<Vol>(*ip, r, st, active);
    bool cross = false;
    int term = o.term;
    if (o.ok) {
      const float s0 = dth_split(r.y[0]), s1 = dth_split(o.y1[0]);
      cross = (s0 > 0.f && s1 <= 0.f) || (s0 < 0.f && s1 >= 0.f);
      w_acc++;
    } else if (active) {
      w_rej++;
    }
    // parked crossings wait for the next exchange of rays, or are evaluated
    // when a lane needs its slot again (so a ray's crossings stay in order)
    if (__any_sync(kFull, cross && r.xpend) && r.xpend) {
      CrossState cs = r.cs;
      cross_split(*ip, r.k.E, r.k.ell, xp, cs, cross_out(a, item, img));
      r.cs = cs;
      r.xpend = false;
    }
    bool spill = false;
    if (o.ok) {
      if (cross) {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          xp.y0[p] = r.y[p];
          xp.d[p] = o.dl[p];
          xp.k0[p] = st.get(0, p);
          xp.k6[p] = st.get(6, p);
        }
#pragma unroll 1
        for (int p = 0; p < 3; ++p) {
          F2x2 q = v_prod(kDP2.d[0], st.get(0, p));
          q.l = v_sub(0ull, q.l);
#pragma unroll 1
          for (int j = 2; j < 7; ++j) q = v_acc(kDP2.d[j], st.get(j, p), q);
          xp.sd[p] = q;
        }
        xp.lam = r.lam;
        xp.h = r.h;
        r.xpend = true;
      }
      term = split_commit<Vol>(*ip, r, st, o);
      // outgoing beyond the strong-field zone, or away from the double root
      // of its radial potential: finish in FP32
      const float pR = lo_of(r.y[1].a), kappa = (float)ip->kappa;
      spill = !term && a.allow_spill && pR > 0.f &&
              (lo_of(r.y[0].a) > (float)ip->demote_R ||
               (kappa > 0.f && o.mon.DpR * o.mon.DpR > kDemoteKappa * kappa * o.mon.P * o.mon.P));
    }
    if (term || spill) {
      wait = term ? term : kSpill;
      active = false;
    }
    if (budget && ((++iter & 255u) == 0u)) {
      unsigned long long now = __shfl_sync(kFull, globaltimer(), 0);
      if (now - t0 > budget) {
        if (lane == 0) atomicCAS(&a.hdr->status, 0, (int)BH_ERR_TIMEOUT);
        break;
      }
    }
  }
  flush_tally(&a.hdr->accepted, w_acc, lane);
  flush_tally(&a.hdr->rejected, w_rej, lane);
  flush_tally(&a.hdr->rays[a.level], w_rays, lane);
  if (lane == 0) {
    atomicMax(&a.hdr->t_pass[2][pass][a.level], globaltimer());
    atomicAdd(&a.hdr->warp_iters[1], (unsigned long long)w_iters);
    atomicAdd(&a.hdr->lane_iters[1], w_lanes);
  }
  if (w_max) atomicMax(&a.hdr->max_ray_steps, (unsigned long long)w_max);
  flush_tally(&a.hdr->spill_full, w_full, lane);
}

cudaError_t launch_trace_split(const TraceArgs& a, LaunchShape s, cudaStream_t st) {
  if (a.source == 1) {
    promote_kernel<<<num_sms() * 8, 128, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (a.any_volumetric) {
    if (s.variant == 1)
      trace_split_kernel<4, true><<<s.blocks, s.threads, 0, st>>>(a);
    else
      trace_split_kernel<3, true><<<s.blocks, s.threads, 0, st>>>(a);
  } else if (s.variant == 1) {
    trace_split_kernel<4, false><<<s.blocks, s.threads, 0, st>>>(a);
  } else {
    trace_split_kernel<3, false><<<s.blocks, s.threads, 0, st>>>(a);
  }
  return cudaGetLastError();
}

int trace_split_blocks_per_sm(int threads, int variant) {
  int nb = 0;
  if (variant == 1)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, trace_split_kernel<4, false>, threads, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, trace_split_kernel<3, false>, threads, 0);
  return nb > 0 ? nb : 1;
}

}  // namespace bhrt
