// Forward rollouts in the limb layout (brax_limb.cuh): the wide kernel (a limb
// of two environments a lane) for many environments, the split kernel (a limb
// body of one environment a lane) for few.
//
// The arithmetic is the paired kernel's (brax_pair.cuh), operation for
// operation and in the same order, so all three give the same bits.
#include <cstddef>

#include "brax_kernels.h"
#include "brax_limb.cuh"

namespace brax {

__constant__ __align__(16) unsigned char c_pool[kPoolBytes];
static_assert(offsetof(SysP, limb_upper) % 8 == 0 && offsetof(SysP, limb_lower) % 8 == 0 && BRAX_MAX_CHILDREN == 8,
              "the split kernel loads the limbs' bodies as 8-byte words");

namespace p2 {
// integrate()'s potential integrator alone: the velocities before contacts.
template <class Par, class Fl>
__device__ __forceinline__ void potential(const SysP2& S2, Fl flags, const Par& q, const Wrench& wr, const Body& s,
                                          const Frame& f, V& v, V& w) {
  v = vfma(S2.h, vfma(q.inv_mass, wr.F, vld(S2.g)), s.v);
  w = vfma(S2.h, mul6(f.Ii, wr.tau), s.w);
  if (frozen(flags)) {
    v = mask(flags, v);
    w = mask(rot_bits(flags), w);
  }
}
}  // namespace p2

// The wide kernel.  What bounds it is the register file: an SM sub-partition
// reads two 32-bit operands a cycle, so a packed multiply-add with three
// distinct operands takes three cycles (measured: 3.0; packed multiply or add
// 2.0; two scalar multiply-adds 3.1).  More resident warps therefore do not help
// (12 warps an SM with state parked in shared memory: 88 us a step against 80
// at the time), and neither does a longer straight run of code; fewer
// instructions and a better order of them do.  Quadruped, 65,536 environments,
// us a step: 82.3 with the lower body's contacts before the upper's and all
// counts read in the loop; 74.4 in this order (the upper body's state is dead
// sooner) with the counts read before it; 72.0 (910 M env-steps/s) with kTwo,
// the two contact points of every limb body known at compile time (capsule
// limbs).  The paired kernel: 84.9 at its best launch, 95.5 at its default one.
template <int L, bool kFrozen, bool kEnv, bool kTwo>
__global__ void __launch_bounds__(128, 2) rollout_limb_kernel(const __grid_constant__ Launch Ln) {
  using namespace p2;
  constexpr int E = 32 / L;  // slots of a warp; a slot is two environments
  static_assert(2 * E * (1 + 2 * L) * 13 * 4 <= kLimbStageBytes, "a warp's checkpoint fits its stage");
  const Seg& sg = Ln.seg[0];
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  const bool chunked = Ln.sc.n_chunks > 0;
  int unit = blockIdx.x, c = 0, t0 = 0, t1 = Ln.T;
  if (chunked) {
    const int n_units = Ln.sc.n_units, n_items = Ln.sc.n_chunks * n_units;
    if (threadIdx.x == 0) {
      int ticket;
      const int it = take_item(Ln.sc, n_items, &ticket);
      if (it == -2) atomicOr(sg.status, kStatusTimeout);
      s_item = it;
    }
    __syncthreads();
    const int it = s_item;
    if (it < 0 || it >= n_items) return;
    unit = it % n_units;
    c = it / n_units;
    t0 = c * Ln.sc.chunk_steps;
    t1 = min(Ln.T, t0 + Ln.sc.chunk_steps);
  }
  const unsigned char* blob = c_pool + sg.pool_off;
  const SysP& S = *reinterpret_cast<const SysP*>(blob);
  const BodyP* bodies = reinterpret_cast<const BodyP*>(blob + blob_bodies_off());
  const SysP2& S2 = *reinterpret_cast<const SysP2*>(blob + S.pair_off);
  const BodyP2* bodies2 = reinterpret_cast<const BodyP2*>(blob + S.pair_off + sizeof(SysP2));
  LimbTab2* tab = reinterpret_cast<LimbTab2*>(smem);
  load_limb_tab2(S, sg.blob, tab);
  __syncthreads();

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int n_warps = blockDim.x >> 5;
  const int lane = threadIdx.x & 31, limb = lane % L, slot = lane / L;
  const int64_t N = sg.n_envs;
  const int64_t e0 = ((int64_t)unit * n_warps + warp) * (2 * E);
  const int64_t ea = e0 + slot, eb = ea + E;
  const bool va = ea < N, vb = eb < N;
  if (e0 >= N) t1 = t0;  // a warp past the last environment steps nothing
  float4* react = reinterpret_cast<float4*>(smem + limb_tab_bytes(L) + warp * kLimbWarpBytes);
  float* const stage = reinterpret_cast<float*>(smem + limb_tab_bytes(L) + warp * kLimbWarpBytes + kLimbReactBytes);
  const int B = sg.B, A = sg.A, K = Ln.K;
  const int br = S.limb_root, bu = S.limb_upper[limb], bl = S.limb_lower[limb];
  // the scalars of all upper (lower) bodies are those of limb 0's
  const BodyP &pr = bodies[br], &pu = bodies[S.limb_upper[0]], &pl = bodies[S.limb_lower[0]];
  const BodyP2 &qr = bodies2[br], &qu = bodies2[S.limb_upper[0]], &ql = bodies2[S.limb_lower[0]];
  const LimbGeo2 &gu = tab[limb].upper, &gl = tab[limb].lower;
  const int au = bodies[bu].act[0], al = bodies[bl].act[0];
  const bool act_u = pu.act[0] >= 0, act_l = pl.act[0] >= 0;
  // without frozen axes every masking folds away
  const uint32_t fr_ = kFrozen ? pr.flags : 0u, fu_ = kFrozen ? pu.flags : 0u, fl_ = kFrozen ? pl.flags : 0u;
  const bool average = S.average != 0;
  // counts the substep loop reads, held in registers
  const int npr = pr.n_points, npu = kTwo ? 2 : pu.n_points, npl = kTwo ? 2 : pl.n_points;
  const int nsub = S.substeps;

  p2::Body sr, su, sl;
  {  // chunk 0 starts from state0, a later chunk from what the previous one left in state_T
    const float* src = c == 0 ? sg.state0 : sg.state_T;
    auto ld = [&](int b, p2::Body& s) {
      load_pair(va ? src + (ea * B + b) * 13 : nullptr, vb ? src + (eb * B + b) * 13 : nullptr, bodies[b], s);
    };
    ld(br, sr);
    ld(bu, su);
    ld(bl, sl);
  }
  int cca = 0, ccb = 0;
  bool bad = false, staged = false;
  // a step's actions are loaded during the step before it
  f2 nu = zero2(), nl = zero2();
  auto load_act = [&](int t) {
    const float* ap = sg.actions + (int64_t)t * N * A;
    if (act_u) nu = make_float2(va ? __ldg(ap + ea * A + au) : 0.f, vb ? __ldg(ap + eb * A + au) : 0.f);
    if (act_l) nl = make_float2(va ? __ldg(ap + ea * A + al) : 0.f, vb ? __ldg(ap + eb * A + al) : 0.f);
  };
  if (t0 < t1) load_act(t0);
  int buf = 0;
  for (int t = t0; t < t1; ++t) {
    if (sg.ckpt && (t % K) == 0) {
      float* ck = sg.ckpt + ((int64_t)(t / K) * N) * B * 13;
      // the warp's environments are one contiguous block of the checkpoint
      // ([N][B][13]): staged in shared memory and stored with one bulk
      // asynchronous copy; a block not 16-byte sized and aligned directly
      const int64_t nv = N - e0 < 2 * E ? N - e0 : 2 * E;
      float* dst = ck + e0 * B * 13;
      const uint32_t bytes = nv > 0 ? (uint32_t)(nv * B * 13) * 4u : 0u;
      if (bytes && (bytes & 15u) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
        if (lane == 0 && staged) bulk_wait_read();  // the previous copy has read the buffer
        __syncwarp();
        float* pa = stage + slot * B * 13;
        float* pb = stage + (E + slot) * B * 13;
        if (limb == 0) {
          store_half(pa + br * 13, sr, 0);
          store_half(pb + br * 13, sr, 1);
        }
        store_half(pa + bu * 13, su, 0);
        store_half(pb + bu * 13, su, 1);
        store_half(pa + bl * 13, sl, 0);
        store_half(pb + bl * 13, sl, 1);
        fence_proxy_async();  // the staged states, written by this thread, precede the bulk read
        __syncwarp();
        if (lane == 0) {
          bulk_copy_s2g(dst, stage, bytes);
          staged = true;
        }
      } else {
        if (va) {
          if (limb == 0) store_half(ck + (ea * B + br) * 13, sr, 0);
          store_half(ck + (ea * B + bu) * 13, su, 0);
          store_half(ck + (ea * B + bl) * 13, sl, 0);
        }
        if (vb) {
          if (limb == 0) store_half(ck + (eb * B + br) * 13, sr, 1);
          store_half(ck + (eb * B + bu) * 13, su, 1);
          store_half(ck + (eb * B + bl) * 13, sl, 1);
        }
      }
    }
    const f2 actu = nu, actl = nl;
    if (t + 1 < t1) load_act(t + 1);
    const f2 x0 = sr.x.x;  // the root's x before the step (environment layer)
#pragma unroll 1
    for (int k = 0; k < nsub; ++k) {
      // the table is read anew in every substep instead of being kept in
      // registers (or spilled) across the loop
      asm volatile("" ::: "memory");
      kinematic(S2, fr_, sr);
      kinematic(S2, fu_, su);
      kinematic(S2, fl_, sl);
      p2::Frame fr, fu, fl;
      fr.R = qmat(sr.qw, sr.qx, sr.qy, sr.qz, S2.one);
      fu.R = qmat(su.qw, su.qx, su.qy, su.qz, S2.one);
      const JointOut ju = joint(qu, gu, true, p2::Pub{sr.x, fr.R, sr.v, sr.w}, su, fu.R, actu);
      float4* rx = react + buf * 96;
      if (L > 1) {
        rx[lane] = make_float4(ju.F_.x.x, ju.F_.x.y, ju.F_.y.x, ju.F_.y.y);
        rx[32 + lane] = make_float4(ju.F_.z.x, ju.F_.z.y, ju.tp.x.x, ju.tp.x.y);
        rx[64 + lane] = make_float4(ju.tp.y.x, ju.tp.y.y, ju.tp.z.x, ju.tp.z.y);
      }
      fl.R = qmat(sl.qw, sl.qx, sl.qy, sl.qz, S2.one);
      const JointOut jl = joint(ql, gl, true, p2::Pub{su.x, fu.R, su.v, su.w}, sl, fl.R, actl);
      fl.Ii = inv_inertia_world(fl.R, ql.inv_I);
      fu.Ii = inv_inertia_world(fu.R, qu.inv_I);
      {  // upper body
        p2::Acc acc{vzero(), vzero(), 0, 0};
        plane_points_z(S2, qu, gu, fu_, npu, su, fu, acc);
        cca += acc.na;
        ccb += acc.nb;
        integrate(S2, average, fu_, qu, p2::Wrench{vsub(ju.F_, jl.F_), vadd(ju.tc, jl.tp)}, su, fu, acc);
      }
      {  // lower body: contacts, integrators
        p2::Acc acc{vzero(), vzero(), 0, 0};
        plane_points_z(S2, ql, gl, fl_, npl, sl, fl, acc);
        cca += acc.na;
        ccb += acc.nb;
        integrate(S2, average, fl_, ql, p2::Wrench{jl.F_, jl.tc}, sl, fl, acc);
      }
      {  // root: the limbs' reactions in child order, alike on all its lanes
        p2::Wrench wr{vzero(), vzero()};
        if (L > 1) {
          // one barrier a substep: the other buffer is written only after
          // every lane has read this one's predecessor
          __syncwarp();
#pragma unroll
          for (int j = 0; j < L; ++j) {
            const float4* p = rx + (slot * L + j);
            const float4 a = p[0], b = p[32], d = p[64];
            wr.F = vsub(wr.F, V{make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y)});
            wr.tau = vadd(wr.tau, V{make_float2(b.z, b.w), make_float2(d.x, d.y), make_float2(d.z, d.w)});
          }
          buf ^= 1;
        } else {
          wr.F = vsub(wr.F, ju.F_);
          wr.tau = vadd(wr.tau, ju.tp);
        }
        fr.Ii = inv_inertia_world(fr.R, qr.inv_I);
        p2::Acc acc{vzero(), vzero(), 0, 0};
        plane_points_z(S2, qr, qr, fr_, npr, sr, fr, acc);
        if (limb == 0) {
          cca += acc.na;
          ccb += acc.nb;
        }
        integrate(S2, average, fr_, qr, wr, sr, fr, acc);
      }
    }
    if (sg.torso && br == 0 && limb == 0) {  // (the root is body 0; without the test the code came out slower)
      float* tp = sg.torso + (int64_t)t * N * 3;
      if (va) {
        tp[ea * 3 + 0] = sr.x.x.x;
        tp[ea * 3 + 1] = sr.x.y.x;
        tp[ea * 3 + 2] = sr.x.z.x;
      }
      if (vb) {
        tp[eb * 3 + 0] = sr.x.x.y;
        tp[eb * 3 + 1] = sr.x.y.y;
        tp[eb * 3 + 2] = sr.x.z.y;
      }
    }
    if (kEnv) {
      // environment layer (Sec. 4.2 gym-like env), each environment of the
      // pair in turn: a lane observes its own limb's joints (the parent's
      // rotation is the substep's, which the step's quaternion gives again),
      // limb 0 the root; the limbs' squared actions are summed in child order.
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const bool vh = h ? vb : va;
        const int64_t eh = h ? eb : ea;
        auto hv = [h](f2 v) { return h ? v.y : v.x; };
        const brax::Body hr = half_body(sr, h), hu = half_body(su, h), hl = half_body(sl, h);
        float* ob = sg.obs + ((int64_t)t * N + eh) * sg.obs_dim;
        if (vh) {
          auto joint_fields = [&](const p2::Body& par, const brax::Body& ph, const brax::Body& ch, int b) {
            const M R2 = qmat(par.qw, par.qx, par.qy, par.qz, S2.one);
            M3 Rp;
#pragma unroll
            for (int i = 0; i < 9; ++i) Rp.m[i] = hv(R2.m[i]);
            float ang[3], rate[3];
            joint_obs<false>(bodies[b], Rp, ph.w, brax::qmat(ch.qw, ch.qx, ch.qy, ch.qz), ch.w, ang, rate);
            ob[11 + bodies[b].dof_offset] = ang[0];
            ob[11 + S.D + bodies[b].dof_offset] = rate[0];
          };
          joint_fields(sr, hr, hu, bu);
          joint_fields(su, hu, hl, bl);
        }
        const float ua = clamp1(hv(actu)), la = clamp1(hv(actl));
        const float cu = act_u ? ua * ua : 0.f, cl = act_l ? la * la : 0.f;
        float ctrl = 0.f;
#pragma unroll
        for (int j = 0; j < L; ++j) {
          ctrl += __shfl_sync(0xffffffffu, cu, slot * L + j);
          ctrl += __shfl_sync(0xffffffffu, cl, slot * L + j);
        }
        int done = 0;
        if (vh && limb == 0)
          done = root_env(sg, hr, hv(x0), ctrl, ob, sg.reward + (int64_t)t * N + eh, sg.done + (int64_t)t * N + eh);
        done = __shfl_sync(0xffffffffu, done, slot * L);
        if (sg.auto_reset && vh && done) {
          const float* rs = sg.reset_state + eh * B * 13;
          load_half(rs + br * 13, sr, h);
          load_half(rs + bu * 13, su, h);
          load_half(rs + bl * 13, sl, h);
        }
      }
    }
    bad |= !finite_pair(sr) || !finite_pair(su) || !finite_pair(sl);
  }
  if (staged) bulk_wait_all();  // the checkpoint stores are complete before the block ends
  if (va) {
    float* p = sg.state_T + ea * B * 13;
    if (limb == 0) store_half(p + br * 13, sr, 0);
    store_half(p + bu * 13, su, 0);
    store_half(p + bl * 13, sl, 0);
  }
  if (vb) {
    float* p = sg.state_T + eb * B * 13;
    if (limb == 0) store_half(p + br * 13, sr, 1);
    store_half(p + bu * 13, su, 1);
    store_half(p + bl * 13, sl, 1);
  }
  if (bad && (va || vb)) atomicOr(sg.status, kStatusNonfinite);
  if (sg.ccount) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) {
      cca += __shfl_xor_sync(0xffffffffu, cca, o);
      ccb += __shfl_xor_sync(0xffffffffu, ccb, o);
    }
    if (limb == 0) {
      if (va) __stcg(sg.ccount + ea, (c ? __ldcg(sg.ccount + ea) : 0) + cca);
      if (vb) __stcg(sg.ccount + eb, (c ? __ldcg(sg.ccount + eb) : 0) + ccb);
    }
  }
  if (chunked) {  // the item is done: its stores are made visible, then the unit's flag says so
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) store_release(Ln.sc.sched + 32 + unit, c + 1);
  }
}

// ------------------------------------------------------------------ one body a lane
namespace p2 {
// Parameters of a lane's own body and its joint, in registers (the root's
// beside the own body's where both go through packed arithmetic).
struct SplitPar {
  float off_p[3], off_c[3], ap[6], ac[6];        // geometry of the own joint
  float k, mc, ka, mca, kl, lo, hi, gear;        // its scalars
  static constexpr int dof = 1;
};
struct SplitPoint {
  f2 o[3], r, mr, mu, me, p0z;
};
struct SplitBody {
  f2 inv_mass, inv_I[3];
  SplitPoint pt[2];
  __device__ __forceinline__ const f2* point(int i) const { return pt[i].o; }
};
__device__ __forceinline__ float2 halves(float a, float b) { return make_float2(keep(a), keep(b)); }
__device__ __forceinline__ SplitPar split_par(const BodyP2& q) {
  SplitPar p;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p.off_p[i] = keep(q.off_p[i].x);
    p.off_c[i] = keep(q.off_c[i].x);
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    p.ap[i] = keep(q.ap[i].x);
    p.ac[i] = keep(q.ac[i].x);
  }
  p.k = keep(q.k.x);
  p.mc = keep(q.mc.x);
  p.ka = keep(q.ka.x);
  p.mca = keep(q.mca.x);
  p.kl = keep(q.kl.x);
  p.lo = keep(q.lo.x);
  p.hi = keep(q.hi.x);
  p.gear = keep(q.gear.x);
  return p;
}
// Points a body does not have get the radius -inf: they never touch.
__device__ __forceinline__ SplitBody split_body(const BodyP2& r, int nr, const BodyP2& q, int nq) {
  SplitBody p;
  p.inv_mass = halves(r.inv_mass.x, q.inv_mass.x);
#pragma unroll
  for (int i = 0; i < 3; ++i) p.inv_I[i] = halves(r.inv_I[i].x, q.inv_I[i].x);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
#pragma unroll
    for (int j = 0; j < 3; ++j) p.pt[i].o[j] = halves(r.pt[i].o[j].x, q.pt[i].o[j].x);
    p.pt[i].r = halves(i < nr ? r.pt[i].r.x : -INFINITY, i < nq ? q.pt[i].r.x : -INFINITY);
    p.pt[i].mr = halves(r.pt[i].mr.x, q.pt[i].mr.x);
    p.pt[i].mu = halves(r.pt[i].mu.x, q.pt[i].mu.x);
    p.pt[i].me = halves(r.pt[i].me.x, q.pt[i].me.x);
    p.pt[i].p0z = halves(r.pt[i].p0[2].x, q.pt[i].p0[2].x);
  }
  return p;
}
__device__ __forceinline__ VT<float> lo_half(V a) { return VT<float>{a.x.x, a.y.x, a.z.x}; }
__device__ __forceinline__ VT<float> hi_half(V a) { return VT<float>{a.x.y, a.y.y, a.z.y}; }
__device__ __forceinline__ V join(VT<float> a, VT<float> b) {
  return V{make_float2(a.x, b.x), make_float2(a.y, b.y), make_float2(a.z, b.z)};
}
__device__ __forceinline__ float shfl(float a, int src) { return __shfl_sync(0xffffffffu, a, src); }
__device__ __forceinline__ VT<float> shfl(VT<float> a, int src) {
  return VT<float>{shfl(a.x, src), shfl(a.y, src), shfl(a.z, src)};
}
__device__ __forceinline__ VT<float> pick(bool second, VT<float> a, VT<float> b) {
  return VT<float>{second ? b.x : a.x, second ? b.y : a.y, second ? b.z : a.z};
}
__device__ __forceinline__ f2 pick(bool sx, bool sy, f2 a, f2 b) {
  return make_float2(sx ? b.x : a.x, sy ? b.y : a.y);
}
// Plane contacts of the split kernel, whose single warps are bound by latency:
// each half's first touching point is answered in straight code (masked where
// there is none) that overlaps the joint's, and only a warp with a body that
// touches at both its points answers the second.  The first touching point is
// added before the second, as in plane_points_z.
template <class Fl>
__device__ __forceinline__ void contacts_first(const SysP2& S2, bool average, Fl flags, const SplitBody& q,
                                               const Body& s, const Frame& f, V& dv, V& dw, f2& inv, int& cca,
                                               int& ccb) {
  f2 d[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const f2* o = q.point(i);
    const f2 rz = fma(f.R.m[6], o[0], fma(f.R.m[7], o[1], mul(f.R.m[8], o[2])));
    d[i] = sub(q.pt[i].r, sub(add(s.x.z, rz), q.pt[i].p0z));
  }
  const bool a0 = d[0].x > 0.f, b0 = d[0].y > 0.f, a1 = d[1].x > 0.f, b1 = d[1].y > 0.f;
  SplitPoint p;
#pragma unroll
  for (int j = 0; j < 3; ++j) p.o[j] = pick(!a0, !b0, q.pt[0].o[j], q.pt[1].o[j]);
  p.mr = pick(!a0, !b0, q.pt[0].mr, q.pt[1].mr);
  p.mu = pick(!a0, !b0, q.pt[0].mu, q.pt[1].mu);
  p.me = pick(!a0, !b0, q.pt[0].me, q.pt[1].me);
  Acc acc{vzero(), vzero(), 0, 0};
  {
    const V ro = mulc(f.R, p.o);
    point_response_z<false>(S2, flags, q.inv_mass, p, V{ro.x, ro.y, add(ro.z, p.mr)}, pick(!a0, !b0, d[0], d[1]),
                            a0 || a1, b0 || b1, s, f, acc);
  }
  if (__any_sync(0xffffffffu, (a0 && a1) || (b0 && b1))) {
    const V ro = mulc(f.R, q.pt[1].o);
    point_response_z(S2, flags, q.inv_mass, q.pt[1], V{ro.x, ro.y, add(ro.z, q.pt[1].mr)}, d[1], a0 && a1, b0 && b1, s,
                     f, acc);
  }
  cca += acc.na;
  ccb += acc.nb;
  inv = make_float2((average && acc.na > 1) ? __fdividef(1.f, (float)acc.na) : 1.f,
                    (average && acc.nb > 1) ? __fdividef(1.f, (float)acc.nb) : 1.f);
  dv = acc.dv;
  dw = acc.dw;
}
}  // namespace p2

// Forward rollout with one limb body a lane (lane = ((slot * L) + limb) * 2 +
// level, level 0: upper, 1: lower), one environment a slot.  A packed register
// pair holds the root (.x) and the own body (.y), so that the integrators, the
// rotations and the contact responses of both run as one packed stream; the
// own joint runs in single FP32.  The operations and their order are those of
// the wide kernel, so the bits are.
//
// Few environments leave a warp alone on its SM sub-partition, where a substep
// lasts as long as one warp takes: the wide kernel's lane does a whole limb of
// two environments (1,260 instructions a substep), this one's a body of one
// (560), with the contact responses in straight code beside the joint's.  Its
// root is computed by 2 L lanes, the wide kernel's by L / 2 per environment, so
// it loses where warps fill the SMs (us a step of both and of the body layout:
// the table at limb_rule in brax_capi.cu).
//
// kFew: at most 8 warps an SM, no spills (36 bytes under the 168 registers that
// let 12 be resident, which more warps need).  With the start's loads taken
// from the constant pool: 2,048 environments 5.9 -> 5.5 us a step.
template <int L, bool kFrozen, bool kEnv, bool kFew>
__global__ void __launch_bounds__(128, kFew ? 2 : 3) rollout_limb_split_kernel(const __grid_constant__ Launch Ln) {
  using namespace p2;
  using F3 = VT<float>;
  constexpr int E = 16 / L;  // environments of a warp
  const Seg& sg = Ln.seg[0];
  __shared__ int s_item;
  __shared__ float4 s_react[4][2][2][16];  // [warp][buffer][chunk][upper body of the warp]
  const bool chunked = Ln.sc.n_chunks > 0;
  int unit = blockIdx.x, c = 0, t0 = 0, t1 = Ln.T;
  if (chunked) {
    const int n_units = Ln.sc.n_units, n_items = Ln.sc.n_chunks * n_units;
    if (threadIdx.x == 0) {
      int ticket;
      const int it = take_item(Ln.sc, n_items, &ticket);
      if (it == -2) atomicOr(sg.status, kStatusTimeout);
      s_item = it;
    }
    __syncthreads();
    const int it = s_item;
    if (it < 0 || it >= n_items) return;
    unit = it % n_units;
    c = it / n_units;
    t0 = c * Ln.sc.chunk_steps;
    t1 = min(Ln.T, t0 + Ln.sc.chunk_steps);
  }
  const unsigned char* blob = c_pool + sg.pool_off;
  const SysP& S = *reinterpret_cast<const SysP*>(blob);
  const BodyP* bodies = reinterpret_cast<const BodyP*>(blob + blob_bodies_off());
  const SysP2& S2 = *reinterpret_cast<const SysP2*>(blob + S.pair_off);
  const BodyP2* bodies2 = reinterpret_cast<const BodyP2*>(blob + S.pair_off + sizeof(SysP2));
  // lane-varying parameters come from the blob's copy in global memory
  const BodyP* gbodies = reinterpret_cast<const BodyP*>(sg.blob + blob_bodies_off());
  const BodyP2* gbodies2 = reinterpret_cast<const BodyP2*>(sg.blob + S.pair_off + sizeof(SysP2));

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31, level = lane & 1, limb = (lane >> 1) % L, slot = lane / (2 * L);
  const int64_t N = sg.n_envs;
  const int64_t e = ((int64_t)unit * (blockDim.x >> 5) + warp) * E + slot;
  const bool valid = e < N;
  if (e - slot >= N) t1 = t0;  // a warp past the last environment steps nothing
  const int B = sg.B, A = sg.A, K = Ln.K;
  const int br = S.limb_root;
  // the lane's body out of eight in one uniform load (a lane-varying index would
  // cost the launch another round trip to L2)
  const uint64_t ids = *reinterpret_cast<const uint64_t*>(level ? S.limb_lower : S.limb_upper);
  const int bo = (int)(ids >> (8 * limb)) & 255;
  const BodyP &pr = bodies[br], &po = gbodies[bo];
  const SplitPar jp = split_par(gbodies2[bo]);
  const SplitBody bp = split_body(bodies2[br], pr.n_points, gbodies2[bo], po.n_points);
  const Flags2 fl = kFrozen ? Flags2{pr.flags, po.flags} : Flags2{0u, 0u};
  const int act_idx = po.act[0];
  const bool average = S.average != 0;
  const bool root_lane = limb == 0 && level == 0;  // speaks for the slot's root

  p2::Body s;
  {
    const float* src = c == 0 ? sg.state0 : sg.state_T;
    const float* p = src + e * B * 13;
    auto ld = [&](int i) {
      const BodyP& pb = gbodies[br];
      const float r0 = i < 3 ? pb.rest_pos[i] : (i < 7 ? pb.rest_rot[i - 3] : 0.f);
      const float r1 = i < 3 ? po.rest_pos[i] : (i < 7 ? po.rest_rot[i - 3] : 0.f);
      return make_float2(valid ? __ldcg(p + br * 13 + i) : r0, valid ? __ldcg(p + bo * 13 + i) : r1);
    };
    s.x = V{ld(0), ld(1), ld(2)};
    s.qw = ld(3);
    s.qx = ld(4);
    s.qy = ld(5);
    s.qz = ld(6);
    s.v = V{ld(7), ld(8), ld(9)};
    s.w = V{ld(10), ld(11), ld(12)};
  }
  int ccr = 0, cco = 0;
  bool bad = false;
  float next_act = 0.f;
  auto load_act = [&](int t) {
    if (valid && act_idx >= 0) next_act = __ldg(sg.actions + ((int64_t)t * N + e) * A + act_idx);
  };
  if (t0 < t1) load_act(t0);
  int buf = 0;
  for (int t = t0; t < t1; ++t) {
    if (sg.ckpt && (t % K) == 0 && valid) {
      float* ck = sg.ckpt + ((int64_t)(t / K) * N + e) * B * 13;
      if (root_lane) store_half(ck + br * 13, s, 0);
      store_half(ck + bo * 13, s, 1);
    }
    const float act = next_act;
    if (t + 1 < t1) load_act(t + 1);
    const float x0 = s.x.x.x;  // the root's x before the step (environment layer)
#pragma unroll 1
    for (int k = 0; k < S.substeps; ++k) {
      if (kFrozen) {
        s.v = mask(fl, s.v);
        s.w = mask(rot_bits(fl), s.w);
      }
      advance(S2.h, S2.mhh, S2.hh, s);
      p2::Frame f;
      f.R = qmat(s.qw, s.qx, s.qy, s.qz, S2.one);
      f.Ii = inv_inertia_world(f.R, bp.inv_I);
      V dv, dw;
      f2 inv;
      contacts_first(S2, average, fl, bp, s, f, dv, dw, inv, ccr, cco);
      // the parent of an upper body is the root (own registers), of a lower
      // one the upper body in the lane before
      const int up = lane & ~1;
      PubT<float> pp;
      pp.x = pick(level, lo_half(s.x), shfl(hi_half(s.x), up));
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const float r = shfl(f.R.m[i].y, up);
        pp.R.m[i] = level ? r : f.R.m[i].x;
      }
      pp.v = pick(level, lo_half(s.v), shfl(hi_half(s.v), up));
      pp.w = pick(level, lo_half(s.w), shfl(hi_half(s.w), up));
      BodyT<float> o;
      o.x = hi_half(s.x);
      o.v = hi_half(s.v);
      o.w = hi_half(s.w);
      MT<float> Ro;
#pragma unroll
      for (int i = 0; i < 9; ++i) Ro.m[i] = f.R.m[i].y;
      const JointOutT<float> j = joint(jp, jp, true, pp, o, Ro, act);
      float4(*rx)[16] = s_react[warp][buf];
      if (!level) {
        rx[0][lane >> 1] = make_float4(j.F_.x, j.F_.y, j.F_.z, j.tp.x);
        *reinterpret_cast<f2*>(&rx[1][lane >> 1]) = make_float2(j.tp.y, j.tp.z);
      }
      // an upper body takes its lower body's reaction (the lane after)
      const F3 rF = shfl(j.F_, lane | 1), rt = shfl(j.tp, lane | 1);
      const F3 Fo = pick(level, vsub(j.F_, rF), j.F_), to = pick(level, vadd(j.tc, rt), j.tc);
      __syncwarp();
      F3 Fr = vzero<float>(), tr = vzero<float>();  // the root's, in child order
#pragma unroll
      for (int i = 0; i < L; ++i) {
        const float4 a = rx[0][slot * L + i];
        const f2 b = *reinterpret_cast<const f2*>(&rx[1][slot * L + i]);
        Fr = vsub(Fr, F3{a.x, a.y, a.z});
        tr = vadd(tr, F3{a.w, b.x, b.y});
      }
      buf ^= 1;
      V nv, nw;
      potential(S2, fl, bp, p2::Wrench{join(Fr, Fo), join(tr, to)}, s, f, nv, nw);
      s.v = vfma(inv, dv, nv);
      s.w = vfma(inv, dw, nw);
    }
    if (sg.torso && br == 0 && root_lane && valid) {
      float* tp = sg.torso + ((int64_t)t * N + e) * 3;
      tp[0] = s.x.x.x;
      tp[1] = s.x.y.x;
      tp[2] = s.x.z.x;
    }
    if (kEnv) {
      // environment layer, as in the wide kernel
      const M R2 = qmat(s.qw, s.qx, s.qy, s.qz, S2.one);
      M3 Rp;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const float r = shfl(R2.m[i].y, lane & ~1);
        Rp.m[i] = level ? r : R2.m[i].x;
      }
      const F3 w2 = pick(level, lo_half(s.w), shfl(hi_half(s.w), lane & ~1));
      const brax::Body hr = half_body(s, 0), ho = half_body(s, 1);
      float* ob = sg.obs + ((int64_t)t * N + e) * sg.obs_dim;
      if (valid) {
        float ang[3], rate[3];
        joint_obs<false>(jp, Rp, mk3(w2.x, w2.y, w2.z), brax::qmat(ho.qw, ho.qx, ho.qy, ho.qz), ho.w, ang, rate);
        ob[11 + po.dof_offset] = ang[0];
        ob[11 + S.D + po.dof_offset] = rate[0];
      }
      const float u = clamp1(act), cu = act_idx >= 0 ? u * u : 0.f;
      float ctrl = 0.f;
#pragma unroll
      for (int j = 0; j < 2 * L; ++j) ctrl += shfl(cu, slot * 2 * L + j);
      int done = 0;
      if (valid && root_lane)
        done = root_env(sg, hr, x0, ctrl, ob, sg.reward + (int64_t)t * N + e, sg.done + (int64_t)t * N + e);
      done = __shfl_sync(0xffffffffu, done, slot * 2 * L);
      if (sg.auto_reset && valid && done) {
        const float* rs = sg.reset_state + e * B * 13;
        load_half(rs + br * 13, s, 0);
        load_half(rs + bo * 13, s, 1);
      }
    }
    bad |= !finite_pair(s);
  }
  if (valid) {
    float* p = sg.state_T + e * B * 13;
    if (root_lane) store_half(p + br * 13, s, 0);
    store_half(p + bo * 13, s, 1);
  }
  if (bad && valid) atomicOr(sg.status, kStatusNonfinite);
  if (sg.ccount) {
    int cc = cco + (root_lane ? ccr : 0);
#pragma unroll
    for (int o = 1; o < 2 * L; o <<= 1) cc += __shfl_xor_sync(0xffffffffu, cc, o);
    if (root_lane && valid) __stcg(sg.ccount + e, (c ? __ldcg(sg.ccount + e) : 0) + cc);
  }
  if (chunked) {  // the item is done: its stores are made visible, then the unit's flag says so
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) store_release(Ln.sc.sched + 32 + unit, c + 1);
  }
}

// ------------------------------------------------------------------ launchers
using LimbKernel = void (*)(const Launch);
template <int L, bool kFrozen, bool kEnv>
static LimbKernel limb_kernel_e(const LimbLaunch& l) {
  if (!l.split) return l.two ? rollout_limb_kernel<L, kFrozen, kEnv, true> : rollout_limb_kernel<L, kFrozen, kEnv, false>;
  return l.few ? rollout_limb_split_kernel<L, kFrozen, kEnv, true> : rollout_limb_split_kernel<L, kFrozen, kEnv, false>;
}
template <int L>
static LimbKernel limb_kernel_l(const LimbLaunch& l) {
  if (l.frozen) return l.env ? limb_kernel_e<L, true, true>(l) : limb_kernel_e<L, true, false>(l);
  return l.env ? limb_kernel_e<L, false, true>(l) : limb_kernel_e<L, false, false>(l);
}
static LimbKernel limb_kernel(const LimbLaunch& l) {
  switch (l.n_limbs) {
    case 1: return limb_kernel_l<1>(l);
    case 2: return limb_kernel_l<2>(l);
    case 4: return limb_kernel_l<4>(l);
    default: return limb_kernel_l<8>(l);
  }
}
static size_t limb_smem_bytes(const LimbLaunch& l) {
  return l.split ? 0 : limb_tab_bytes(l.n_limbs) + l.warps * kLimbWarpBytes;
}
int limb_blocks_per_sm(const LimbLaunch& l) {
  const LimbKernel k = limb_kernel(l);
  const size_t smem = limb_smem_bytes(l);
  if (allow_smem(k, smem) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 32 * l.warps, smem) != cudaSuccess) return 0;
  return n;
}
cudaError_t launch_rollout_limb(const Launch& L, const LimbLaunch& l, int grid, cudaStream_t st) {
  const LimbKernel k = limb_kernel(l);
  const size_t smem = limb_smem_bytes(l);
  cudaError_t e = allow_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<grid, 32 * l.warps, smem, st>>>(L);
  return cudaGetLastError();
}
cudaError_t upload_pool_limb(int off, const void* data, size_t bytes) {
  return cudaMemcpyToSymbol(c_pool, data, bytes, (size_t)off, cudaMemcpyHostToDevice);
}

}  // namespace brax
