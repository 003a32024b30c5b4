// Limb layout: systems that are one root body with L limbs of two hinged
// bodies each (upper: child of the root, lower: child of the upper), L a
// power of two, the limbs alike up to their geometry (the quadruped: 4, the
// pendulum: 1).
//
// In the body layout (brax_pair.cuh, brax_physics.cuh) a warp is a body, so a
// substep's joints exchange states and reactions through shared memory at two
// group barriers, at which eight warps wait for the slowest.  Here one lane
// holds a whole limb and a copy of the root: both joints of the limb find
// parent and child in the lane's own registers, the root's kinematics are
// computed by each of an environment's L lanes alike (the same instructions on
// the same values, so the copies stay bitwise equal), and what is left to
// exchange is each limb's reaction on the root: three 16-byte stores and 3 L
// loads a lane and substep through the warp's own shared memory.  No warp ever
// waits for another one.
//
// Lane i of a warp is limb i % L of slot i / L.
#pragma once
#include "brax_pair.cuh"

namespace brax {

// A limb body's geometry in shared memory, as (value, value) pairs: the
// parameters that differ from limb to limb.  The scalars, alike for all limbs,
// are read from the constant pool.
struct alignas(16) LimbGeo2 {
  float2 off_p[3], off_c[3], ap[6], ac[6], o[2][3];
  __device__ __forceinline__ const float2* point(int i) const { return o[i]; }
};
// Upper and lower body of one limb; the 16 bytes at the end put the limbs'
// equal fields on different banks (8 limbs x 16 bytes: all 32 banks).
struct alignas(16) LimbTab2 {
  LimbGeo2 upper, lower;
  float pad[4];
};
static_assert(sizeof(LimbGeo2) == 192 && sizeof(LimbTab2) == 400, "LimbTab2 layout");

// Copy the limbs' geometry from the system's blob into shared memory (the
// whole block takes part; the caller synchronises the block).
__device__ __forceinline__ void load_limb_tab2(const SysP& S, const unsigned char* blob, LimbTab2* tab) {
  const BodyP2* b2 = reinterpret_cast<const BodyP2*>(blob + S.pair_off + sizeof(SysP2));
  for (int i = threadIdx.x; i < S.n_limbs * 48; i += blockDim.x) {
    const int limb = i / 48, r = i - limb * 48, low = r / 24, f = r - low * 24;
    const float2* q = reinterpret_cast<const float2*>(b2 + (low ? S.limb_lower[limb] : S.limb_upper[limb]));
    const float2* src = f < 18 ? q + f : (f < 21 ? b2[0].pt[0].o - reinterpret_cast<const float2*>(b2) + q + (f - 18)
                                                 : b2[0].pt[1].o - reinterpret_cast<const float2*>(b2) + q + (f - 21));
    reinterpret_cast<float2*>(low ? &tab[limb].lower : &tab[limb].upper)[f] = __ldg(src);
  }
}

// Shared memory of the wide kernel (bytes): the table, then per warp two
// buffers of reactions [2][3][32] float4 and the stage of a checkpoint (the
// largest: 64 environments of three bodies).
__host__ __device__ inline size_t limb_tab_bytes(int n_limbs) { return n_limbs * sizeof(LimbTab2); }
constexpr size_t kLimbReactBytes = 2 * 3 * 32 * 16;
constexpr size_t kLimbStageBytes = 64 * 3 * 13 * 4;
constexpr size_t kLimbWarpBytes = kLimbReactBytes + kLimbStageBytes;
}  // namespace brax
