// qtb_normal.cuh -- the white noise: Philox words to normals (Box-Muller pairs,
// (w0, w1) -> steps 4q, 4q+1 (cos, sin), (w2, w3) -> 4q+2, 4q+3).
#pragma once
#include "qtb_dev.cuh"

namespace qtb {

__device__ __forceinline__ void bm_pair(uint32_t a, uint32_t b, double &z0, double &z1)
{
    double u1 = ((double)a + 1.0) * 2.3283064365386963e-10;  // 2^-32, (0, 1]
    double u2 = (double)b * 2.3283064365386963e-10;          // [0, 1)
    double r = sqrt(-2.0 * log(u1));
    double s, c;
    sincospi(2.0 * u2, &s, &c);
    z0 = r * c;
    z1 = r * s;
}

__device__ __forceinline__ void bm_pair(uint32_t a, uint32_t b, float &z0, float &z1)
{
    float u1 = ((float)a + 1.0f) * 2.3283064365386963e-10f;
    float u2 = (float)b * 2.3283064365386963e-10f;
    float r = sqrtf(-2.0f * logf(u1));
    float s, c;
    sincospif(2.0f * u2, &s, &c);
    z0 = r * c;
    z1 = r * s;
}

// the normals of steps 4 q .. 4 q + 3 of dof `dof` of system `sys`
template <class C> __device__ __forceinline__ void white4(const Dev &d, uint32_t sys, int dof, long long q, C (&z)[4])
{
    const unsigned long long uq = (unsigned long long)q;
    const uint4 ctr = make_uint4((uint32_t)uq, (uint32_t)dof, 0u, (uint32_t)(uq >> 32));
    const uint4 w = philox4x32_10(ctr, (uint32_t)d.seed, (uint32_t)(d.seed >> 32) ^ sys);
    bm_pair(w.x, w.y, z[0], z[1]);
    bm_pair(w.z, w.w, z[2], z[3]);
}

}  // namespace qtb
