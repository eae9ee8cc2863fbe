// Reference seeds of an iterative scan (Sec. 2.1): the seeds of lowest RSS become reference points
// for a finer scan in their vicinity, kept sparse enough that the new seed sets do not overlap.
//
// refine_refs_kernel (one block): takes the candidates idx[0..M) in their given order (ascending RSS, as
// comet_scan_select returns them) and accepts a candidate unless, for some accepted reference, every
// lattice coordinate (z0, phi, pz, pT) differs by less than twice the new half-width: the two new
// lattices (reference +- half-width) would then overlap.  The block forms the coordinates of kTile
// candidates at a time, one per thread (atan2 and hypot in double, the only costly part); its first warp
// then walks them in order: lane j holds accepted reference j, so each candidate costs one lane-parallel
// test and one vote.  The test is decided in float where the float difference clears the width by more
// than its rounding, in double only otherwise (this part's double rate is 1/64 of its float rate).  One
// warp doing everything in double, a candidate at a time, and this: 64 candidates of the iterative scan's
// coarse lattice 165 and 13 us, 1,000 spread ones 709 and 89.  phi differences are taken modulo 2 pi.
#include <math.h>

#include "device.cuh"
#include "internal.h"

namespace comet {

namespace {

constexpr int kTile = 128;
constexpr double kTwoPi = 6.283185307179586;

template <typename T>
__global__ void __launch_bounds__(kTile) refine_refs_kernel(RefArgs a)
{
    __shared__ double sv[kTile][4];
    __shared__ int s_use[kTile], s_n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T *__restrict__ sd = (const T *)a.seeds;
    const int64_t S = a.S;
    double mine[4] = {0.0, 0.0, 0.0, 0.0};   // accepted reference `lane` (warp 0)
    float minef[4] = {0.f, 0.f, 0.f, 0.f}, w2f[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) w2f[d] = (float)(2.0 * a.half_width[d]);
    int n = 0;
    for (int c0 = 0; c0 < a.M && n < a.K; c0 += kTile) {
        const int c = c0 + threadIdx.x;
        bool use = false;
        if (c < a.M) {
            const int64_t s = a.idx[c];
            use = s >= 0 && s < S;   // else an unused slot of a short selection
            if (use) {
                const double px = (double)sd[3 * S + s], py = (double)sd[4 * S + s];
                sv[threadIdx.x][0] = (double)sd[2 * S + s];
                sv[threadIdx.x][1] = atan2(py, px);
                sv[threadIdx.x][2] = (double)sd[5 * S + s];
                sv[threadIdx.x][3] = hypot(px, py);
            }
        }
        s_use[threadIdx.x] = use;
        __syncthreads();
        if (warp == 0) {
            for (int t = 0; t < kTile && n < a.K; ++t) {
                if (!s_use[t]) continue;
                double v[4];
                float vf[4];
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    v[d] = sv[t][d];
                    vf[d] = (float)v[d];
                }
                bool in = lane < n, sure = true;
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    float r = fabsf(vf[d] - minef[d]);
                    const float e = 1e-6f * (fabsf(vf[d]) + fabsf(minef[d]) + w2f[d] + (d == 1 ? 7.f : 0.f));
                    if (d == 1) r = fminf(r, (float)kTwoPi - r);
                    if (r > w2f[d] + e) in = false;          // clear of each other
                    if (!(r < w2f[d] - e)) sure = false;     // not clearly inside (or not a number)
                }
                if (in && !sure) {
                    // |phi| <= pi, so one turn at most comes off the difference, exactly: what
                    // remainder(dv, 2 pi) gives
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        double r = fabs(v[d] - mine[d]);
                        if (d == 1 && !(r <= 0.5 * kTwoPi)) r = kTwoPi - r;
                        in = in && r < 2.0 * a.half_width[d];
                    }
                }
                if (__any_sync(0xffffffffu, in)) continue;
                if (lane == n) {
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        mine[d] = v[d];
                        minef[d] = vf[d];
                    }
                }
                ++n;
            }
            if (lane == 0) s_n = n;
        }
        __syncthreads();
        n = s_n;
    }
    if (warp == 0) {
        if (lane < n) {
#pragma unroll
            for (int d = 0; d < 4; ++d) a.refs_out[lane * 4 + d] = mine[d];
        }
        if (lane == 0) *a.n_refs_out = n;
    }
}

} // namespace

cudaError_t launch_refine_refs(comet_dtype dt, const RefArgs &a, cudaStream_t st)
{
    if (dt == COMET_F32)
        refine_refs_kernel<float><<<1, kTile, 0, st>>>(a);
    else
        refine_refs_kernel<double><<<1, kTile, 0, st>>>(a);
    return cudaGetLastError();
}

} // namespace comet
