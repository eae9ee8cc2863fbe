// DCA finding and RSS (Algorithm 2, Eq. 1, Sec. 2.2.2).
//
// Layout of the work: one thread per seed, a warp per 32-seed group.  The persistent kernel (up to
// 1024 wires) stages every wire's geometry, the CSR hit offsets and (when they fit) the drift
// distances and masks once per CTA in shared memory with the bulk-copy engine (cp.async.bulk +
// mbarrier), and its warps take (group, wire chunk) items; the tiled kernel (more wires) stages
// them in tiles of 256 wires per 128-seed CTA.
//
// Closest recorded state of a (seed, wire) pair, found exactly without visiting every state.  The
// recorded states of each seed are cut into at most 8 super-segments of G0 states, each cut into at
// most 24 level-1 segments of G1 states.  Because the seed lattice numbers neighbouring nodes
// consecutively, the 32 tracks of a warp are close, and one bounding sphere per segment covers all
// 32 of them: its centre is the midpoint of the first and the last lane's segment centres, its
// radius the largest distance from it to any lane's segment centre plus (g/2) h_rec (a recorded
// state within g/2 recording intervals of a centre is at most that far from it along the track).
// Every recorded state x of that segment of every seed of the warp then satisfies
// dist(x, wire) >= dist(C, wire) - radius.  The spheres are read in place from the table the
// recording kernel wrote (or built in shared memory when no table is given).  For each wire, the
// lanes test the spheres in parallel (lane t: wire t against the super-segment spheres; then lane
// m: level-1 sphere m of a candidate super-segment) and only segments whose bound does not exceed
// the wire's capture radius (largest unmasked drift + lambda + h_rec/2) are searched, each lane its own
// seed's states, for the lexicographic (distance, index) minimum: runs of a few states are scanned state
// by state, longer ones in an axial field walked down the valley of the distance (group_wires_long).
// If a seed's closest state is within the capture radius it lies in a
// searched segment, so the minimum is exact; if not, every residual of the wire is at least lambda
// and the wire adds exactly lambda^2 to the RSS, with or without a refinement.  Beyond the first
// and the last recorded state the refinement reaches up to h_rec (not h_rec/2) from the nearest
// recorded state, so segments that may hold a track end are tested, and an end state refined,
// within capture radius + h_rec.  With dca_out (exact DCA for every wire) the spheres leave the segments
// that may hold a lane's closest state; without a sphere table, or where a group's tracks all have a few
// states, every state is then scanned.
//
// RSS: each thread sums its wires' d_i^2 in ascending wire order within each wire chunk (FP32 as a
// TwoSum pair, FP64 plainly), then the chunks' sums in chunk order.  Atomics only hand out work
// and count arrivals: the result does not depend on scheduling (the paper's GPU kernel summed with
// atomics and was not deterministic, Sec. 4.1).
#include <float.h>

#include "device.cuh"
#include "internal.h"

// Tuning constants (compile-time): minimum resident CTAs per SM requested from the register
// allocator, and how many states are loaded together.  FP32 axial, short runs and every DCA: issue and
// latency both count (8 CTAs: 2^18 x 70 states the same, 2^17 odd lattice 514 -> 547 us; 6: 469 us
// against 452 at 2^18).  Long runs: 6 (2^14 x 2,229 states 157 us; 219 at 7, 227 at 8).
#ifndef COMET_DCA_MINB
#define COMET_DCA_MINB 7
#endif
#ifndef COMET_DCA_MINB_LONG
#define COMET_DCA_MINB_LONG 6
#endif
// FP64: bound by the FP64 pipe rather than by resident warps; fewer CTAs per SM buy registers (at
// 72 the FP64 kernels spill ~300 B per thread; 4 CTAs take 1% longer than 3 at 2^15 x 139 states)
#ifndef COMET_DCA_MINB_F64
#define COMET_DCA_MINB_F64 3
#endif
// FP32 in a non-axial field (tabulated or general uniform): RK4 stages in the refinement; at 72
// registers the tabulated-field kernel spilled ~200 B per thread
#ifndef COMET_DCA_MINB_FIELD
#define COMET_DCA_MINB_FIELD 5
#endif
// States per trip to memory of the long form's scan (11,475 seeds of an odd lattice x 275 states, FP32 axial:
// 2 states 298 us, 4 206, 8 231; general uniform field, which has fewer registers free: 263, 4 237, 3 242,
// but 2^14 seeds x 69 states, whose runs are short: 4 91, 3 89).  FP64 waits for its pipe, not for memory: 2, or 4 when
// every DCA is wanted (2^15 seeds x 137 states 2 1517, 4 1555; every DCA of 256 x 137 without spheres 457 and 403)
#ifndef COMET_DCA_U
#define COMET_DCA_U 4
#endif
#ifndef COMET_DCA_U_FIELD
#define COMET_DCA_U_FIELD 3
#endif
// wires per chunk of the per-seed sums (the persistent kernel's finest work item)
#ifndef COMET_DCA_CHUNK_W
#define COMET_DCA_CHUNK_W 32
#endif

namespace comet {

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
static_assert(kWarps == kDcaWarpsPerCta, "persistent DCA CTA size");
constexpr int kWireTile = 256;
constexpr int kWireCap = kWireTile + 32;     // elements per staged row (room for the 16-B shift)
constexpr int kHitMax = 1024;                // hits staged in shared memory when H <= kHitMax
constexpr int kHitCap = kHitMax + 32;
constexpr uint64_t kWaitNs = 2000000000ull;  // limit of the wait for an abandoned copy (2 s)

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

template <typename T>
struct Smem {
    static constexpr size_t bar = 0;
    static constexpr size_t sph0 = 16;                                            // [warp][j][4]
    static constexpr size_t sph1 = align16(sph0 + sizeof(float) * kWarps * kN0Max * 4);  // [warp][j][m][4]
    static constexpr size_t wrow = align16(sph1 + sizeof(float) * kWarps * kN0Max * kN1Max * 4);
    static constexpr size_t orow = align16(wrow + sizeof(T) * 6 * kWireCap);
    static constexpr size_t cap = align16(orow + sizeof(int32_t) * (kWireCap + 8));
    static constexpr size_t frame = align16(cap + sizeof(T) * kWireTile);
    static constexpr size_t drift = align16(frame + sizeof(T) * 16 * kWireTile);
    static constexpr size_t mask = align16(drift + sizeof(T) * kHitCap);
    static constexpr size_t total = align16(mask + kHitCap);
};

// Plans the staging of one array, issues its bulk copy (thread 0) and plain-loads its ragged ends
// (all threads).  Returns the element offset of element 0 in dst.
template <typename E>
__device__ __forceinline__ int stage_issue(E *dst, const E *src, int n, uint64_t *bar, bool issuer)
{
    const StagePlan p = stage_plan(src, n, (int)sizeof(E));
    if (issuer && p.body > 0)
        bulk_g2s(dst + p.off + p.head, src + p.head, (uint32_t)(p.body * sizeof(E)), bar);
    for (int i = threadIdx.x; i < p.head; i += blockDim.x) dst[p.off + i] = src[i];
    for (int i = p.head + p.body + threadIdx.x; i < n; i += blockDim.x) dst[p.off + i] = src[i];
    return p.off;
}

template <typename E>
__device__ __forceinline__ uint32_t stage_bytes(const E *src, int n)
{
    const StagePlan p = stage_plan(src, n, (int)sizeof(E));
    return (uint32_t)(p.body * sizeof(E));
}

// After a timed-out wait: copy the bulk parts with plain loads.
template <typename E>
__device__ __forceinline__ void stage_fallback(E *dst, const E *src, int n)
{
    const StagePlan p = stage_plan(src, n, (int)sizeof(E));
    for (int i = p.head + threadIdx.x; i < p.head + p.body; i += blockDim.x) dst[p.off + i] = src[i];
}

// A launch scalar in the working precision: the host-rounded float copy for FP32.
template <typename T>
__device__ __forceinline__ T in_prec(double d, float f)
{
    if constexpr (sizeof(T) == 4)
        return f;
    else
        return d;
}

// Twosum accumulator for FP32, plain for FP64.
template <typename T>
struct Acc;
template <>
struct Acc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add_square(float d) { two_sum_add(hi, lo, __fmul_rn(d, d)); }
    __device__ __forceinline__ void add_pair(float h2, float l2)
    {
        two_sum_add(hi, lo, h2);
        two_sum_add(hi, lo, l2);
    }
    __device__ __forceinline__ float value() const { return hi + lo; }
};
template <>
struct Acc<double> {
    double hi = 0.0, lo = 0.0;
    __device__ __forceinline__ void add_square(double d) { hi = fma(d, d, hi); }
    __device__ __forceinline__ void add_pair(double h2, double) { hi += h2; }
    __device__ __forceinline__ double value() const { return hi; }
};

} // namespace

// Extra reach (m) when an FP64 kernel tests a sphere in FP32: float rounding of the wire frame (unit
// vectors and the offsets av = a.v, aw = a.w) and of the distance arithmetic moves the distance by
// a few ulp of the coordinates involved, ~1e-7 m per metre of |av| + |aw| + reach; 2 um plus 1 um
// per metre is a generous bound (the FP64 test it stands in for then never rejects more).
__device__ __forceinline__ float sph_margin_f32(float av, float aw)
{
    return 2e-6f + 1e-6f * (fabsf(av) + fabsf(aw));
}

// ------------------------------------------------------------------------------------------------
// One 32-seed group (one warp): per-lane seed state, bounding spheres, and the wire loop
// ------------------------------------------------------------------------------------------------

template <typename T>
struct Group {
    int64_t s;       // this lane's seed
    bool valid;
    int nv;          // recorded states of the seed
    int n0w;         // super-segments of the longest track of the warp
    int elo, ehi;    // smallest and largest last state index over the warp's tracks
    T c, ip;         // KAPPA q / P0, 1 / P0
    float sz;        // |pz| / P0 (constant along the track in an axial field)
};

template <typename T>
__device__ __forceinline__ Group<T> load_group(const DcaArgs &a, int64_t g, int lane)
{
    const T *__restrict__ P = (const T *)a.points;
    const int64_t S = a.S;
    const int64_t plane = (int64_t)a.n_rec * S;
    Group<T> gr;
    gr.s = g * 32 + lane;
    gr.valid = gr.s < S;
    gr.nv = 1;
    gr.c = T(0);
    gr.ip = T(0);
    gr.sz = 0.f;
    if (gr.valid) {
        gr.nv = a.n_valid[gr.s];
        const T pz = P[5 * plane + gr.s];
        seed_kinematics<T>(P[3 * plane + gr.s], P[4 * plane + gr.s], pz, a.charge[gr.s], gr.c, gr.ip);
        gr.sz = fabsf((float)(pz * gr.ip));
    }
    int n0w = gr.valid ? (gr.nv + a.G0 - 1) / a.G0 : 0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) n0w = max(n0w, __shfl_xor_sync(0xffffffffu, n0w, off));
    gr.n0w = n0w;
    gr.elo = (int)__reduce_min_sync(0xffffffffu, (unsigned)(gr.valid ? gr.nv - 1 : 0x7fffffff));
    gr.ehi = (int)__reduce_max_sync(0xffffffffu, (unsigned)(gr.valid ? gr.nv - 1 : 0));
    return gr;
}

// The warp's bounding spheres of its super-segments (sph0[j]) and level-1 segments
// (sph1[j * kN1Max + m]), written by lane 0.
template <typename T>
__device__ __forceinline__ void build_spheres(const DcaArgs &a, const Group<T> &gr, int lane,
                                              float4 *sph0, float4 *sph1, int64_t g)
{
    if (g * 32 >= a.S) return;   // no seed in this group: nothing will be searched
    if (a.bounds) {
        // written by comet_scan_propagate: copy this group's table into the warp's slot
        const float4 *src = (const float4 *)a.bounds + g * kBoundsPerGroup;
        for (int i = lane; i < kBoundsPerGroup; i += 32) {
            const float4 v = __ldg(src + i);
            if (i < kN0Max)
                sph0[i] = v;
            else
                sph1[i - kN0Max] = v;
        }
        __syncwarp();
        return;
    }
    const T *__restrict__ P = (const T *)a.points;
    const int64_t S = a.S;
    const int64_t plane = (int64_t)a.n_rec * S;
    const int G0 = a.G0, G1 = a.G1;
    const int N1 = (G0 + G1 - 1) / G1;
    for (int j = 0; j < kN0Max; ++j) {
        const int sb = j * G0, se = min(sb + G0, gr.nv);
        const bool has = gr.valid && sb < gr.nv;
        T x = T(0), y = T(0), z = T(0);
        if (has) {
            const int64_t o = (int64_t)min(sb + G0 / 2, se - 1) * S + gr.s;
            x = P[o];
            y = P[plane + o];
            z = P[2 * plane + o];
        }
        const float4 sp = warp_sphere<T>(has, x, y, z, (T)a.R0);
        if (lane == 0) sph0[j] = sp;
        for (int m = 0; m < N1; ++m) {
            const int st = sb + m * G1;
            const bool h1 = has && st < se;
            T x1 = T(0), y1 = T(0), z1 = T(0);
            if (h1) {
                const int64_t o = (int64_t)min(st + G1 / 2, min(st + G1, se) - 1) * S + gr.s;
                x1 = P[o];
                y1 = P[plane + o];
                z1 = P[2 * plane + o];
            }
            const float4 sp1 = warp_sphere<T>(h1, x1, y1, z1, (T)a.R1);
            if (lane == 0) sph1[j * kN1Max + m] = sp1;
        }
    }
    __syncwarp();
}

// Per-wire record of a staged tile, four of them per wire: (v, a.v), (w, a.w), (a, capture radius),
// (u, 0) -- one 16-byte-aligned load each (two for double).
template <typename T>
struct alignas(16) Q4 {
    T x, y, z, w;
};

// A staged range of wires [w0, w0 + wn) in shared memory.
template <typename T>
struct Tile {
    const T *ax, *ay, *az, *ux, *uy, *uz;   // wire point and direction, element i = wire w0 + i
    const Q4<T> *rec;                        // [wire][4]: (v, a.v), (w, a.w), (a, cap), (u, 0)
    const float4 *ff;                        // FP64 only: [wire][2], (v, a.v) and (w, a.w) in float
    const T *cap;                            // capture radius (< 0: no unmasked hit)
    const int32_t *offs;                     // CSR offsets, element i = wire w0 + i
    const T *dsm;                            // drifts / masks: staged (global hit index) or global
    const uint8_t *msm;
    int w0, wn;
};

// Wire i's frame (v, a.v), (w, a.w) for the sphere tests, which are made in float in either precision:
// the part's FP64 rate would be the limit there, and an FP64 tile keeps a float copy of its frames.
template <typename T>
__device__ __forceinline__ void sphere_frame(const Tile<T> &tl, int i, float4 &v, float4 &w)
{
    if constexpr (sizeof(T) == 4) {
        const Q4<T> a = tl.rec[4 * i + 0], b = tl.rec[4 * i + 1];
        v = make_float4(a.x, a.y, a.z, a.w);
        w = make_float4(b.x, b.y, b.z, b.w);
    } else {
        v = tl.ff[2 * i + 0];
        w = tl.ff[2 * i + 1];
    }
}

// Extra reach of a sphere test of the FP64 kernels (none in FP32, whose margins are in the spheres).
template <typename T>
__device__ __forceinline__ float sphere_margin(float av, float aw)
{
    return sizeof(T) == 4 ? 0.f : sph_margin_f32(av, aw);
}

// Whether the sphere reaches within lim of the wire; d2 = the squared distance of its centre.  A comparison
// that is not a number does not exclude: the spheres of a group with a track that is not finite hold it.
__device__ __forceinline__ bool sphere_within(const float4 &sp, const float4 &v, const float4 &w, float lim, float &d2)
{
    d2 = frame_dist2<float>(sp.x, sp.y, sp.z, v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w);
    const float l = lim + sp.w;
    return !(sp.w < 0.f) && !(d2 > l * l);
}

// Capture radius and frame of wire i of a staged tile (one thread per wire), packed with its
// point and direction into the wire's four records.
template <typename T>
__device__ __forceinline__ void tile_wire_setup(const Tile<T> &tl, int i, T lam, T *capv, Q4<T> *rec)
{
    const int hb = tl.offs[i], he = tl.offs[i + 1];
    T mr = T(-1);
    for (int j = hb; j < he; ++j)
        if (!tl.msm[j] && tl.dsm[j] > mr) mr = tl.dsm[j];
    const T cap = mr >= T(0) ? mr + lam : T(-1);
    capv[i] = cap;
    const T ax = tl.ax[i], ay = tl.ay[i], az = tl.az[i], ux = tl.ux[i], uy = tl.uy[i], uz = tl.uz[i];
    const WireFrame<T> fr = wire_frame<T>(ax, ay, az, ux, uy, uz);
    rec[4 * i + 0] = Q4<T>{fr.vx, fr.vy, fr.vz, fr.av};
    rec[4 * i + 1] = Q4<T>{fr.wx, fr.wy, fr.wz, fr.aw};
    rec[4 * i + 2] = Q4<T>{ax, ay, az, cap};
    rec[4 * i + 3] = Q4<T>{ux, uy, uz, T(0)};
}

// The float copies of an FP64 tile's frames, in the shared memory of its staged rows (read for the last
// time by tile_wire_setup: the caller's barrier lies between).
template <typename T>
__device__ __forceinline__ void tile_float_frames(const Q4<T> *rec, int wn, float4 *ff)
{
    if constexpr (sizeof(T) == 8)
        for (int i = threadIdx.x; i < 2 * wn; i += blockDim.x) {
            const Q4<T> r = rec[4 * (i >> 1) + (i & 1)];
            ff[i] = make_float4((float)r.x, (float)r.y, (float)r.z, (float)r.w);
        }
}

// Tighter reach of the refinement from an interior closest state (axial field): at a point of
// closest approach X* with distance D, the recorded state within delta <= h_rec/2 of it along the
// track is at most sqrt(D^2 + delta^2) + kappa delta^2 / 2 from the wire (the tangent line from
// X* moves away from the wire as sqrt(D^2 + delta^2 |t_perp|^2), the track leaves the tangent by
// at most kappa delta^2 / 2, kappa = |KAPPA q B / P0| its curvature).  So a closest recorded state
// farther than sqrt(cap^2 + (h_rec/2)^2) + kappa (h_rec/2)^2 / 2 cannot refine to D < cap: the
// wire adds lambda^2.  Returned: the warp's largest kappa times (h_rec/2)^2 / 2, plus the margin
// (infinite in other fields).
template <typename T, class F>
__device__ __forceinline__ T warp_curvature(const F &f, const Group<T> &gr)
{
    T kap = T(0);
    if constexpr (F::kAxial) {
        kap = fabs(gr.c * f.bz);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) kap = fmax(kap, __shfl_xor_sync(0xffffffffu, kap, off));
    }
    return kap;
}

template <typename T, class F>
__device__ __forceinline__ T interior_margin(const F &f, const DcaArgs &a, const Group<T> &gr)
{
    if constexpr (!F::kAxial) return T(INFINITY);
    const T half_rec = in_prec<T>(a.half_rec, a.half_rec_f);
    return T(0.5) * warp_curvature<T, F>(f, gr) * half_rec * half_rec + in_prec<T>(a.margin, a.margin_f);
}

// Lane m's one-state segments m that may hold a track end, a bit per super-segment: the first state, or
// between the warp's smallest and largest last state.  The others need only the interior reach.  (Formed
// once per item in the long form: tabulated field 638 -> 612 us; in the short form the registers it costs made
// 76,545 x 139 states 512 -> 530 us.)
template <typename T>
__device__ __forceinline__ uint32_t end_segments(const DcaArgs &a, const Group<T> &gr, int lane)
{
    uint32_t ends = 0;
    if (a.G1 == 1)
        for (int j = 0; j < gr.n0w; ++j) {
            const int k = j * a.G0 + lane;
            if (k == 0 || (k >= gr.elo && k <= gr.ehi)) ends |= 1u << j;
        }
    return ends;
}

// First refinement step, to the vertex of the parabola through the squared distances of the
// closest state and its two neighbours (exact for a straight track, where the squared distance is
// quadratic in arc length); then Newton steps as usual.  0 (none) unless both neighbours were
// looked at and the step budget allows (max_iter >= 4).
template <typename T>
__device__ __forceinline__ T first_step(const DcaArgs &a, T h_rec, T bdm, T bd, T bdp)
{
    T s0 = T(0);
    if (a.max_iter >= 4 && bdm < T(INFINITY) && bdp < T(INFINITY)) {
        const T den = bdm - T(2) * bd + bdp;
        if (den > T(0)) {
            s0 = T(0.5) * h_rec * (bdm - bdp) / den;
            s0 = fmin(fmax(s0, -h_rec), h_rec);
        }
    }
    return s0;
}

// Whether a wire has an unmasked hit (capture radius not negative; the sign bit, off the FP64 pipe).
template <typename T>
__device__ __forceinline__ bool has_hit(T cap)
{
    if constexpr (sizeof(T) == 4)
        return cap >= T(0);
    else
        return __double2hiint(cap) >= 0;
}

// Whether the squared distance a is below b (both not negative; as integers, which order alike and spare
// the FP64 pipe a comparison).  A NaN is below nothing.
template <typename T>
__device__ __forceinline__ bool nearer(T a, T b)
{
    if constexpr (sizeof(T) == 4)
        return a < b;
    else
        return (unsigned long long)__double_as_longlong(a) < (unsigned long long)__double_as_longlong(b);
}

// Wire ii's residual of Eq. 1 for a refined seed: the smallest |D - r| over its unmasked hits, capped at
// lambda (below lambda it counts into n_in).
template <typename T>
__device__ __forceinline__ T residual(const Tile<T> &tl, int ii, T D, T lam, int &nin)
{
    T emin = T(INFINITY);
    const int hb = tl.offs[ii], he = tl.offs[ii + 1];
    for (int j = hb; j < he; ++j) {
        if (tl.msm[j]) continue;
        const T e = fabs(D - tl.dsm[j]);
        if (nearer<T>(e, emin)) emin = e;
    }
    if (!nearer<T>(emin, lam)) return lam;
    ++nin;
    return emin;
}

// Shorter runs are scanned one state after the other with its momentum, longer ones two positions at a
// time and the momentum of the closest state loaded at the end (group_wires_short).  Recordings of 32 mm
// give runs of 1.5 states, where both ways cost the same; of 16 mm up to 13 in an odd lattice's wide
// groups: 76,545 seeds x 139 states all one by one 675 us, in pairs with momentum 569, so 514.
constexpr int kFewStates = 4;

// Runs of more than this many states are walked, not scanned (group_wires_long): a walk looks at about
// four states, costs as much as ten in FP32 (less in FP64, where distances are dear).
template <typename T>
constexpr int kWalkMin = sizeof(T) == 4 ? 10 : 4;

// Wires [wb, we) of one tile for one 32-seed group: accumulates d_i^2, n_in and unconverged counts.  Two
// forms with the same results.  SHORT: runs of a few candidate states (one-state segments), each scanned
// with its momentum loaded beside its position, so that the refinement starts without another round trip
// to memory (with few warps resident, latency counts as much as issue).  Otherwise group_wires_long:
// positions only, runs of many states walked, and the search bounded by the spheres when every DCA
// is wanted.  The short form is bound by instruction issue (72% of it used at 2^18 seeds), the refinement
// taking about half; the long one by the latency of the walk's loads in FP32, by the FP64 pipe in FP64.
// One form for all, with 64-bit addresses and momenta, and these, FP32: 2^18 seeds x 70 states 463 and 425 us,
// 76,545 x 139 592 and 510, 2^14 x 2,229 560 and 156, every DCA of 2^14 x 70 373 and 98; FP64: 4,096 x 2,229
// 808 and 245, 2^15 x 139 1415 and 970.
// Off: the byte offset of a recorded value, 32 bits when the track array is small enough.
template <typename T, class F, typename Off>
__device__ __forceinline__ void group_wires_short(const F &f, const DcaArgs &a, const Group<T> &gr,
                                                  const Tile<T> &tl, const float4 *sph0,
                                                  const float4 *sph1, int lane, Acc<T> &acc, int &nin,
                                                  int &nunc, int wb, int we)
{
    const int64_t S = a.S;
    const int64_t s = gr.s;
    const char *__restrict__ pts = (const char *)a.points;
    const Off row = (Off)S * (Off)sizeof(T), col = (Off)s * (Off)sizeof(T), plane = (Off)a.n_rec * row;
    auto val = [=](int c, Off o) { return *(const T *)(pts + (Off)(o + (Off)c * plane)); };
    const bool valid = gr.valid;
    const int nv = gr.nv;
    const T lam = in_prec<T>(a.lambda, a.lambda_f), tol = in_prec<T>(a.tol, a.tol_f),
            half_rec = in_prec<T>(a.half_rec, a.half_rec_f), h_rec = in_prec<T>(a.h_rec, a.h_rec_f);
    const int G0 = a.G0, G1 = a.G1;
    const int N1 = (G0 + G1 - 1) / G1;
    const Q4<T> *rec = tl.rec;
    const T kq2 = interior_margin<T, F>(f, a, gr);
    const T hq2 = half_rec * half_rec;

    for (int base = wb; base < we; base += 32) {
        const int clen = min(32, we - base);
        // lane t: which super-segments can bring wire base + t within its capture radius, and the wire's
        // interior reach
        uint32_t mask0 = 0;
        T thin_t = T(0);
        if (lane < clen) {
            const int iw = base + lane;
            const T capw = tl.cap[iw];
            if (capw >= T(0)) {
                float4 q0, q1;
                sphere_frame<T>(tl, iw, q0, q1);
                const float l = (float)(capw + half_rec) + sphere_margin<T>(q0.w, q1.w);
                for (int j = 0; j < gr.n0w; ++j) {
                    float d2;
                    if (sphere_within(sph0[j], q0, q1, l, d2)) mask0 |= 1u << j;
                }
                thin_t = fmin(capw + half_rec, sqrt(capw * capw + hq2) + kq2);
            }
        }
        for (int t = 0; t < clen; ++t) {
            const int ii = base + t;
            const uint32_t m0 = __shfl_sync(0xffffffffu, mask0, t);
            const Q4<T> r2 = rec[4 * ii + 2];
            const T cap = r2.w;
            const bool used = valid && has_hit<T>(cap);
            if (m0 == 0u) {
                // beyond every seed's capture radius (or no unmasked hit): lambda^2 if in the sum
                if (used) acc.add_square(lam);
                continue;
            }
            const T thin = __shfl_sync(0xffffffffu, thin_t, t);
            const Q4<T> r0 = rec[4 * ii + 0], r1 = rec[4 * ii + 1];
            const T capth = cap + half_rec;
            // the closest state so far, loaded with the scan (no second round trip to refine), and the
            // squared distances of the states scanned just before and after it (for the first
            // refinement step); the state scanned last: its distance, and whether it is the closest
            T bd = T(INFINITY), bdm = T(INFINITY), bdp = T(INFINITY), dprev = T(INFINITY);
            T by[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
            int bk = 0x7fffffff, kend = -1;
            bool last = false;
            float4 q0, q1;
            sphere_frame<T>(tl, ii, q0, q1);
            const float mg = sphere_margin<T>(q0.w, q1.w);
            uint32_t u0 = m0;
            while (u0) {
                const int j = __ffs(u0) - 1;
                u0 &= u0 - 1;
                // lane m tests level-1 segment m of super-segment j; a one-state segment
                // that may hold a track end (the first state, or between the warp's smallest
                // and largest last state) gets the refinement's extra half interval there;
                // one-state segments away from the track ends need only the interior reach
                const int k1 = j * G0 + lane;
                const bool end1 = G1 == 1 && (k1 == 0 || (k1 >= gr.elo && k1 <= gr.ehi));
                const float lim1 = (float)(G1 == 1 ? (end1 ? capth + half_rec : thin) : capth) + mg;
                float d2;
                const uint32_t u1 = __ballot_sync(0xffffffffu, lane < N1 && sphere_within(sph1[j * kN1Max + lane], q0, q1, lim1, d2));
                if (u1) {
                    // one contiguous range from the first to the last candidate level-1 segment (a
                    // superset of the candidates; their loads go out together), kU states at a time;
                    // ranges come in ascending order, so an equal distance never replaces the one found
                    const int k0 = j * G0 + (__ffs(u1) - 1) * G1;
                    const int ke = min(j * G0 + (32 - __clz(u1)) * G1, j * G0 + G0);
                    const int kv = used ? min(ke, nv) : 0;
                    if (k0 != kend) {
                        dprev = T(INFINITY);
                        last = false;
                    }
                    kend = ke;
                    auto dist = [&](T x, T y, T z) {
                        return frame_dist2<T>(x, y, z, r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w);
                    };
                    auto look = [&](int k, T d) {   // the next state's distance; whether it is the closest
                        const bool now = nearer<T>(d, bd);
                        if (last) bdp = d;
                        if (now) {
                            bdm = dprev;
                            bdp = T(INFINITY);
                            bd = d;
                            bk = k;
                        }
                        dprev = d;
                        last = now;
                        return now;
                    };
                    Off o = (Off)k0 * row + col;
                    if (ke - k0 < kFewStates) {
                        for (int k = k0; k < ke; ++k, o += row)
                            if (k < kv) {
                                T x[6];
#pragma unroll
                                for (int c = 0; c < 6; ++c) x[c] = val(c, o);
                                if (look(k, dist(x[0], x[1], x[2])))
#pragma unroll
                                    for (int c = 0; c < 6; ++c) by[c] = x[c];
                            }
                    } else {
                        const int before = bk;
                        for (int k = k0; k < ke; k += 2, o += 2 * row) {
                            T xa[3], xb[3];
                            if (k < kv)
#pragma unroll
                                for (int c = 0; c < 3; ++c) xa[c] = val(c, o);
                            if (k + 1 < kv)
#pragma unroll
                                for (int c = 0; c < 3; ++c) xb[c] = val(c, o + row);
                            if (k < kv) look(k, dist(xa[0], xa[1], xa[2]));
                            if (k + 1 < kv) look(k + 1, dist(xb[0], xb[1], xb[2]));
                        }
                        if (bk != before) {
                            o = (Off)bk * row + col;
#pragma unroll
                            for (int c = 0; c < 6; ++c) by[c] = val(c, o);
                        }
                    }
                }
            }

            // refinement from the closest recorded state, only where it can bring the wire within
            // its capture radius (group_wires_long)
            const T th = (bk == 0 || bk == nv - 1) ? capth + half_rec : thin;
            const bool refine = bk != 0x7fffffff && bd <= th * th;
            T d = lam;   // lambda when the wire is not refined
            if (refine) {
                T D;
                const Q4<T> r3 = rec[4 * ii + 3];
                const T s0 = first_step<T>(a, h_rec, bdm, bd, bdp);
                const int conv = refine_dca<T, F>(f, gr.c, gr.ip, by, r2.x, r2.y, r2.z, r3.x, r3.y, r3.z, tol,
                                                  a.max_iter, h_rec, D, s0);
                nunc += 1 - conv;
                d = residual<T>(tl, ii, D, lam, nin);
            }
            if (used) acc.add_square(d);
        }
    }
}

template <typename T, class F, typename Off, bool ALL, bool WIDE>
__device__ __forceinline__ void group_wires_long(const F &f, const DcaArgs &a, const Group<T> &gr,
                                            const Tile<T> &tl, const float4 *sph0,
                                            const float4 *sph1, int lane, Acc<T> &acc, int &nin,
                                            int &nunc, int wb, int we)
{
    const int64_t S = a.S;
    const int64_t s = gr.s;
    const char *__restrict__ pts = (const char *)a.points;
    const Off row = (Off)S * (Off)sizeof(T), col = (Off)s * (Off)sizeof(T), plane = (Off)a.n_rec * row;
    auto val = [=](int c, Off o) { return *(const T *)(pts + (Off)(o + (Off)c * plane)); };
    const bool valid = gr.valid;
    const int nv = gr.nv;
    const T lam = in_prec<T>(a.lambda, a.lambda_f), tol = in_prec<T>(a.tol, a.tol_f),
            half_rec = in_prec<T>(a.half_rec, a.half_rec_f), h_rec = in_prec<T>(a.h_rec, a.h_rec_f);
    const int G0 = a.G0, G1 = a.G1;
    const int N1 = (G0 + G1 - 1) / G1;
    const Q4<T> *rec = tl.rec;
    constexpr int kU = sizeof(T) == 8 && !ALL ? 2 : F::kAxial ? COMET_DCA_U : COMET_DCA_U_FIELD;
    const T kq2 = interior_margin<T, F>(f, a, gr);
    const uint32_t ends = end_segments<T>(a, gr, lane);
    // for the walk to the closest state (see below)
    [[maybe_unused]] float szw = 0.f, dcv_k = 0.f, hg_k = 0.f;
    if constexpr (F::kAxial) {
        szw = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(gr.sz)));
        const float kf = fmaxf((float)warp_curvature<T, F>(f, gr), 1e-6f);
        dcv_k = 0.8f / kf;
        hg_k = 0.25f * kf * a.h_rec_f * a.h_rec_f;
    }
    const T hq2 = half_rec * half_rec;
    const bool pruned = !ALL || sph0 != nullptr;   // no spheres: every state is scanned (dca_out without bounds)

    for (int base = wb; base < we; base += 32) {
        const int clen = min(32, we - base);
        // lane t: which super-segments can bring wire base + t within its capture radius
        uint32_t mask0 = 0;
        T thin_t = T(INFINITY);   // interior reach (see interior_margin), never above cap + half_rec
        [[maybe_unused]] float dcv_t = 0.f;   // distance below which wire base + t's valley is convex
        if (lane < clen) {
            const int iw = base + lane;
            const T capw = tl.cap[iw];
            if constexpr (F::kAxial) {
                const float uzf = fabsf((float)rec[4 * iw + 3].z);
                const float tau = szw * uzf + sqrtf(fmaxf(1.f - uzf * uzf, 0.f)) + 1e-3f;
                const float conv = 1.f - tau * tau;
                dcv_t = conv > 0.05f ? conv * dcv_k : 0.f;
            }
            if (ALL) {
                mask0 = (1u << gr.n0w) - 1u;
            } else if (capw >= T(0)) {
                thin_t = fmin(capw + half_rec, sqrt(capw * capw + hq2) + kq2);
                float4 q0, q1;
                sphere_frame<T>(tl, iw, q0, q1);
                const float l = (float)(capw + half_rec) + sphere_margin<T>(q0.w, q1.w);
                for (int j = 0; j < gr.n0w; ++j) {
                    float d2;
                    if (sphere_within(sph0[j], q0, q1, l, d2)) mask0 |= 1u << j;
                }
            }
        }
        for (int t = 0; t < clen; ++t) {
            const int ii = base + t;
            const uint32_t m0 = __shfl_sync(0xffffffffu, mask0, t);
            [[maybe_unused]] const float dcv = F::kAxial ? __shfl_sync(0xffffffffu, dcv_t, t) : 0.f;
            const Q4<T> r2 = rec[4 * ii + 2];
            const T cap = r2.w;
            const bool used = valid && has_hit<T>(cap);
            if (m0 == 0u) {
                // beyond every seed's capture radius (or no unmasked hit): lambda^2 if in the sum
                if (used) acc.add_square(lam);
                continue;
            }
            const Q4<T> r0 = rec[4 * ii + 0], r1 = rec[4 * ii + 1];
            const T thin = __shfl_sync(0xffffffffu, thin_t, t);
            const bool want = used || (valid && ALL);
            const T capth = ALL ? T(INFINITY) : cap + half_rec;
            // the closest state so far, and the squared distances of the states before and after it
            // (for the first refinement step; infinite where there is none or it was not looked at)
            T bd = T(INFINITY), bdm = T(INFINITY), bdp = T(INFINITY);
            int bk = 0x7fffffff;
            auto dist_at = [&](Off o) {
                return frame_dist2<T>(val(0, o), val(1, o), val(2, o), r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w);
            };
            // every state of [k0, k1) of this lane's seed (span is warp-uniform); ranges come in ascending
            // order, so an equal distance never replaces the one found
            auto scan = [&](int k0, int k1, int span) {
                T dprev = T(INFINITY);
                bool last = false;   // the previous state is the closest so far
                auto look = [&](int k, T d) {
                    const bool now = nearer<T>(d, bd);
                    bdp = now ? T(INFINITY) : (last ? d : bdp);
                    if (now) {
                        bdm = dprev;
                        bd = d;
                        bk = k;
                    }
                    dprev = d;
                    last = now;
                };
                k1 = want ? k1 : 0;
                int k = k0;
                Off o = (Off)k0 * row + col;
                // kU at a time without a condition between their loads, so that they wait for memory once
                // (past the lane's last state it is loaded again)
                for (; WIDE && span > 2; span -= kU, k += kU, o += kU * row) {
                    const int left = k1 - k;
                    T d[kU];
                    if (left > 0) {
                        T x[kU][3];
                        Off ou = o;
#pragma unroll
                        for (int u = 0; u < kU; ++u) {
#pragma unroll
                            for (int c = 0; c < 3; ++c) x[u][c] = val(c, ou);
                            if (u + 1 < left) ou += row;
                        }
#pragma unroll
                        for (int u = 0; u < kU; ++u)
                            d[u] = u < left ? frame_dist2<T>(x[u][0], x[u][1], x[u][2], r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w)
                                            : T(INFINITY);
                    } else {
#pragma unroll
                        for (int u = 0; u < kU; ++u) d[u] = T(INFINITY);
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u) look(k + u, d[u]);
                }
                for (; span > 0; span -= 2, k += 2, o += 2 * row) {
                    T d[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) d[u] = k + u < k1 ? dist_at(o + u * row) : T(INFINITY);
#pragma unroll
                    for (int u = 0; u < 2; ++u) look(k + u, d[u]);
                }
            };
            // The closest state of a run [ra, rb] of candidate states.  Axial field: down the valley from a
            // start state, without scanning it.  Along a track f = d^2 / 2 has f'' = |t_perp|^2 + e . dt/ds
            // >= 1 - (t.u)^2 - kappa d, and |t.u| <= |tz uz| + sqrt(1 - uz^2) (tz = pz / P0 is constant), so
            // f'' >= 0.2 (1 - tau^2) wherever d <= dcv = 0.8 (1 - tau^2) / kappa.  Where that holds for the
            // whole run (its states lie at most their arc length farther than the state found), a state
            // with no closer neighbour is its closest.  Rounding: two states beyond the found one d^2 has
            // grown by 0.4 (1 - tau^2) h^2, which hg requires to be above 16 d times an eighth of the search
            // margin, the rounding of a distance.  A warp with a lane that does not meet this, or that is
            // not there after kSteps moves, scans the run.
            // The neighbours' distances are handed on where a scan of the run would have them, so both ways
            // give the same bits.  A walk that leaves the run adds nothing: the run's closest state is then
            // its boundary, farther than the state found, which is another run's to find or, in no run, is out
            // of reach (and the boundary with it, unless it is the track's end: such a run is scanned).
            auto closest_in = [&](int ra, int rb, int kst) {
                const int side = ALL ? 1 : 0;   // a scan of every state knows all neighbours
                if constexpr (F::kAxial)
                    if (rb - ra >= kWalkMin<T>) {
                        bool ok = true, here = false;
                        T d0 = T(INFINITY), dm = T(INFINITY), dp = T(INFINITY);
                        int k = 0;
                        if (want && nv > ra) {
                            k = min(kst, nv - 1);
                            if (G1 > 1) {
                                // the start is a segment's centre, several states from this lane's closest:
                                // one Newton step of d^2 along the track's tangent, in whole states
                                float4 v, w;
                                sphere_frame<T>(tl, ii, v, w);
                                const Off o = (Off)k * row + col;
                                const float x = (float)val(0, o), y = (float)val(1, o), z = (float)val(2, o);
                                const float px = (float)val(3, o), py = (float)val(4, o), pz = (float)val(5, o);
                                const float ev = fmaf(x, v.x, fmaf(y, v.y, fmaf(z, v.z, -v.w)));
                                const float ew = fmaf(x, w.x, fmaf(y, w.y, fmaf(z, w.z, -w.w)));
                                const float pv = px * v.x + py * v.y + pz * v.z, pw = px * w.x + py * w.y + pz * w.z;
                                const float n = __fdividef(-(ev * pv + ew * pw),
                                                           (pv * pv + pw * pw) * (float)gr.ip * a.h_rec_f);
                                k = max(0, min(k + (int)rintf(fminf(fmaxf(n, -256.f), 256.f)), nv - 1));
                            }
                            Off o = (Off)k * row + col;
                            d0 = dist_at(o);
                            if (k > 0) dm = dist_at(o - row);
                            if (k < nv - 1) dp = dist_at(o + row);
                            constexpr int kSteps = 6;
                            for (int it = 0; it < kSteps && (dm <= d0 || dp < d0); ++it) {
                                if (dm <= d0) {
                                    --k;
                                    o -= row;
                                    dp = d0;
                                    d0 = dm;
                                    dm = k > 0 ? dist_at(o - row) : T(INFINITY);
                                } else {
                                    ++k;
                                    o += row;
                                    dm = d0;
                                    d0 = dp;
                                    dp = k < nv - 1 ? dist_at(o + row) : T(INFINITY);
                                }
                            }
                            const float far = dcv - a.h_rec_f * (float)(1 + max(k - ra, min(rb, nv - 1) - k));
                            const float hg = hg_k * dcv, f0 = (float)d0;
                            here = k >= ra && k <= rb;
                            ok = !(dm <= d0 || dp < d0) && far > 0.f && f0 <= far * far &&
                                 f0 * (a.margin_f * a.margin_f) <= hg * hg && (ALL || k >= ra || ra < nv - 1);
                        }
                        if (__all_sync(0xffffffffu, ok)) {
                            if (here && (d0 < bd || (d0 == bd && k < bk))) {
                                bd = d0;
                                bk = k;
                                bdm = k > ra - side ? dm : T(INFINITY);
                                bdp = k < rb + side ? dp : T(INFINITY);
                            }
                            return;
                        }
                    }
                const int k0 = max(ra - side, 0);
                scan(k0, min(rb + 1 + side, nv), rb + 1 + side - k0);
            };
            if (!pruned) {
                scan(0, nv, gr.ehi + 1);
            } else {
                float4 q0, q1;
                sphere_frame<T>(tl, ii, q0, q1);
                const float mg = sphere_margin<T>(q0.w, q1.w);
                float lim_end = (float)(capth + half_rec) + mg, lim_in = (float)(G1 == 1 ? thin : capth) + mg;
                if (ALL) {
                    // no state of any lane's closest is farther than the nearest sphere that all lanes have
                    // reaches: spheres beyond it hold no closest state
                    float ub = INFINITY;
                    for (int j = 0; j < gr.n0w; ++j) {
                        const float4 sp = lane < N1 ? sph1[j * kN1Max + lane] : make_float4(0.f, 0.f, 0.f, -1.f);
                        float d2;
                        if (j * G0 + lane * G1 <= gr.elo && sphere_within(sp, q0, q1, INFINITY, d2))
                            ub = fminf(ub, sqrtf(d2) + sp.w);
                    }
                    lim_in = lim_end = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(ub))) +
                                       a.margin_f + 2.f * mg;
                }
                // Runs of candidate level-1 segments, super-segment by super-segment (lane m tests segment
                // m); a run that goes on into the next super-segment is one run.
                uint32_t u0 = m0;
                int ra = -1, rb = -1, kst = 0;
                uint32_t near = 0xffffffffu;
                for (bool more = true; more;) {
                    more = false;
                    int j = 0;
                    uint32_t u1 = 0, key = 0;
                    while (u0) {
                        j = __ffs(u0) - 1;
                        u0 &= u0 - 1;
                        // a segment that may hold a track end gets the refinement's extra half interval
                        float d2 = 0.f;
                        bool hit1 = false;
                        if (lane < N1) {
                            const float4 sp = sph1[j * kN1Max + lane];
                            hit1 = sphere_within(sp, q0, q1, ends >> j & 1u ? lim_end : lim_in, d2);
                        }
                        u1 = __ballot_sync(0xffffffffu, hit1);
                        if (u1) {
                            if constexpr (F::kAxial)
                                key = __reduce_min_sync(0xffffffffu,
                                                        hit1 ? (__float_as_uint(d2) & ~31u) | (unsigned)lane : 0xffffffffu);
                            more = true;
                            break;
                        }
                    }
                    const int k0 = j * G0 + (__ffs(u1) - 1) * G1;
                    const bool joins = more && ra >= 0 && k0 <= rb + 1;
                    if (!joins && ra >= 0) closest_in(ra, rb, kst);
                    if (more) {
                        if (!joins) {
                            ra = k0;
                            near = 0xffffffffu;
                        }
                        rb = min(j * G0 + (32 - __clz(u1)) * G1, min(j * G0 + G0, a.n_rec)) - 1;
                        if ((key & ~31u) < near) {
                            near = key & ~31u;
                            kst = segment_centre(j * G0 + (int)(key & 31u) * G1, G1, min(j * G0 + G0, a.n_rec));
                        }
                    }
                }
            }

            if constexpr (ALL) {
                // no squared distance is below infinity: the first that overflows, if there is one
                if (want && bk == 0x7fffffff)
                    for (int k = 0; k < nv && bk == 0x7fffffff; ++k)
                        if (dist_at((Off)k * row + col) == T(INFINITY)) bk = k;
            }

            // refinement from the closest recorded state, only where it can bring the wire within
            // its capture radius: from an interior state within the interior reach thin, from the
            // first or the last recorded state within a whole interval more than capth (the
            // refinement may extrapolate h_rec beyond the track); compared squared: the thresholds
            // carry margins far above the rounding of the square
            const T th = (bk == 0 || bk == nv - 1) ? capth + half_rec : thin;
            const bool refine = want && bk != 0x7fffffff && (ALL || !nearer<T>(th * th, bd));
            T d = lam;   // lambda when the wire is not refined
            if (refine) {
                T D;
                T yv[6];
                const Off o = (Off)bk * row + col;
                yv[0] = val(0, o);
                yv[1] = val(1, o);
                yv[2] = val(2, o);
                yv[3] = val(3, o);
                yv[4] = val(4, o);
                yv[5] = val(5, o);
                const Q4<T> r3 = rec[4 * ii + 3];
                const T s0 = first_step<T>(a, h_rec, bdm, bd, bdp);
                const int conv = refine_dca<T, F>(f, gr.c, gr.ip, yv, r2.x, r2.y, r2.z, r3.x, r3.y, r3.z, tol,
                                                  a.max_iter, h_rec, D, s0);
                if (ALL) ((T *)a.dca_out)[(int64_t)(tl.w0 + ii) * S + s] = D;
                if (used) {
                    nunc += 1 - conv;
                    d = residual<T>(tl, ii, D, lam, nin);
                }
            } else if (ALL && want) {
                ((T *)a.dca_out)[(int64_t)(tl.w0 + ii) * S + s] = T(NAN);   // no state has a distance
            }
            if (used) acc.add_square(d);
        }
    }
}

// How a launch searches for the closest states.
enum Search { kShort, kFew, kLong, kAll };   // runs of a few states (two ways); runs of many; every DCA wanted

template <typename T, class F, typename Off, Search HOW>
__device__ __forceinline__ void group_wires(const F &f, const DcaArgs &a, const Group<T> &gr,
                                            const Tile<T> &tl, const float4 *sph0,
                                            const float4 *sph1, int lane, Acc<T> &acc, int &nin,
                                            int &nunc, int wb, int we)
{
    if constexpr (HOW == kShort)
        group_wires_short<T, F, Off>(f, a, gr, tl, sph0, sph1, lane, acc, nin, nunc, wb, we);
    else
        group_wires_long<T, F, Off, HOW == kAll, HOW != kFew>(f, a, gr, tl, sph0, sph1, lane, acc, nin, nunc, wb, we);
}

// Wire chunk c of n over W wires: [c * wc, min((c + 1) * wc, W)), wc = ceil(W / n).
__device__ __forceinline__ int2 chunk_range(int W, int n, int c)
{
    const int wc = (W + n - 1) / n;
    return make_int2(min(c * wc, W), min((c + 1) * wc, W));
}

// All wire chunks of one group in this warp: each chunk's partial sum, added in chunk order (the
// arithmetic the cross-warp schedule of the persistent kernel reproduces).
template <typename T, class F, typename Off, Search HOW>
__device__ __forceinline__ void group_all_chunks(const F &f, const DcaArgs &a, const Group<T> &gr,
                                                 const Tile<T> &tl, const float4 *sph0,
                                                 const float4 *sph1, int lane, Acc<T> &acc,
                                                 int &nin, int &nunc)
{
    for (int c = 0; c < a.n_chunks; ++c) {
        const int2 r = chunk_range(tl.wn, a.n_chunks, c);
        Acc<T> part;
        group_wires<T, F, Off, HOW>(f, a, gr, tl, sph0, sph1, lane, part, nin, nunc, r.x, r.y);
        acc.add_pair(part.hi, part.lo);
    }
}

// Waits for a staging transaction of `bytes` (thread 0 issued it; everyone waits) for at most
// wait_ns; wait_ns = 0 gives up at once without waiting (the context's test setting).  Returns true
// if the wait gave up anywhere in the CTA: the caller then re-reads the data with plain loads and,
// before its shared memory or barrier is used again, waits (up to kWaitNs) for the abandoned copy.
__device__ __forceinline__ bool finish_stage(uint64_t *bar, uint32_t &parity, uint32_t bytes,
                                             uint64_t wait_ns)
{
    bool to = false;
    if (bytes > 0) {
        to = wait_ns == 0 ? true : !mbar_wait(bar, parity, wait_ns);
        parity ^= 1u;
    }
    return __syncthreads_or(to);
}

// ------------------------------------------------------------------------------------------------
// The seed of lowest RSS, selected inside the DCA launch (optional; the k = 1 case of
// comet_scan_select, in its order: ascending RSS, NaN after every number, ties by lowest index).
// The warp that finalises a group folds the group's best into its warp's best (shared memory); at
// the end each CTA folds its warps into a slot, and the last CTA to finish folds the slots.
// ------------------------------------------------------------------------------------------------

template <typename T>
struct Best {
    T v;
    int64_t i;
};

template <typename T>
__device__ __forceinline__ T nan_value()
{
    if constexpr (sizeof(T) == 4)
        return __int_as_float(0x7fc00000);
    else
        return __longlong_as_double(0x7ff8000000000000ll);
}

template <typename T>
__device__ __forceinline__ Best<T> best_none()
{
    return Best<T>{nan_value<T>(), INT64_MAX};
}

// (v, i) before (b.v, b.i) in comet_scan_select's order
template <typename T>
__device__ __forceinline__ bool precedes(T v, int64_t i, const Best<T> &b)
{
    const bool vn = v != v, bn = b.v != b.v;
    if (vn != bn) return bn;
    if (!vn && v != b.v) return v < b.v;
    return i < b.i;
}

template <typename T>
__device__ __forceinline__ void best_fold(Best<T> &b, T v, int64_t i)
{
    if (precedes<T>(v, i, b)) {
        b.v = v;
        b.i = i;
    }
}

// The best of the warp's 32 candidates, in every lane.
template <typename T>
__device__ __forceinline__ Best<T> warp_best(Best<T> b)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const T v = __shfl_xor_sync(0xffffffffu, b.v, off);
        const int64_t i = __shfl_xor_sync(0xffffffffu, b.i, off);
        best_fold<T>(b, v, i);
    }
    return b;
}

// A finalised group: the best of its valid seeds folded into this warp's best (s_warp[warp]).
template <typename T>
__device__ __forceinline__ void group_best_fold(Best<T> *s_warp, int warp, int lane, bool valid, T rss,
                                                int64_t s)
{
    Best<T> b = valid ? Best<T>{rss, s} : best_none<T>();
    b = warp_best<T>(b);
    if (lane == 0) best_fold<T>(s_warp[warp], b.v, b.i);
}

// End of the launch (every thread of the CTA): the CTA's best into its slot; the last CTA to finish
// folds every slot and writes the selection, then leaves the counter at zero for the next launch.
template <typename T>
__device__ __forceinline__ void finish_best(const DcaArgs &a, Best<T> *s_warp, int *s_last)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int64_t *slot_i = (int64_t *)a.best_slots;
    T *slot_v = (T *)(slot_i + gridDim.x);
    __syncthreads();
    if (tid == 0) {
        Best<T> b = s_warp[0];
        for (int w = 1; w < kWarps; ++w) best_fold<T>(b, s_warp[w].v, s_warp[w].i);
        slot_i[blockIdx.x] = b.i;
        slot_v[blockIdx.x] = b.v;
        __threadfence();
        const unsigned int t = atomicAdd(a.best_counter, 1u);
        *s_last = t == gridDim.x - 1;
    }
    __syncthreads();
    if (*s_last) {
        __threadfence();
        Best<T> b = best_none<T>();
        for (unsigned int k = tid; k < gridDim.x; k += blockDim.x) best_fold<T>(b, __ldcg(slot_v + k), __ldcg(slot_i + k));
        b = warp_best<T>(b);
        if (lane == 0) s_warp[warp] = b;
        __syncthreads();
        if (tid == 0) {
            Best<T> r = s_warp[0];
            for (int w = 1; w < kWarps; ++w) best_fold<T>(r, s_warp[w].v, s_warp[w].i);
            *a.best_idx_out = r.i;
            if (a.best_rss_out) *(T *)a.best_rss_out = r.v;
            *a.best_counter = 0u;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Persistent kernel: all wires fit one shared-memory tile (the common case).  Each CTA stages the
// wires and hits once; each warp then takes work items -- (32-seed group, wire chunk) pairs, or
// whole groups when no partial-sum scratch is given -- from a device counter until none is left,
// with no CTA-wide barrier between items.
// ------------------------------------------------------------------------------------------------

struct PLayout {
    size_t sph, wrow, orow, cap, frame, drift, mask, total;
    int wcap;
    int nsph;    // float4 sphere entries per warp
};

// Sphere entries each warp keeps in shared memory: the whole table (built here) when no bounds
// table was given; with the recording kernel's table, the part a group can use -- its kN0Max
// super-segment spheres and the level-1 spheres of the super-segments an n_rec-state track has --
// copied in per work item (about 1.3 KB per warp at 70 recorded states, so that the per-wire
// level-1 tests read shared memory, not L2); none when every state is scanned (dca_out requested and
// no table given).
__host__ __device__ inline int p_sph_entries(const DcaArgs &a)
{
    if (a.bounds == nullptr) return a.exact_all ? 0 : kBoundsPerGroup;
    int n0 = (a.n_rec + a.G0 - 1) / a.G0;
    n0 = n0 < kN0Max ? n0 : kN0Max;
    return kN0Max + n0 * kN1Max;
}

__host__ __device__ inline PLayout p_layout(int W, int es, int nsph)
{
    PLayout L;
    int wc = ((W + 31) / 32) * 32;
    wc = wc < 32 ? 32 : wc;
    L.wcap = wc;
    L.nsph = nsph;
    L.sph = 16;
    L.wrow = align16(L.sph + (size_t)16 * kWarps * nsph);
    L.orow = align16(L.wrow + (size_t)es * 6 * (wc + 32));
    L.cap = align16(L.orow + (size_t)4 * (wc + 40));
    L.frame = align16(L.cap + (size_t)es * wc);
    L.drift = align16(L.frame + (size_t)es * 16 * wc);
    L.mask = align16(L.drift + (size_t)es * kHitCap);
    L.total = align16(L.mask + kHitCap);
    return L;
}

constexpr int kPersistMaxW = 1024;

// Every DCA wanted: a group whose tracks all have fewer states than this is scanned without spheres, whose table
// is not even loaded.  All tracks out of the region at once (with spheres, without): 2^14 seeds recorded for up
// to 2,192 states 126 and 76 us, for 137 73 and 62, 59,535 seeds 194 and 182; with 3 to 22 states 2^14 seeds take
// 92 us either way, above that the spheres are faster.
constexpr int kFewForSpheres = 8;

template <typename T, Search HOW>
__device__ __forceinline__ bool use_spheres(const DcaArgs &a, const Group<T> &gr)
{
    return HOW != kAll || (a.bounds && gr.ehi + 1 >= kFewForSpheres);
}

// Resident CTAs per SM that the registers are allocated for.
template <typename T, class F>
constexpr int min_ctas(Search how)
{
    return sizeof(T) == 8 ? COMET_DCA_MINB_F64
                          : (!F::kAxial ? COMET_DCA_MINB_FIELD : (how == kLong ? COMET_DCA_MINB_LONG : COMET_DCA_MINB));
}

template <typename T, class F, typename Off, Search HOW>
__global__ void __launch_bounds__(kThreads, min_ctas<T, F>(HOW)) dca_persistent_kernel(F f, DcaArgs a)
{
    const bool sph_smem = a.bounds == nullptr && !a.exact_all;
    const PLayout L = p_layout(a.W, (int)sizeof(T), p_sph_entries(a));
    extern __shared__ __align__(128) unsigned char sm[];
    uint64_t *bar = (uint64_t *)sm;
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    float4 *sph0 = (float4 *)(sm + L.sph) + warp * L.nsph;
    float4 *sph1 = sph0 + kN0Max;
    T *wrow = (T *)(sm + L.wrow);
    int32_t *orow = (int32_t *)(sm + L.orow);
    T *capv = (T *)(sm + L.cap);
    Q4<T> *frm = (Q4<T> *)(sm + L.frame);
    T *dsm = (T *)(sm + L.drift);
    uint8_t *msm = (uint8_t *)(sm + L.mask);
    const int rcap = L.wcap + 32;
    const T *__restrict__ Wg = (const T *)a.wires;
    const T *__restrict__ Dg = (const T *)a.drift;
    const int W = a.W;
    const int H = W > 0 ? a.offs[W] : 0;
    const bool hits_sm = H <= kHitMax;
    __shared__ Best<T> s_best[kWarps];
    __shared__ int s_last;

    if (tid == 0) mbar_init(bar, 1);
    if (lane == 0) s_best[warp] = best_none<T>();
    __syncthreads();

    // ---- stage wires, offsets and (when they fit) hits: one bulk-copy transaction (W > 0 only:
    // with no wires the pointers may be NULL and every RSS is 0)
    uint32_t parity = 0;
    uint32_t bytes = 0;
    int woff[6] = {0, 0, 0, 0, 0, 0};
    int ooff = 0, doff = 0, moff = 0;
    if (W > 0) {
        bytes = stage_bytes<int32_t>(a.offs, W + 1);
#pragma unroll
        for (int r = 0; r < 6; ++r) bytes += stage_bytes<T>(Wg + (size_t)r * a.ldw, W);
        if (hits_sm && H > 0) bytes += stage_bytes<T>(Dg, H) + stage_bytes<uint8_t>(a.mask, H);
        if (tid == 0 && bytes > 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bar, bytes);
        }
#pragma unroll
        for (int r = 0; r < 6; ++r)
            woff[r] = stage_issue<T>(wrow + r * rcap, Wg + (size_t)r * a.ldw, W, bar, tid == 0);
        ooff = stage_issue<int32_t>(orow, a.offs, W + 1, bar, tid == 0);
        if (hits_sm && H > 0) {
            doff = stage_issue<T>(dsm, Dg, H, bar, tid == 0);
            moff = stage_issue<uint8_t>(msm, a.mask, H, bar, tid == 0);
        }
    }
    const bool any_timeout = finish_stage(bar, parity, bytes, a.wait_ns);
    if (any_timeout && W > 0) {
#pragma unroll
        for (int r = 0; r < 6; ++r) stage_fallback<T>(wrow + r * rcap, Wg + (size_t)r * a.ldw, W);
        stage_fallback<int32_t>(orow, a.offs, W + 1);
        if (hits_sm && H > 0) {
            stage_fallback<T>(dsm, Dg, H);
            stage_fallback<uint8_t>(msm, a.mask, H);
        }
    }
    __syncthreads();
    Tile<T> tl;
    tl.ax = wrow + 0 * rcap + woff[0];
    tl.ay = wrow + 1 * rcap + woff[1];
    tl.az = wrow + 2 * rcap + woff[2];
    tl.ux = wrow + 3 * rcap + woff[3];
    tl.uy = wrow + 4 * rcap + woff[4];
    tl.uz = wrow + 5 * rcap + woff[5];
    tl.rec = frm;
    tl.cap = capv;
    tl.offs = orow + ooff;
    tl.dsm = hits_sm ? dsm + doff : Dg;
    tl.msm = hits_sm ? msm + moff : a.mask;
    tl.w0 = 0;
    tl.wn = W;
    tl.ff = (const float4 *)wrow;
    for (int i = tid; i < W; i += kThreads) tile_wire_setup<T>(tl, i, in_prec<T>(a.lambda, a.lambda_f), capv, frm);
    __syncthreads();
    if constexpr (sizeof(T) == 8) {
        // a copy given up on above may still land in the rows
        if (any_timeout) mbar_wait(bar, parity ^ 1u, kWaitNs);
        tile_float_frames<T>(frm, W, (float4 *)wrow);
        __syncthreads();
    }

    // ---- work items taken dynamically by each warp: 32-seed groups, or (group, wire chunk) pairs
    // when partial sums can be parked in `part` (finer items balance the warps' loads)
    const int64_t n_groups = (a.S + 31) / 32;
    const bool split = a.n_chunks > 1 && a.part && a.arrive;
    const int nc = split ? a.n_chunks : 1;
    const int64_t n_items = n_groups * nc;
    int nunc = 0;
    for (;;) {
        unsigned int it = 0;
        if (lane == 0) it = atomicAdd((unsigned int *)a.counter, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if ((int64_t)it >= n_items) break;
        const int64_t g = (int64_t)(it / (unsigned)nc);
        const int c = (int)(it % (unsigned)nc);
        const Group<T> gr = load_group<T>(a, g, lane);
        const bool spheres = use_spheres<T, HOW>(a, gr);
        if (sph_smem) {
            build_spheres<T>(a, gr, lane, sph0, sph1, g);
        } else if (spheres) {
            // the usable part of this group's table from the recording kernel
            const float4 *src = (const float4 *)a.bounds + g * kBoundsPerGroup;
            for (int i = lane; i < L.nsph; i += 32) sph0[i] = __ldg(src + i);
            __syncwarp();
        }
        const float4 *s0 = spheres ? sph0 : nullptr, *s1 = sph1;
        Acc<T> acc;
        int nin = 0;
        if (!split) {
            group_all_chunks<T, F, Off, HOW>(f, a, gr, tl, s0, s1, lane, acc, nin, nunc);
            const T v = acc.value();
            if (gr.valid) {
                ((T *)a.rss)[gr.s] = v;
                a.n_in[gr.s] = nin;
            }
            if (a.best_idx_out) group_best_fold<T>(s_best, warp, lane, gr.valid, v, gr.s);
        } else {
            const int2 r = chunk_range(W, nc, c);
            group_wires<T, F, Off, HOW>(f, a, gr, tl, s0, s1, lane, acc, nin, nunc, r.x, r.y);
            T *ph = (T *)a.part;
            T *pl = ph + (size_t)nc * a.S;
            int32_t *pn = (int32_t *)(pl + (size_t)nc * a.S);
            if (gr.valid) {
                ph[(int64_t)c * a.S + gr.s] = acc.hi;
                pl[(int64_t)c * a.S + gr.s] = acc.lo;
                pn[(int64_t)c * a.S + gr.s] = nin;
            }
            __threadfence();
            __syncwarp();
            unsigned int done = 0;
            if (lane == 0) done = atomicAdd(a.arrive + g, 1u);
            done = __shfl_sync(0xffffffffu, done, 0);
            if (done == (unsigned)(nc - 1)) {
                // the group's last chunk: add the partial sums in chunk order
                __threadfence();
                T v = T(0);
                if (gr.valid) {
                    Acc<T> tot;
                    int nt = 0;
                    for (int k = 0; k < nc; ++k) {
                        const int64_t o = (int64_t)k * a.S + gr.s;
                        tot.add_pair(__ldcg(ph + o), __ldcg(pl + o));
                        nt += __ldcg(pn + o);
                    }
                    v = tot.value();
                    ((T *)a.rss)[gr.s] = v;
                    a.n_in[gr.s] = nt;
                }
                if (a.best_idx_out) group_best_fold<T>(s_best, warp, lane, gr.valid, v, gr.s);
                if (lane == 0) a.arrive[g] = 0u;   // left zero for the next launch
            }
        }
        __syncwarp();   // the next group's spheres overwrite this warp's slot
    }
    if (a.n_unconv) {
        int t = nunc;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0 && t) atomicAdd(a.n_unconv, t);
    }
    if (a.best_idx_out) finish_best<T>(a, s_best, &s_last);
    if (any_timeout) {
        if (tid == 0 && a.status) atomicOr(a.status, 1);
        mbar_wait(bar, parity ^ 1u, kWaitNs);
    }
}

// ------------------------------------------------------------------------------------------------
// Tiled kernel: more wires than one tile holds.  One 128-seed block per CTA; wires staged in tiles.
// ------------------------------------------------------------------------------------------------

template <typename T, class F, typename Off, Search HOW>
__global__ void __launch_bounds__(kThreads, min_ctas<T, F>(HOW)) dca_tiled_kernel(F f, DcaArgs a)
{
    using L = Smem<T>;
    extern __shared__ __align__(128) unsigned char sm[];
    uint64_t *bar = (uint64_t *)(sm + L::bar);
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    float4 *sph0 = (float4 *)(sm + L::sph0) + warp * kN0Max;
    float4 *sph1 = (float4 *)(sm + L::sph1) + warp * kN0Max * kN1Max;
    T *wrow = (T *)(sm + L::wrow);
    int32_t *orow = (int32_t *)(sm + L::orow);
    T *capv = (T *)(sm + L::cap);
    Q4<T> *frm = (Q4<T> *)(sm + L::frame);
    T *dsm = (T *)(sm + L::drift);
    uint8_t *msm = (uint8_t *)(sm + L::mask);
    const T *__restrict__ Wg = (const T *)a.wires;
    const T *__restrict__ Dg = (const T *)a.drift;

    if (tid == 0) mbar_init(bar, 1);
    const int64_t g = (int64_t)blockIdx.x * kWarps + warp;
    const Group<T> gr = load_group<T>(a, g, lane);
    const bool pruned = use_spheres<T, HOW>(a, gr);
    if (pruned) build_spheres<T>(a, gr, lane, sph0, sph1, g);

    const int W = a.W;
    const int H = W > 0 ? a.offs[W] : 0;
    const bool hits_sm = H <= kHitMax;
    uint32_t parity = 0;
    bool any_timeout = false;
    int doff = 0, moff = 0;
    __syncthreads();   // barrier initialised

    if (hits_sm && H > 0) {
        const uint32_t bytes = stage_bytes<T>(Dg, H) + stage_bytes<uint8_t>(a.mask, H);
        if (tid == 0 && bytes > 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bar, bytes);
        }
        doff = stage_issue<T>(dsm, Dg, H, bar, tid == 0);
        moff = stage_issue<uint8_t>(msm, a.mask, H, bar, tid == 0);
        if (finish_stage(bar, parity, bytes, a.wait_ns)) {
            any_timeout = true;
            stage_fallback<T>(dsm, Dg, H);
            stage_fallback<uint8_t>(msm, a.mask, H);
            // the barrier is reused by the wire tiles: let the abandoned copy land first (bounded)
            mbar_wait(bar, parity ^ 1u, kWaitNs);
        }
        __syncthreads();
    }

    Acc<T> acc;
    int nin = 0, nunc = 0;
    for (int w0 = 0; w0 < W; w0 += kWireTile) {
        const int wn = min(kWireTile, W - w0);
        uint32_t bytes = stage_bytes<int32_t>(a.offs + w0, wn + 1);
#pragma unroll
        for (int r = 0; r < 6; ++r) bytes += stage_bytes<T>(Wg + (size_t)r * a.ldw + w0, wn);
        if (tid == 0 && bytes > 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bar, bytes);
        }
        int woff[6];
#pragma unroll
        for (int r = 0; r < 6; ++r)
            woff[r] = stage_issue<T>(wrow + r * kWireCap, Wg + (size_t)r * a.ldw + w0, wn, bar, tid == 0);
        const int ooff = stage_issue<int32_t>(orow, a.offs + w0, wn + 1, bar, tid == 0);
        if (finish_stage(bar, parity, bytes, a.wait_ns)) {
            any_timeout = true;
#pragma unroll
            for (int r = 0; r < 6; ++r)
                stage_fallback<T>(wrow + r * kWireCap, Wg + (size_t)r * a.ldw + w0, wn);
            stage_fallback<int32_t>(orow, a.offs + w0, wn + 1);
            // the next tile reuses these buffers and the barrier: let the abandoned copy land
            // first (bounded)
            mbar_wait(bar, parity ^ 1u, kWaitNs);
        }
        __syncthreads();
        Tile<T> tl;
        tl.ax = wrow + 0 * kWireCap + woff[0];
        tl.ay = wrow + 1 * kWireCap + woff[1];
        tl.az = wrow + 2 * kWireCap + woff[2];
        tl.ux = wrow + 3 * kWireCap + woff[3];
        tl.uy = wrow + 4 * kWireCap + woff[4];
        tl.uz = wrow + 5 * kWireCap + woff[5];
        tl.rec = frm;
        tl.cap = capv;
        tl.offs = orow + ooff;
        tl.dsm = hits_sm ? dsm + doff : Dg;
        tl.msm = hits_sm ? msm + moff : a.mask;
        tl.w0 = w0;
        tl.wn = wn;
        tl.ff = (const float4 *)wrow;
        for (int i = tid; i < wn; i += kThreads) tile_wire_setup<T>(tl, i, in_prec<T>(a.lambda, a.lambda_f), capv, frm);
        __syncthreads();
        if constexpr (sizeof(T) == 8) {
            tile_float_frames<T>(frm, wn, (float4 *)wrow);
            __syncthreads();
        }
        group_wires<T, F, Off, HOW>(f, a, gr, tl, pruned ? sph0 : nullptr, sph1, lane, acc, nin, nunc, 0, wn);
        if (w0 + kWireTile < W) {
            // tile consumed before the next staging's bulk copies overwrite it
            fence_proxy_async_smem();
            __syncthreads();
        }
    }

    const T v = acc.value();
    if (gr.valid) {
        ((T *)a.rss)[gr.s] = v;
        a.n_in[gr.s] = nin;
    }
    if (a.n_unconv) {
        int t = nunc;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0 && t) atomicAdd(a.n_unconv, t);
    }
    if (a.best_idx_out) {
        __shared__ Best<T> s_best[kWarps];
        __shared__ int s_last;
        if (lane == 0) s_best[warp] = best_none<T>();
        __syncwarp();
        group_best_fold<T>(s_best, warp, lane, gr.valid, v, gr.s);
        finish_best<T>(a, s_best, &s_last);
    }
    if (any_timeout && tid == 0 && a.status) atomicOr(a.status, 1);
}

static int sm_count()
{
    static int n = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return n;
}

template <typename T, class F, typename Off, Search HOW>
static cudaError_t dca_launch_off(const F &fld, const DcaArgs &a, cudaStream_t st)
{
    if (a.W <= kPersistMaxW && a.counter) {
        const PLayout L = p_layout(a.W, (int)sizeof(T), p_sph_entries(a));
        cudaError_t e = cudaFuncSetAttribute(dca_persistent_kernel<T, F, Off, HOW>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.total);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dca_persistent_kernel<T, F, Off, HOW>,
                                                          kThreads, L.total);
        if (e != cudaSuccess) return e;
        per_sm = per_sm < 1 ? 1 : per_sm;
        if (a.max_ctas_per_sm > 0 && a.max_ctas_per_sm < per_sm) per_sm = a.max_ctas_per_sm;
        const int64_t items = (a.S + 31) / 32 * ((a.part && a.arrive) ? a.n_chunks : 1);
        int64_t nb = (items + kWarps - 1) / kWarps;
        const int64_t cap = (int64_t)per_sm * sm_count();
        nb = nb < cap ? nb : cap;
        e = cudaMemsetAsync(a.counter, 0, sizeof(int32_t), st);
        if (e != cudaSuccess) return e;
        if (a.best_idx_out && nb > a.best_slots_cap) return cudaErrorInvalidValue;   // one slot per CTA
        dca_persistent_kernel<T, F, Off, HOW><<<(unsigned)nb, kThreads, L.total, st>>>(fld, a);
        return cudaGetLastError();
    }
    using L = Smem<T>;
    static const cudaError_t attr = cudaFuncSetAttribute(
        dca_tiled_kernel<T, F, Off, HOW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::total);
    if (attr != cudaSuccess) return attr;
    const int64_t nb = (a.S + kThreads - 1) / kThreads;
    if (a.best_idx_out && nb > a.best_slots_cap) return cudaErrorInvalidValue;   // one slot per CTA
    dca_tiled_kernel<T, F, Off, HOW><<<(unsigned)nb, kThreads, L::total, st>>>(fld, a);
    return cudaGetLastError();
}

template <typename T, class F, Search HOW>
static cudaError_t dca_launch_how(const F &fld, const DcaArgs &a, cudaStream_t st)
{
    // 32-bit offsets (one register and no carry per address) into a track array below 4 GiB
    return 6 * a.S * (int64_t)a.n_rec * (int64_t)sizeof(T) < ((int64_t)1 << 32)
               ? dca_launch_off<T, F, uint32_t, HOW>(fld, a, st)
               : dca_launch_off<T, F, size_t, HOW>(fld, a, st);
}

template <class F>
constexpr bool is_general = false;
template <typename T>
constexpr bool is_general<FieldUniform<T>> = true;

// FP32 in an axial field takes the short form (group_wires_short) when a level-1 segment is one state:
// runs are then a few states long.  In the tiled kernel too (long and short form): 2^16 seeds x 69 states x
// 1,100 wires 605 and 574 us, 11,475 seeds of an odd lattice x 138 states x 1,100 wires 3,043 and 2,097 us.
// In a general uniform field it takes the long form without the wide scan then (with and without, 2^14 seeds x 69
// states 88 and 82 us, 2^18 804 and 718; a table's refinement takes so long that it makes no difference).
template <typename T, class F>
static cudaError_t dca_launch(const F &fld, const DcaArgs &a, cudaStream_t st)
{
    if (a.exact_all) return dca_launch_how<T, F, kAll>(fld, a, st);
    if constexpr (sizeof(T) == 4 && F::kAxial)
        if (a.G1 == 1) return dca_launch_how<T, F, kShort>(fld, a, st);
    if constexpr (sizeof(T) == 4 && is_general<F>)
        if (a.G1 == 1) return dca_launch_how<T, F, kFew>(fld, a, st);
    return dca_launch_how<T, F, kLong>(fld, a, st);
}

template <typename T>
static cudaError_t dca_dispatch(const comet_field &f, const DcaArgs &a, cudaStream_t st)
{
    switch (field_kind(f)) {
    case FieldKind::Axial:
        return dca_launch<T>(FieldAxial<T>{(T)f.b[2]}, a, st);
    case FieldKind::Uniform:
        return dca_launch<T>(FieldUniform<T>{(T)f.b[0], (T)f.b[1], (T)f.b[2]}, a, st);
    case FieldKind::Table:
    default:
        return dca_launch<T>(make_table<T>(f),
                             a, st);
    }
}

int dca_wire_chunks(int W, int64_t S, int chunk_wires)
{
    if (W <= 0 || W > kPersistMaxW) return 1;
    if (chunk_wires > 0) {
        // a fixed width (the context's setting), at most kDcaBatchSub chunks
        const int n = (W + chunk_wires - 1) / chunk_wires;
        return n < kDcaBatchSub ? n : kDcaBatchSub;
    }
    int nc = (W + COMET_DCA_CHUNK_W - 1) / COMET_DCA_CHUNK_W;
    // few seeds: narrower chunks (at least 4 wires, at most kDcaBatchSub of them), so that the
    // (32-seed group, chunk) work items occupy every SM
    constexpr int64_t kTargetItems = 4096;
    const int64_t groups = (S + 31) / 32;
    if (groups > 0 && groups * nc < kTargetItems) {
        const int64_t want = (kTargetItems + groups - 1) / groups;
        int cap = W / 4;
        cap = cap < kDcaBatchSub ? cap : kDcaBatchSub;
        if (want > nc && cap > nc) nc = (int)(want < cap ? want : cap);
    }
    return nc;
}

void dca_segments(int n_rec, int *G0, int *G1)
{
    if (n_rec <= kN0Max * kN1Max) {
        // one state per level-1 segment: its sphere is then just the spread of the group's tracks
        const int n0 = (n_rec + kN1Max - 1) / kN1Max;
        *G0 = (n_rec + n0 - 1) / n0;
        *G1 = 1;
        return;
    }
    // up to 8 super-segments, each cut into level-1 segments of 3 states (more when a super-segment
    // would have more than kN1Max of them)
    int n0 = (int)lround(cbrt((double)n_rec));
    n0 = n0 < 1 ? 1 : (n0 > kN0Max ? kN0Max : n0);
    const int g0 = (n_rec + n0 - 1) / n0;
    int g1 = 3;
    if ((g0 + g1 - 1) / g1 > kN1Max) g1 = (g0 + kN1Max - 1) / kN1Max;
    *G0 = g0;
    *G1 = g1 > g0 ? g0 : g1;
}

// ------------------------------------------------------------------------------------------------
// Batch of events: persistent CTAs take items -- dca_batch_groups(n_chunks) consecutive 32-seed
// groups of one event -- from ONE counter over all events (items numbered event by event,
// BL.dca_start the prefix), so the load balances across events as it does in the single-event
// kernel.  Inside an item the warps share out its (group, wire chunk) sub-items from a shared
// counter, park the partial sums in the CTA's slice of BL.dca_part, and add them per seed in chunk
// order once the item is done (the single-event kernel's arithmetic).  A CTA restages wires and
// hits only when its next item belongs to another event (a few KB by bulk copy).  Shared memory is
// laid out for the batch's largest W.
// ------------------------------------------------------------------------------------------------

#ifndef COMET_DCA_BATCH_MINB
#define COMET_DCA_BATCH_MINB 4   // the event's arguments come from a table, not the parameter bank: at 6 the
                                 // kernel spilled (three rounds of 16 events 1438 us at 6, 1210 at 5, 1183 at 4)
#endif

template <typename T, class F>
__global__ void __launch_bounds__(kThreads, COMET_DCA_BATCH_MINB) dca_batch_kernel(F f, BatchLaunch BL)
{
    const PLayout L = p_layout(BL.W_max, (int)sizeof(T), 0);   // batches read their bounds in place
    extern __shared__ __align__(128) unsigned char sm[];
    uint64_t *bar = (uint64_t *)sm;
    __shared__ int64_t s_chunk;
    __shared__ int s_sub;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    T *wrow = (T *)(sm + L.wrow);
    int32_t *orow = (int32_t *)(sm + L.orow);
    T *capv = (T *)(sm + L.cap);
    Q4<T> *frm = (Q4<T> *)(sm + L.frame);
    T *dsm = (T *)(sm + L.drift);
    uint8_t *msm = (uint8_t *)(sm + L.mask);
    const int rcap = L.wcap + 32;
    if (tid == 0) mbar_init(bar, 1);
    __syncthreads();

    const int64_t n_chunks = BL.dca_start[BL.B];
    uint32_t parity = 0;
    bool timed_out = false;
    int cur = -1;
    // the current event's arguments and staged tile live in shared memory (they change only on a
    // restage): registers stay free for the group loop
    __shared__ DcaArgs s_a;
    __shared__ Tile<T> s_tl;
    const DcaArgs &a = s_a;
    const Tile<T> &tl = s_tl;
    int nunc = 0;
    for (;;) {
        if (tid == 0) {
            s_chunk = (int64_t)atomicAdd((unsigned long long *)BL.chunk_counter, 1ull);
            s_sub = 0;
        }
        __syncthreads();
        const int64_t chunk = s_chunk;
        if (chunk >= n_chunks) break;
        int e;
        int64_t lc;
        batch_find(BL.dca_start, BL.B, chunk, e, lc);
        if (e != cur) {
            // flush this CTA's unconverged count to the event it leaves
            if (cur >= 0 && a.n_unconv) {
                int t = nunc;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
                if (lane == 0 && t) atomicAdd(a.n_unconv, t);
            }
            nunc = 0;
            // every thread is past its last use of s_a / s_tl (the barrier closing the chunk)
            if (tid == 0) s_a = BL.ev[e].dca;
            __syncthreads();
            cur = e;
            const T *__restrict__ Wg = (const T *)a.wires;
            const T *__restrict__ Dg = (const T *)a.drift;
            const int W = a.W;
            const int H = W > 0 ? a.offs[W] : 0;
            const bool hits_sm = H <= kHitMax;
            // every thread's earlier shared-memory accesses before the bulk copies overwrite them
            fence_proxy_async_smem();
            __syncthreads();
            uint32_t bytes = 0;
            int woff[6] = {0, 0, 0, 0, 0, 0};
            int ooff = 0, doff = 0, moff = 0;
            if (W > 0) {
                bytes = stage_bytes<int32_t>(a.offs, W + 1);
#pragma unroll
                for (int r = 0; r < 6; ++r) bytes += stage_bytes<T>(Wg + (size_t)r * a.ldw, W);
                if (hits_sm && H > 0) bytes += stage_bytes<T>(Dg, H) + stage_bytes<uint8_t>(a.mask, H);
                if (tid == 0 && bytes > 0) mbar_arrive_expect_tx(bar, bytes);
#pragma unroll
                for (int r = 0; r < 6; ++r)
                    woff[r] = stage_issue<T>(wrow + r * rcap, Wg + (size_t)r * a.ldw, W, bar, tid == 0);
                ooff = stage_issue<int32_t>(orow, a.offs, W + 1, bar, tid == 0);
                if (hits_sm && H > 0) {
                    doff = stage_issue<T>(dsm, Dg, H, bar, tid == 0);
                    moff = stage_issue<uint8_t>(msm, a.mask, H, bar, tid == 0);
                }
            }
            const bool to = finish_stage(bar, parity, bytes, a.wait_ns);
            if (to && W > 0) {
#pragma unroll
                for (int r = 0; r < 6; ++r) stage_fallback<T>(wrow + r * rcap, Wg + (size_t)r * a.ldw, W);
                stage_fallback<int32_t>(orow, a.offs, W + 1);
                if (hits_sm && H > 0) {
                    stage_fallback<T>(dsm, Dg, H);
                    stage_fallback<uint8_t>(msm, a.mask, H);
                }
            }
            if (to) {
                // a timed-out copy may still land: wait for it (bounded) before anything reuses
                // the buffers, and report it
                timed_out = true;
                if (tid == 0 && a.status) atomicOr(a.status, 1);
                mbar_wait(bar, parity ^ 1u, kWaitNs);
            }
            if (tid == 0) {
                s_tl.ax = wrow + 0 * rcap + woff[0];
                s_tl.ay = wrow + 1 * rcap + woff[1];
                s_tl.az = wrow + 2 * rcap + woff[2];
                s_tl.ux = wrow + 3 * rcap + woff[3];
                s_tl.uy = wrow + 4 * rcap + woff[4];
                s_tl.uz = wrow + 5 * rcap + woff[5];
                s_tl.rec = frm;
                s_tl.ff = (const float4 *)wrow;
                s_tl.cap = capv;
                s_tl.offs = orow + ooff;
                s_tl.dsm = hits_sm ? dsm + doff : Dg;
                s_tl.msm = hits_sm ? msm + moff : a.mask;
                s_tl.w0 = 0;
                s_tl.wn = W;
            }
            __syncthreads();
            for (int i = tid; i < W; i += kThreads) tile_wire_setup<T>(tl, i, in_prec<T>(a.lambda, a.lambda_f), capv, frm);
            __syncthreads();
            if constexpr (sizeof(T) == 8) {
                tile_float_frames<T>(frm, W, (float4 *)wrow);
                __syncthreads();
            }
        }
        // the item's (group, wire chunk) sub-items, taken by the warps as they come free
        const int nc = a.n_chunks;
        const int64_t n_groups = (a.S + 31) / 32;
        const int gpi = a.batch_groups > 0 ? a.batch_groups : dca_batch_groups(nc);
        const int64_t g0 = lc * gpi;
        const int ng = (int)min((int64_t)gpi, n_groups - g0);
        const int n_sub = ng * nc;
        T *ph = (T *)((unsigned char *)BL.dca_part +
                      (size_t)blockIdx.x * kDcaBatchSub * 32 * (2 * sizeof(T) + 4));
        T *pl = ph + kDcaBatchSub * 32;
        int32_t *pn = (int32_t *)(pl + kDcaBatchSub * 32);
        for (;;) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&s_sub, 1);
            k = __shfl_sync(0xffffffffu, k, 0);
            if (k >= n_sub) break;
            const int64_t g = g0 + k / nc;
            const Group<T> gr = load_group<T>(a, g, lane);
            const float4 *s0 = (const float4 *)a.bounds + g * kBoundsPerGroup;   // read in place
            Acc<T> acc;
            int nin = 0;
            const int2 r = chunk_range(a.W, nc, k % nc);
            // one form for every recording (an event's decides it, the launch is for all): runs of several states
            // and FP64 are scanned where a launch of their own walks them, with the same bits
            group_wires<T, F, size_t, kShort>(f, a, gr, tl, s0, s0 + kN0Max, lane, acc, nin, nunc, r.x, r.y);
            ph[k * 32 + lane] = acc.hi;
            pl[k * 32 + lane] = acc.lo;
            pn[k * 32 + lane] = nin;
        }
        __syncthreads();   // every sub-item of the item done (and its partial sums visible)
        for (int gi = warp; gi < ng; gi += kWarps) {
            const int64_t s = (g0 + gi) * 32 + lane;
            if (s < a.S) {
                Acc<T> tot;
                int nt = 0;
                for (int c = 0; c < nc; ++c) {
                    const int k = (gi * nc + c) * 32 + lane;
                    tot.add_pair(ph[k], pl[k]);
                    nt += pn[k];
                }
                ((T *)a.rss)[s] = tot.value();
                a.n_in[s] = nt;
            }
        }
        __syncthreads();   // every warp done with this item before a restage or the next s_chunk
    }
    if (cur >= 0 && a.n_unconv) {
        int t = nunc;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
        if (lane == 0 && t) atomicAdd(a.n_unconv, t);
    }
    (void)timed_out;
}

template <typename T, class F>
static cudaError_t dca_batch_launch(const F &fld, const BatchLaunch &BL, cudaStream_t st)
{
    // (the shared-memory attribute for W_max was set when the batch was prepared: nothing here but
    // stream work, so that the launch can be captured)
    const PLayout L = p_layout(BL.W_max, (int)sizeof(T), 0);
    cudaError_t e = cudaMemsetAsync(BL.chunk_counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (BL.dca_ctas == 0) return cudaSuccess;
    dca_batch_kernel<T, F><<<BL.dca_ctas, kThreads, L.total, st>>>(fld, BL);
    return cudaGetLastError();
}

template <typename T, class F>
static int dca_ctas_per_sm_t(int W)
{
    const PLayout L = p_layout(W, (int)sizeof(T), 0);
    if (cudaFuncSetAttribute(dca_batch_kernel<T, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)L.total) != cudaSuccess)
        return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dca_batch_kernel<T, F>, kThreads,
                                                      L.total) != cudaSuccess)
        return 0;
    return per_sm;
}

template <typename T>
static int dca_ctas_per_sm_field(const comet_field &f, int W)
{
    switch (field_kind(f)) {
    case FieldKind::Axial: return dca_ctas_per_sm_t<T, FieldAxial<T>>(W);
    case FieldKind::Uniform: return dca_ctas_per_sm_t<T, FieldUniform<T>>(W);
    default: return dca_ctas_per_sm_t<T, FieldTable<T>>(W);
    }
}

int dca_persistent_ctas_per_sm(comet_dtype dt, const comet_field &f, int W)
{
    return dt == COMET_F32 ? dca_ctas_per_sm_field<float>(f, W) : dca_ctas_per_sm_field<double>(f, W);
}

int device_sm_count() { return sm_count(); }

template <typename T>
static cudaError_t dca_batch_dispatch(const comet_field &f, const BatchLaunch &BL, cudaStream_t st)
{
    switch (field_kind(f)) {
    case FieldKind::Axial:
        return dca_batch_launch<T>(FieldAxial<T>{(T)f.b[2]}, BL, st);
    case FieldKind::Uniform:
        return dca_batch_launch<T>(FieldUniform<T>{(T)f.b[0], (T)f.b[1], (T)f.b[2]}, BL, st);
    case FieldKind::Table:
    default:
        return dca_batch_launch<T>(make_table<T>(f),
                                   BL, st);
    }
}

cudaError_t launch_dca_batch(comet_dtype dt, const comet_field &f, const BatchLaunch &BL, cudaStream_t st)
{
    return dt == COMET_F32 ? dca_batch_dispatch<float>(f, BL, st) : dca_batch_dispatch<double>(f, BL, st);
}

cudaError_t launch_dca(comet_dtype dt, const comet_field &f, const DcaArgs &a, cudaStream_t st)
{
    return dt == COMET_F32 ? dca_dispatch<float>(f, a, st) : dca_dispatch<double>(f, a, st);
}

} // namespace comet
