// Probe-ray kernels of the update (Sec. 2.3 and Sec. 6.3):
//   k_classify, k_classify_split  distance-only trace of UNINIT probes -> OFF /
//                     NEWLY_VIGILANT / SLEEPING; k_optimize moves them first
//   k_trace_primary, k_trace_shadow, k_shade  the update's three passes
//   k_trace_shade     closest hit + shading of every ray of every active probe
//                     (the allocation-free update)
// plus two utility kernels over arbitrary rays (raw closest hit, camera G-buffer).
//
// Work layout: rays of one probe are consecutive work items, so a warp
// traces 32 rays of the same probe (same origin, a compact cone of directions
// by the ray order).  Kernels are persistent: the grid is sized to the machine
// and warps take work up to the device-side count, so the host never waits for
// the active-probe count.
#include <algorithm>

#include "traverse.cuh"

namespace ddgi {

__global__ void __launch_bounds__(256) k_classify(DevScene s, VolView v, const float4* __restrict__ dirs,
                                                  int R, const int32_t* __restrict__ perm,
                                                  const int32_t* __restrict__ list,
                                                  const int32_t* __restrict__ count) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int n = *count;
    int2 stack[kStackSize4];
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    for (int q = warp; q < n; q += nwarps) {
        const int p = list[q];
        float3 o = probe_pos_phys(v, p);
        int bf = 0;
        float dmin = INFINITY;
        // the warp's lanes take 32 rays at a time through the warp-cooperative
        // 4-wide walk (lanes past R take part without a ray)
        for (int j0 = 0; j0 < R; j0 += 32) {
            const int j = j0 + lane;
            const bool valid = j < R;
            const int i = valid ? (perm ? __ldg(perm + j) : j) : 0;
            const float4 d4 = __ldg(dirs + i);
            const float3 d = f3(d4.x, d4.y, d4.z);
            const RayPre r = ray_pre_packed(o, d, __ldg(dirs + R + 2 * i), __ldg(dirs + R + 2 * i + 1));
            ww_start(s, w, valid);
            do {
                ww4_round<false>(s, r, w);
            } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
            const Hit& h = w.h;
            if (valid && h.orig >= 0) {
                const float4* T = s.tris + 3 * (int64_t)h.k;
                float4 p0 = __ldg(T), p1 = __ldg(T + 1), p2 = __ldg(T + 2);
                float3 ng = cross(f3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z),
                                  f3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z));
                if (dot(d, ng) > 0.0f) bf++;
                else dmin = fminf(dmin, h.t);
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            bf += __shfl_xor_sync(0xffffffffu, bf, off);
            dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, off));
        }
        if (lane == 0) {
            uint8_t st;
            if (4 * bf > R) st = DDGI_STATE_OFF;
            else if (dmin < v.min_spacing) st = DDGI_STATE_NEWLY_VIGILANT;
            else st = DDGI_STATE_SLEEPING;
            v.states[p] = st;
        }
    }
}

// Persistent passes: a warp walks its lanes' rays in while-while rounds and,
// once every lane has finished, takes the next 32 work items (Aila and Laine
// 2009, persistent threads; refilling at 4, 8 or 16 idle lanes measured
// slower on the city workload, in lost ray coherence).  The first batch is
// the warp's own index and only later ones come from the global counter,
// which starts after them: with few rays, thousands of warps would
// otherwise queue on one word to learn that nothing is left.  Work items are
// below 2^31 (probes x rays is), a batch past the end below 2^32.
__device__ __forceinline__ unsigned first_batch() { return (blockIdx.x * blockDim.x + threadIdx.x) & ~31u; }
__device__ __forceinline__ unsigned next_batch(uint32_t* next) {
    unsigned base = 0;
    if ((threadIdx.x & 31) == 0) base = gridDim.x * blockDim.x + atomicAdd(next, 32u);
    return __shfl_sync(0xffffffffu, base, 0);
}

// CTAs per SM that classification and the optimizer are built for (64
// registers a thread: their reductions spill at 48).
constexpr int kClassCtas = 4;

// Classification in 32-ray batches: one work item per (list entry, batch),
// so the R rays of the few probes a frame classifies (the planes a tracking
// window scrolls in) spread over all warps instead of R / 32 sequential
// batches in one warp each.  A batch adds its backface count and maxes its
// nearest front-face distance (as 0x7f800000 - bits, so a zeroed word
// stands for +inf) into the entry's scratch, then counts itself done; the
// warp that completes an entry's last batch sets the state as k_classify
// does and zeroes the scratch for the next classification.  Counts and
// minima do not depend on the order the batches run in, so the states are
// k_classify's.  scratch: one zeroed int4 per list entry.
template <bool MULTI>
__global__ void __launch_bounds__(256, kClassCtas) k_classify_split(DevScene s, VolSet vs,
                                                                    const float4* __restrict__ dirs, int R,
                                                                    const int32_t* __restrict__ perm,
                                                                    const int32_t* __restrict__ list,
                                                                    const int32_t* __restrict__ count, int4* scratch,
                                                                    uint32_t* next) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const unsigned nb = (unsigned)(R + 31) / 32;
    const unsigned total = (unsigned)(*count) * nb * 32u;   // below 2^32: probes x R is below 2^31, probes 2^26
    int2 stack[kStackSize4];
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    for (unsigned at = first_batch(); at < total; at = next_batch(next)) {
        const unsigned it = at >> 5;
        const int q = (int)(it / nb), b = (int)(it - (unsigned)q * nb);
        const int e = list[q];
        const VolView& v = vol_of<MULTI>(vs, e >> kEntryShift);
        const int p = entry_probe<MULTI>(e);
        const float3 o = probe_pos_phys(v, p);
        const int j = 32 * b + lane;
        const bool valid = j < R;
        const int i = valid ? (perm ? __ldg(perm + j) : j) : 0;
        const float4 d4 = __ldg(dirs + i);
        const float3 d = f3(d4.x, d4.y, d4.z);
        const RayPre r = ray_pre_packed(o, d, __ldg(dirs + R + 2 * i), __ldg(dirs + R + 2 * i + 1));
        ww_start(s, w, valid);
        do {
            ww4_round<false>(s, r, w);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        const Hit& h = w.h;
        bool back = false;
        float dmin = INFINITY;
        if (valid && h.orig >= 0) {
            const float4* T = s.tris + 3 * (int64_t)h.k;
            float4 p0 = __ldg(T), p1 = __ldg(T + 1), p2 = __ldg(T + 2);
            float3 ng = cross(f3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z), f3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z));
            if (dot(d, ng) > 0.0f) back = true;
            else dmin = h.t;
        }
        const int bf = __popc(__ballot_sync(0xffffffffu, back));
        for (int off = 16; off > 0; off >>= 1) dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, off));
        if (lane == 0) {
            int4* sc = scratch + q;
            if (bf) atomicAdd(&sc->x, bf);
            atomicMax(&sc->y, 0x7f800000 - __float_as_int(dmin));
            __threadfence();   // this batch's sums before its done count
            if (atomicAdd(&sc->z, 1) == (int)nb - 1) {
                __threadfence();
                const int bft = atomicAdd(&sc->x, 0);
                const float dm = __int_as_float(0x7f800000 - atomicAdd(&sc->y, 0));
                uint8_t st;
                if (4 * bft > R) st = DDGI_STATE_OFF;
                else if (dm < v.min_spacing) st = DDGI_STATE_NEWLY_VIGILANT;
                else st = DDGI_STATE_SLEEPING;
                v.states[p] = st;
                *sc = make_int4(0, 0, 0, 0);   // no other batch of this entry is left
            }
        }
    }
}

// Fused trace + shade, one thread per probe ray (the allocation-free
// update's path: it needs no shadow or hit lists); rays and shadow rays go
// through the warp-cooperative 4-wide walk.  Bound by the latency of the walk:
// a volume of this path has some ten warps of rays to an SM.  So a warp takes a
// compact cone of directions (perm) instead of 32 steps of the spiral over the
// sphere, the walk its 64-register form and the shading the specialised query;
// with that, and with every kernel of the update launched while the one before
// it ends, 16 x 8 x 16 probes x 128 rays of a city take 62 us (78 before).
template <int FORM>
__global__ void __launch_bounds__(128, 6) k_trace_shade(DevScene s, VolView v, Lights L,
                                                        const float4* __restrict__ dirs, int R, FastDiv dR,
                                                        const int32_t* __restrict__ perm,
                                                        const int32_t* __restrict__ active,
                                                        const int32_t* __restrict__ count,
                                                        float4* __restrict__ records) {
    pdl_wait();
    pdl_trigger();
    const int total = (*count) * R;   // at most 2^20
    const int stride = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const float3 tol = f3(-L.sun_dir.x, -L.sun_dir.y, -L.sun_dir.z);
    const RayPre r_sun = ray_pre(f3(0.0f, 0.0f, 0.0f), tol);
    int2 stack[kStackSize4];
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    // warp-uniform loop: each warp takes 32 consecutive rays through the
    // warp-cooperative 4-wide walk, then their shadow rays the same way
    for (int base = blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
        const bool valid = base + lane < total;
        const int id = valid ? base + lane : base;
        const int slot = (int)fast_div((uint32_t)id, dR);
        const int i = __ldg(perm + (id - slot * R));   // consecutive items take a compact cone of directions
        const int p = __ldg(active + slot);
        float3 o = probe_pos_phys(v, p);
        float4 d4 = __ldg(dirs + i);
        float3 d = f3(d4.x, d4.y, d4.z);
        const RayPre r = ray_pre_packed(o, d, __ldg(dirs + R + 2 * i), __ldg(dirs + R + 2 * i + 1));
        ww_start(s, w, valid);
        do {
            ww4_round<false, false, true>(s, r, w);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        const Hit h = w.h;
        // the shadow ray of a sunlit front hit
        float3 n = f3(0.0f, 0.0f, 1.0f), x = o;
        float cosl = 0.0f;
        bool front = false;
        float3 ng = f3(0.0f, 0.0f, 1.0f);
        if (valid && h.orig >= 0) {
            const float4* T = s.tris + 3 * (int64_t)h.k;
            float4 p0 = __ldg(T), p1 = __ldg(T + 1), p2 = __ldg(T + 2);
            ng = cross(f3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z), f3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z));
            front = !(dot(d, ng) > 0.0f);
            n = (1.0f / length(ng)) * ng;
            x = o + h.t * d;
            cosl = dot(n, tol);
        }
        const bool shadow = front && L.sun_on && cosl > 0.0f;
        RayPre sr = r_sun;
        if (shadow) ray_set_origin(sr, x + (1e-4f * (1.0f + length(x))) * n);
        ww_start(s, w, shadow);
        do {
            ww4_round<true, false, true>(s, sr, w);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        const bool lit = shadow && w.h.orig < 0;
        if (!valid) continue;
        float4 rec;
        if (h.orig < 0) {
            float c = dot(d, L.sky_up);
            rec = make_float4(L.sky_a.x + L.sky_b.x * c, L.sky_a.y + L.sky_b.y * c,
                              L.sky_a.z + L.sky_b.z * c, v.t_max);
        } else if (!front) {
            // back face: radiance 0, depth shortened by 80% (Sec. 4.1)
            rec = make_float4(0.0f, 0.0f, 0.0f, fminf(0.2f * h.t, v.t_max));
        } else {
            int2 at = __ldg(s.attr + h.orig);
            float4 rho = __ldg(s.albedo + at.x);
            float3 Le = f3(0.0f, 0.0f, 0.0f);
            if (at.y >= 0) {
                float4 e = __ldg(s.emit + at.y);
                Le = f3(e.x, e.y, e.z);
            }
            float3 direct = f3(0.0f, 0.0f, 0.0f);
            if (lit) {
                float k = cosl * 0.318309886183790672f;   // 1/pi
                direct = f3(L.sun_irr.x * k, L.sun_irr.y * k, L.sun_irr.z * k);
            }
            float3 M = query_M<FORM>(v, x, n, f3(-d.x, -d.y, -d.z));
            rec = make_float4(Le.x + rho.x * (direct.x + M.x), Le.y + rho.y * (direct.y + M.y),
                              Le.z + rho.z * (direct.z + M.z), fminf(h.t, v.t_max));
        }
        records[slot * R + i] = rec;
    }
}

// ---------------------------------------------------------------------------
// Wavefront form of trace + shade: three coherent passes over the same rays.
//   k_trace_primary  closest hit of every ray over the 4-wide hierarchy;
//                    writes the final record of misses (sky) and back faces,
//                    stores (t, BVH triangle index, 0, 0) for front hits and
//                    appends them to the hit list, and those facing the sun
//                    to the shadow-ray list
//   k_trace_shadow   any-hit shadow rays over that list; sets the visibility
//   k_shade          shading and the previous-frame query at each front hit;
//                    writes the final (r, g, b, d) record over the hit record
// Each pass keeps its lanes on one kind of work, where the fused kernel ran
// traversal, shadow rays and queries divergently in the same warp.  The
// arithmetic of every value is the fused kernel's, in the same order.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void hit_frame(const DevScene& s, int k, float3& ng) {
    const float4* T = s.tris + 3 * (int64_t)k;
    float4 p0 = __ldg(T), p1 = __ldg(T + 1), p2 = __ldg(T + 2);
    ng = cross(f3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z), f3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z));
}

// CTAs per SM that the passes are built for: four with the 64-register walk
// for a single volume, five (48 registers) for a cascade (ww4_round).
constexpr int trace_ctas(bool multi) { return multi ? 5 : 4; }

// COUNT: measurement build that adds its 4-wide node visits and triangle
// tests to stats[1], stats[2] (otherwise identical).
template <bool MULTI, bool COUNT = false>
__global__ void __launch_bounds__(256, trace_ctas(MULTI)) k_trace_primary(
    DevScene s, VolSet vs, Lights L, const float4* __restrict__ dirs, int R, FastDiv dR,
    const int32_t* __restrict__ perm, const int32_t* __restrict__ active, const int32_t* __restrict__ count,
    float4* __restrict__ hits, int32_t* __restrict__ shadow_list, int32_t* __restrict__ hit_list, int32_t* shadow_count,
    uint32_t* next, unsigned long long* stats) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const unsigned total = (unsigned)(*count) * (unsigned)R;
    TraceCount tc;
    int2 stack[kStackSize4];
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    for (unsigned b = first_batch(); b < total; b = next_batch(next)) {
        // work item -> (probe slot, ray): consecutive items take a compact
        // cone of directions; the record keeps its canonical ray index
        int rec;
        RayPre r;
        {
            const int item = (int)min(b + lane, total - 1);
            const int slot = (int)fast_div((uint32_t)item, dR);
            const int j = item - slot * R;
            const int i = perm ? __ldg(perm + j) : j;
            rec = slot * R + i;
            const int entry = __ldg(active + slot);
            const float4 d4 = __ldg(dirs + i);
            r = ray_pre_packed(probe_pos_phys(vol_of<MULTI>(vs, entry >> kEntryShift), entry_probe<MULTI>(entry)),
                               f3(d4.x, d4.y, d4.z), __ldg(dirs + R + 2 * i), __ldg(dirs + R + 2 * i + 1));
        }
        const bool valid = b + lane < total;
        ww_start(s, w, valid);
        do {
            ww4_round<false, COUNT, !MULTI>(s, r, w, &tc);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        bool need = false, front = false;
        if (valid) {
            // misses and back faces get their final record here; front hits
            // keep (t, triangle) for the shading pass.  The probe and the
            // direction are read again (rec made opaque) rather than held
            // across the walk, whose registers they would push out.
            asm volatile("" : "+r"(rec));
            const int slot = (int)fast_div((uint32_t)rec, dR);
            const float4 d4 = __ldg(dirs + (rec - slot * R));
            const float3 d = f3(d4.x, d4.y, d4.z);
            const Hit& h = w.h;
            const float t_max = MULTI ? vol_of<MULTI>(vs, __ldg(active + slot) >> kEntryShift).t_max : vs.single.t_max;
            float4 out;
            if (h.orig < 0) {
                float c = dot(d, L.sky_up);
                out = make_float4(L.sky_a.x + L.sky_b.x * c, L.sky_a.y + L.sky_b.y * c, L.sky_a.z + L.sky_b.z * c,
                                  t_max);
            } else {
                float3 ng;
                hit_frame(s, h.k, ng);
                if (dot(d, ng) > 0.0f) {
                    out = make_float4(0.0f, 0.0f, 0.0f, fminf(0.2f * h.t, t_max));
                } else {
                    front = true;
                    if (L.sun_on) {
                        float3 n = (1.0f / length(ng)) * ng;
                        need = dot(n, f3(-L.sun_dir.x, -L.sun_dir.y, -L.sun_dir.z)) > 0.0f;
                    }
                    out = make_float4(h.t, __int_as_float(h.k), 0.0f, 0.0f);
                }
            }
            hits[rec] = out;
        }
        // both lists' places with one 64-bit atomic (shadow rays in the low word)
        const unsigned mask_s = __ballot_sync(0xffffffffu, need), mask_f = __ballot_sync(0xffffffffu, front);
        if (mask_f) {
            unsigned long long off = 0;
            if (lane == 0)
                off = atomicAdd(reinterpret_cast<unsigned long long*>(shadow_count),
                                ((unsigned long long)__popc(mask_f) << 32) | (unsigned)__popc(mask_s));
            off = __shfl_sync(0xffffffffu, off, 0);
            const unsigned below = (1u << lane) - 1u;
            if (need) shadow_list[(unsigned)off + __popc(mask_s & below)] = rec;
            if (front) hit_list[(unsigned)(off >> 32) + __popc(mask_f & below)] = rec;
        }
    }
    if (COUNT) {
        atomicAdd(stats + 1, (unsigned long long)tc.nodes);
        atomicAdd(stats + 2, (unsigned long long)tc.tris);
    }
}

// COUNT: adds 4-wide node visits and triangle tests to stats[4], stats[5].
template <bool MULTI, bool COUNT = false>
__global__ void __launch_bounds__(256, trace_ctas(MULTI)) k_trace_shadow(
    DevScene s, VolSet vs, Lights L, const float4* __restrict__ dirs, int R, FastDiv dR,
    const int32_t* __restrict__ active, float4* __restrict__ hits, const int32_t* __restrict__ shadow_list,
    const int32_t* __restrict__ shadow_count, uint32_t* next, unsigned long long* stats) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const unsigned total = (unsigned)*shadow_count;
    TraceCount tc;
    RayPre r = ray_pre(f3(0.0f, 0.0f, 0.0f), f3(-L.sun_dir.x, -L.sun_dir.y, -L.sun_dir.z));   // every shadow ray runs towards the sun
    int stack[kStackSize4];   // any-hit walk: plain references (no hit distance to prune by)
    WwLane<kStackSize4> w;
    w.stack = stack;
    for (unsigned b = first_batch(); b < total; b = next_batch(next)) {
        const bool valid = b + lane < total;
        const int rec = __ldg(shadow_list + (valid ? b + lane : b));
        const int slot = (int)fast_div((uint32_t)rec, dR);
        const int i = rec - slot * R;
        const int e = __ldg(active + slot);
        const float3 o = probe_pos_phys(vol_of<MULTI>(vs, e >> kEntryShift), entry_probe<MULTI>(e));
        const float4 d4 = __ldg(dirs + i);
        const float4 hr = hits[rec];
        float3 ng;
        hit_frame(s, __float_as_int(hr.y), ng);
        const float3 nn = (1.0f / length(ng)) * ng;
        const float3 x = o + hr.x * f3(d4.x, d4.y, d4.z);
        const float off = 1e-4f * (1.0f + length(x));
        ray_set_origin(r, x + off * nn);
        ww_start(s, w, valid);
        do {
            ww4_round<true, COUNT, !MULTI>(s, r, w, &tc);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        if (valid && w.h.orig < 0) reinterpret_cast<float*>(hits)[4 * (int64_t)rec + 2] = 1.0f;
    }
    if (COUNT) {
        atomicAdd(stats + 4, (unsigned long long)tc.nodes);
        atomicAdd(stats + 5, (unsigned long long)tc.tris);
    }
}

// Shading of the front hits (Sec. 2.3 ray radiance, multi-bounce through the
// previous frame's probes), one thread per entry of the compacted hit list.
template <bool MULTI, int FORM>
__global__ void __launch_bounds__(256, 4) k_shade(DevScene s, VolSet vs, Lights L, const float4* __restrict__ dirs,
                                               int R, FastDiv dR, const int32_t* __restrict__ active,
                                               const int32_t* __restrict__ hit_list,
                                               const int32_t* __restrict__ hit_count, float4* records) {
    pdl_wait();
    pdl_trigger();
    const int n_hits = *hit_count;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n_hits; q += gridDim.x * blockDim.x) {
        const int idx = __ldg(hit_list + q);
        const int slot = (int)fast_div((uint32_t)idx, dR);
        const int i = idx - slot * R;
        float4 d4 = __ldg(dirs + i);
        float3 d = f3(d4.x, d4.y, d4.z);
        float4 hr = records[idx];
        int k = __float_as_int(hr.y);
        const int e = __ldg(active + slot);
        const VolView& v = vol_of<MULTI>(vs, e >> kEntryShift);
        float3 ng;
        hit_frame(s, k, ng);
        float t = hr.x;
        float3 o = probe_pos_phys(v, entry_probe<MULTI>(e));
        float3 n = (1.0f / length(ng)) * ng;
        float3 x = o + t * d;
        // the sun's cosine term (zero when the shadow ray was blocked) and the
        // triangle's material index now; the previous frame's probes at the
        // hit (the volume itself, or the whole cascade) next, with little
        // else held across that query; the material terms after it
        const float3 tol = f3(-L.sun_dir.x, -L.sun_dir.y, -L.sun_dir.z);
        const float kk = hr.z != 0.0f ? dot(n, tol) * 0.318309886183790672f : 0.0f;   // 1/pi
        const int orig = __float_as_int(__ldg(&s.tris[3 * (int64_t)k].w));
        float3 M = MULTI ? cascade_M<FORM>(vs.table, vs.n, x, n, f3(-d.x, -d.y, -d.z))
                         : query_M<FORM>(v, x, n, f3(-d.x, -d.y, -d.z));
        int2 at = __ldg(s.attr + orig);
        float4 rho = __ldg(s.albedo + at.x);
        float3 Le = f3(0.0f, 0.0f, 0.0f);
        if (at.y >= 0) {
            float4 em = __ldg(s.emit + at.y);
            Le = f3(em.x, em.y, em.z);
        }
        const float3 direct = f3(L.sun_irr.x * kk, L.sun_irr.y * kk, L.sun_irr.z * kk);
        records[idx] = make_float4(Le.x + rho.x * (direct.x + M.x), Le.y + rho.y * (direct.y + M.y),
                                   Le.z + rho.z * (direct.z + M.z), fminf(t, v.t_max));
    }
}

// Closest hit of a warp's 32 rays over the 4-wide hierarchy (all lanes call;
// valid: the lane has a ray).
template <bool WIDE>
__device__ __forceinline__ Hit closest_hit_warp(const DevScene& s, const RayPre& r, int2* stack, bool valid) {
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    ww_start(s, w, valid);
    do {
        ww4_round<false, false, WIDE>(s, r, w);
    } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
    return w.h;
}

// Closest hits of arbitrary rays, a warp for 32 consecutive ones.  Rays that
// share nothing gain as well against one ray a thread over the binary hierarchy:
// 1 M of them with random origins and directions over 196,610 city triangles
// 471 -> 291 us, bounced from what a camera sees 312 -> 151 us, 1000 of them
// 53 -> 23 us.
__global__ void __launch_bounds__(256, 4) k_trace_rays(DevScene s, const float* __restrict__ orig,
                                                                const float* __restrict__ dir, int64_t n,
                                                                float* __restrict__ t_out,
                                                                int32_t* __restrict__ tri_out,
                                                                int32_t* __restrict__ bf_out) {
    int2 stack[kStackSize4];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < n; q0 += stride) {
        const int64_t q = min(q0 + (threadIdx.x & 31), n - 1);
        const bool valid = q0 + (threadIdx.x & 31) < n;
        const float3 d = f3(dir[3 * q], dir[3 * q + 1], dir[3 * q + 2]);
        const Hit h = closest_hit_warp<true>(s, ray_pre(f3(orig[3 * q], orig[3 * q + 1], orig[3 * q + 2]), d), stack, valid);
        if (!valid) continue;
        t_out[q] = h.t;
        tri_out[q] = h.orig;
        if (bf_out) {
            int b = 0;
            if (h.orig >= 0) {
                float3 ng;
                hit_frame(s, h.k, ng);
                b = dot(d, ng) > 0.0f;
            }
            bf_out[q] = b;
        }
    }
}

// Camera G-buffer, a warp for a tile of 8 x 4 pixels, whose rays stay together
// further down the hierarchy than a row of 32.  Bound by the walk's
// instruction issue, as the probe rays are (81 % of the cycles, 31.7 of 32 lanes):
// 1920 x 1080 over 196,610 city triangles take 139 us, 199 us with one ray a
// thread over the binary hierarchy.
__global__ void __launch_bounds__(256, 4) k_gbuffer(DevScene s, float3 cpos, float3 fwd, float3 right,
                                                             float3 up, float tan_half, float aspect, int w, int h,
                                                             float* __restrict__ out_pos,
                                                             float* __restrict__ out_nrm) {
    int2 stack[kStackSize4];
    const int lane = threadIdx.x & 31;
    const int tx = (w + 7) / 8;
    const int64_t tiles = (int64_t)tx * ((h + 3) / 4), stride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < tiles; t += stride) {
        const int ty = (int)(t / tx), x = 8 * (int)(t - (int64_t)ty * tx) + (lane & 7), y = 4 * ty + (lane >> 3);
        const bool valid = x < w && y < h;
        float sx = ((x + 0.5f) / w * 2.0f - 1.0f) * tan_half * aspect;
        float sy = (1.0f - (y + 0.5f) / h * 2.0f) * tan_half;
        float3 d = fwd + sx * right + sy * up;
        d = (1.0f / length(d)) * d;
        const Hit hh = closest_hit_warp<true>(s, ray_pre(cpos, d), stack, valid);
        if (!valid) continue;
        float3 p = f3(0.0f, 0.0f, 0.0f), nn = f3(0.0f, 0.0f, 0.0f);
        if (hh.orig >= 0) {
            float3 ng;
            hit_frame(s, hh.k, ng);
            nn = (1.0f / length(ng)) * ng;
            p = cpos + hh.t * d;
        }
        const int64_t q = (int64_t)y * w + x;
        out_pos[3 * q] = p.x; out_pos[3 * q + 1] = p.y; out_pos[3 * q + 2] = p.z;
        out_nrm[3 * q] = nn.x; out_nrm[3 * q + 1] = nn.y; out_nrm[3 * q + 2] = nn.z;
    }
}

// One iteration of the probe position optimizer (Sec. 5 and its listing):
// the iteration's rays from the probe's current position reduced, as
// (t bits << 32 | ray) keys, to the closest backface, the closest front face
// and the farthest front face (ties: smaller ray index for closest, larger
// for farthest); then the offset moves:
//   more than 25% backfaces: along t * w of the closest backface, by the
//     largest scale keeping every component within +-limit (less 1 mm),
//     only when that scale exceeds 1 (the move goes through the backface);
//   otherwise, unless the farthest front face lies within 60 degrees of the
//     closest: min(0.2, t) along the farthest front face, clamped to +-limit.
// As in k_classify_split, a work item is a batch of 32 rays in the order
// `perm` (a compact cone), a batch joins the entry's scratch (zeroed; the
// closest keys as maxima of their complements) and counts itself done, and
// the warp that completes an entry moves the probe and zeroes the scratch.
// Counts, minima and maxima do not depend on the order of the batches.  With
// a warp to a probe, its batches one after another over all directions, an
// iteration of 6912 probes x 128 rays took 106-138 us against 91-122 us here
// (and the classification's trace 123 us against 108 us with batches from
// a counter on one resident wave).
__global__ void __launch_bounds__(256, kClassCtas) k_optimize(DevScene s, VolView v, const float4* __restrict__ dirs,
                                                              int R, const int32_t* __restrict__ perm,
                                                              const int32_t* __restrict__ list,
                                                              const int32_t* __restrict__ count,
                                                              OptimizeScratch* scratch, uint32_t* next) {
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const unsigned nb = (unsigned)(R + 31) / 32;
    const unsigned total = (unsigned)(*count) * nb * 32u;   // below 2^32, as in k_classify_split
    int2 stack[kStackSize4];
    for (unsigned at = first_batch(); at < total; at = next_batch(next)) {
        const unsigned it = at >> 5;
        const int q = (int)(it / nb), j = 32 * (int)(it - (unsigned)q * nb) + lane;
        const bool valid = j < R;
        const int i = valid ? __ldg(perm + j) : 0;
        const float4 d4 = __ldg(dirs + i);
        const float3 d = f3(d4.x, d4.y, d4.z);
        // coherent loads: the offsets are written by other launches' warps only
        const Hit h = closest_hit_warp<false>(s, ray_pre_packed(probe_pos_phys(v, list[q]), d, __ldg(dirs + R + 2 * i),
                                                         __ldg(dirs + R + 2 * i + 1)), stack, valid);
        bool back = false;
        unsigned long long cb = ~0ull, cf = ~0ull, ff = 0ull;
        if (valid && h.orig >= 0) {
            float3 ng;
            hit_frame(s, h.k, ng);
            const unsigned long long key = ((unsigned long long)__float_as_uint(h.t) << 32) | (unsigned)i;
            back = dot(d, ng) > 0.0f;
            if (back) cb = key;
            else cf = ff = key;
        }
        const int bf = __popc(__ballot_sync(0xffffffffu, back));
        for (int off = 16; off > 0; off >>= 1) {
            cb = min(cb, __shfl_xor_sync(0xffffffffu, cb, off));
            cf = min(cf, __shfl_xor_sync(0xffffffffu, cf, off));
            ff = max(ff, __shfl_xor_sync(0xffffffffu, ff, off));
        }
        if (lane != 0) continue;
        OptimizeScratch* sc = scratch + q;
        if (bf) atomicAdd(&sc->back, bf);
        if (cb != ~0ull) atomicMax(&sc->near_back, ~cb);
        if (cf != ~0ull) atomicMax(&sc->near_front, ~cf);
        if (ff != 0ull) atomicMax(&sc->far_front, ff);
        __threadfence();   // this batch's part before its done count
        if (atomicAdd(&sc->done, 1) != (int)nb - 1) continue;
        __threadfence();
        const int bft = atomicAdd(&sc->back, 0);
        cb = ~atomicMax(&sc->near_back, 0ull);
        cf = ~atomicMax(&sc->near_front, 0ull);
        ff = atomicMax(&sc->far_front, 0ull);
        *sc = OptimizeScratch{};   // no other batch of this entry is left
        const int p = list[q];
        const float4 c4 = v.offsets[p];
        float3 cur = f3(c4.x, c4.y, c4.z);
        const float3 lim = f3(v.offset_limit * v.spacing.x, v.offset_limit * v.spacing.y,
                              v.offset_limit * v.spacing.z);
        if (4 * bft > R) {
            const float4 w = __ldg(dirs + (int)(cb & 0xffffffffu));
            const float tb = __uint_as_float((unsigned)(cb >> 32));
            const float3 vec = f3(tb * w.x, tb * w.y, tb * w.z);
            const float sx = fmaxf((lim.x - cur.x) / vec.x, (-lim.x - cur.x) / vec.x);
            const float sy = fmaxf((lim.y - cur.y) / vec.y, (-lim.y - cur.y) / vec.y);
            const float sz = fmaxf((lim.z - cur.z) / vec.z, (-lim.z - cur.z) / vec.z);
            const float scale = fminf(fminf(sx, sy), sz) - 1e-3f;
            if (scale > 1.0f) cur = f3(cur.x + vec.x * scale, cur.y + vec.y * scale, cur.z + vec.z * scale);
        } else if (ff != 0ull && cf != ~0ull) {
            const float4 wf = __ldg(dirs + (int)(ff & 0xffffffffu));
            const float4 wc = __ldg(dirs + (int)(cf & 0xffffffffu));
            if (!(wf.x * wc.x + wf.y * wc.y + wf.z * wc.z > 0.5f)) {
                const float step = fminf(0.2f, __uint_as_float((unsigned)(ff >> 32)));
                cur = f3(fminf(fmaxf(cur.x + step * wf.x, -lim.x), lim.x),
                         fminf(fmaxf(cur.y + step * wf.y, -lim.y), lim.y),
                         fminf(fmaxf(cur.z + step * wf.z, -lim.z), lim.z));
            }
        }
        v.offsets[p] = make_float4(cur.x, cur.y, cur.z, 0.0f);
    }
}

// Blocks of 256 threads for at most max_items of them, no more than `grid`
// nor, for the persistent passes, than are resident at once (a block of a
// later wave would start its own first batch when the others are done).
static int bounded_grid(int grid, int64_t max_items) {
    const int64_t need = (max_items + 255) / 256;
    return need < grid ? (need > 0 ? (int)need : 1) : grid;
}

cudaError_t launch_optimize(const DevScene& s, const VolView& v, const float4* dirs, int R, const int32_t* perm,
                            const int32_t* list, const int32_t* count, OptimizeScratch* scratch, uint32_t* next,
                            cudaStream_t st) {
    const int grid = bounded_grid(kClassCtas * sm_count(), (int64_t)v.n_probes * ((R + 31) / 32) * 32);
    return launch_pdl(k_optimize, grid, 256, 0, st, s, v, dirs, R, perm, list, count, scratch, next);
}

cudaError_t launch_classify(const DevScene& s, const VolView& v, const float4* dirs, int R, const int32_t* perm,
                            const int32_t* list, const int32_t* count, int4* scratch, uint32_t* next, int grid,
                            cudaStream_t st) {
    if (scratch)
        return launch_pdl(k_classify_split<false>,
                          bounded_grid(kClassCtas * sm_count(), (int64_t)v.n_probes * ((R + 31) / 32) * 32), 256, 0, st,
                          s, single_set(v), dirs, R, perm, list, count, scratch, next);
    return launch_pdl(k_classify, bounded_grid(grid, (int64_t)v.n_probes * 32), 256, 0, st, s, v, dirs, R, perm, list,
                      count);
}

cudaError_t launch_classify_multi(const DevScene& s, const VolSet& vs, const float4* dirs, int R,
                                  const int32_t* perm, const int32_t* list, const int32_t* count, int4* scratch,
                                  uint32_t* next, cudaStream_t st) {
    return launch_pdl(k_classify_split<true>, kClassCtas * sm_count(), 256, 0, st, s, vs, dirs, R, perm, list, count,
                      scratch, next);
}

cudaError_t launch_trace_shade(const DevScene& s, const VolView& v, const Lights& L, const float4* dirs,
                               int R, const int32_t* perm, const int32_t* active, const int32_t* count,
                               float4* records, int grid, cudaStream_t st) {
    const int64_t need = ((int64_t)v.n_probes * R + 127) / 128;
    const FastDiv dR = make_fast_div((uint32_t)R);
    return with_query_form<true, false>(query_form(v), [&](auto f) {
        constexpr int form = decltype(f)::value == kQueryFp32 ? kQueryFp32First : decltype(f)::value;
        return launch_pdl(k_trace_shade<form>, (int)std::min<int64_t>(grid, need), 128, 0, st, s, v, L, dirs,
                          R, dR, perm, active, count, records);
    });
}

template <bool MULTI>
static cudaError_t trace_wavefront(const DevScene& s, const VolSet& vs, const Lights& L, const float4* dirs, int R,
                                   const int32_t* perm, const int32_t* active, const int32_t* count,
                                   float4* records, int32_t* shadow_list, int32_t* hit_list, int32_t* shadow_count,
                                   int grid, int64_t max_rays, cudaStream_t st, cudaEvent_t* marks, int form) {
    // shadow_count (zeroed by the caller): [0] shadow rays, [1] front hits,
    // [2] and [4] the work counters of the two persistent passes
    uint32_t* next = reinterpret_cast<uint32_t*>(shadow_count + 2);
    uint32_t* next_shadow = reinterpret_cast<uint32_t*>(shadow_count + 4);
    const int shade_grid = bounded_grid(grid, max_rays);
    grid = bounded_grid(std::min(grid, trace_ctas(MULTI) * sm_count()), max_rays);
    cudaError_t e = cudaSuccess;
    if (marks && (e = cudaEventRecord(marks[0], st)) != cudaSuccess) return e;
    const FastDiv dR = make_fast_div((uint32_t)R);
    if ((e = launch_pdl(k_trace_primary<MULTI>, grid, 256, 0, st, s, vs, L, dirs, R, dR, perm, active, count, records,
                        shadow_list, hit_list, shadow_count, next, nullptr)) != cudaSuccess)
        return e;
    if (marks && (e = cudaEventRecord(marks[1], st)) != cudaSuccess) return e;
    if ((e = launch_pdl(k_trace_shadow<MULTI>, grid, 256, 0, st, s, vs, L, dirs, R, dR, active, records, shadow_list,
                        shadow_count, next_shadow, nullptr)) != cudaSuccess)
        return e;
    if (marks && (e = cudaEventRecord(marks[2], st)) != cudaSuccess) return e;
    e = with_query_form<true, !MULTI>(form, [&](auto f) {
        return launch_pdl(k_shade<MULTI, decltype(f)::value>, shade_grid, 256, 0, st, s, vs, L, dirs, R, dR, active, hit_list,
                          shadow_count + 1, records);
    });
    if (e != cudaSuccess) return e;
    if (marks && (e = cudaEventRecord(marks[3], st)) != cudaSuccess) return e;
    return cudaSuccess;
}

cudaError_t launch_trace_count(const DevScene& s, const VolView& v, const Lights& L, const float4* dirs, int R,
                               const int32_t* perm, const int32_t* active, const int32_t* count, float4* records,
                               int32_t* shadow_list, int32_t* hit_list, int32_t* shadow_count,
                               unsigned long long* stats, int grid, cudaStream_t st) {
    const VolSet vs = single_set(v);
    uint32_t* next = reinterpret_cast<uint32_t*>(shadow_count + 2);
    uint32_t* next_shadow = reinterpret_cast<uint32_t*>(shadow_count + 4);
    grid = std::min(grid, trace_ctas(false) * sm_count());
    cudaError_t e = cudaMemsetAsync(shadow_count, 0, 6 * sizeof(int32_t), st);
    if (e != cudaSuccess) return e;
    const FastDiv dR = make_fast_div((uint32_t)R);
    k_trace_primary<false, true><<<grid, 256, 0, st>>>(s, vs, L, dirs, R, dR, perm, active, count, records,
                                                        shadow_list, hit_list, shadow_count, next, stats);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_trace_shadow<false, true><<<grid, 256, 0, st>>>(s, vs, L, dirs, R, dR, active, records, shadow_list,
                                                       shadow_count, next_shadow, stats);
    return cudaGetLastError();
}

cudaError_t launch_trace_wavefront(const DevScene& s, const VolView& v, const Lights& L, const float4* dirs,
                                   int R, const int32_t* perm, const int32_t* active, const int32_t* count,
                                   float4* records, int32_t* shadow_list, int32_t* hit_list, int32_t* shadow_count,
                                   int grid, int64_t max_rays, cudaStream_t st, cudaEvent_t* marks) {
    return trace_wavefront<false>(s, single_set(v), L, dirs, R, perm, active, count, records, shadow_list, hit_list,
                                  shadow_count, grid, max_rays, st, marks, query_form(v));
}

cudaError_t launch_trace_wavefront_multi(const DevScene& s, const VolSet& vs, const Lights& L,
                                         const float4* dirs, int R, const int32_t* perm, const int32_t* active,
                                         const int32_t* count, float4* records, int32_t* shadow_list,
                                         int32_t* hit_list, int32_t* shadow_count, int grid, int64_t max_rays,
                                         cudaStream_t st, int form) {
    return trace_wavefront<true>(s, vs, L, dirs, R, perm, active, count, records, shadow_list, hit_list,
                                 shadow_count, grid, max_rays, st, nullptr, form);
}

cudaError_t launch_trace_rays(const DevScene& s, const float* orig, const float* dir, int64_t n,
                              float* t, int32_t* tri, int32_t* backface, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    int grid = (int)(blocks < 65535 ? blocks : 65535);
    k_trace_rays<<<grid, 256, 0, st>>>(s, orig, dir, n, t, tri, backface);
    return cudaGetLastError();
}

cudaError_t launch_gbuffer(const DevScene& s, float3 pos, float3 fwd, float3 right, float3 up,
                           float tan_half, float aspect, int w, int h, float* out_pos, float* out_nrm,
                           cudaStream_t st) {
    if ((int64_t)w * h == 0) return cudaSuccess;
    const int64_t tiles = (int64_t)((w + 7) / 8) * ((h + 3) / 4), blocks = (tiles + 7) / 8;
    int grid = (int)(blocks < 65535 ? blocks : 65535);
    k_gbuffer<<<grid, 256, 0, st>>>(s, pos, fwd, right, up, tan_half, aspect, w, h, out_pos, out_nrm);
    return cudaGetLastError();
}

}  // namespace ddgi
