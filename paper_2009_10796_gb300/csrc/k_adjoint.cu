// Adjoint of the differentiable forward: n frames of the update from a zero
// atlas with hysteresis 0 (every probe tracing), then the query.  Parameters
// are the emitters' radiance and the objects' albedo; geometry is fixed, so
// hits, distances and the query's backface / Chebyshev / trilinear weights
// are constants.  Reverse order:
//   k_query_adjoint   dE at query points -> texel gradients of the last atlas
//                     (and, of a query alone, k_border_fold: border-texel
//                     gradients -> the interior texels they copy)
//   k_blend_adjoint   texel gradients, the borders' folded in -> per-ray
//                     radiance gradients:
//                     dL_i = sum_t W[t][i] / s_t * de_t * de/dm (gamma chain)
//   k_shade_adjoint   rays re-traced: dL_i -> emitter radiance (front hits),
//                     albedo (direct + previous-frame term), and through the
//                     previous-frame query at the hit -> that atlas's texels
// Gradients accumulate with float atomics (order-dependent rounding only).
#include "blend_epilogue.cuh"
#include "traverse.cuh"

namespace ddgi {

// Per-warp scratch of the query adjoint: each point's eight corner gradients
// (rows padded to 33 so the eight corners of one point lie on distinct
// banks), its four bilinear weights, and one group's 96 sums.
constexpr int kAdjWarps = 4;   // warps per block of the kernels that scatter
struct AdjointScratch {
    float4 d[8][33];
    float4 bw[32];
    float sum[96];
};

// The decode b^(gamma/2) of an encoded value and its slope without the
// factor gamma/2, b^(gamma/2 - 1); both 0 for b <= 0.  The square roots are
// b * rsqrt(b) (hardware reciprocal square root, about 2 ulp; why that is
// enough: corner_weight).
template <int FORM>
__device__ __forceinline__ float decode_slope(float b, float half_gamma, float& slope) {
    if (!(b > 0.0f)) {
        slope = 0.0f;
        return 0.0f;
    }
    const bool general = FORM == kQueryGeneral;
    if (QueryForm<FORM>::kGamma1 || (general && half_gamma == 0.5f)) {
        slope = rsqrtf(b);
        return b * slope;
    }
    if (!general || half_gamma == 2.5f) {
        slope = b * (b * rsqrtf(b));
        return b * slope;
    }
    slope = powf(b, half_gamma - 1.0f);
    return powf(b, half_gamma);
}

// Six consecutive floats (a tap pair's two texels) added at p: pairs where
// they are 8-byte aligned (tile rows start on odd words too).
__device__ __forceinline__ void add_run6(float* p, float a0, float a1, float a2, float b0, float b1, float b2) {
    if ((reinterpret_cast<uintptr_t>(p) & 7) == 0) {
        atomicAdd(reinterpret_cast<float2*>(p), make_float2(a0, a1));
        atomicAdd(reinterpret_cast<float2*>(p + 2), make_float2(a2, b0));
        atomicAdd(reinterpret_cast<float2*>(p + 4), make_float2(b1, b2));
    } else {
        atomicAdd(p, a0);
        atomicAdd(reinterpret_cast<float2*>(p + 1), make_float2(a1, a2));
        atomicAdd(reinterpret_cast<float2*>(p + 3), make_float2(b0, b1));
        atomicAdd(p + 5, b2);
    }
}

// Reverse of query_M for a warp's 32 points (all lanes call; valid: the lane
// has one): M_c = A_c^2, A_c = sum_p w_p a_pc / sum_p w_p, a_pc =
// b_pc^(gamma/2), b the bilinear sample of probe p's tile in direction n.
// Adds dM's texel gradients to g_irr (float [P][tile][3]).
//
// A point touches 8 probes x 4 taps x 3 channels.  Bound by the atomics: one
// float atomic for each of the 96 took 2068 us for a 1280 x 720 G-buffer (16 x
// 8 x 16 probes), because neighbouring pixels share cage and footprint and so
// all add to the same few words.  Here the lanes with the same cage and
// footprint form a group; lane (corner, tap) sums the group's points through
// shared memory, in lane order, and the 96 sums go out as three atomics a
// lane on consecutive addresses (a tap pair's six floats are one run).  With
// more than kAdjMaxGroups groups (scattered points) a group costs more than
// it saves, and each lane adds its own 16 runs in pairs.  1920 x 1080 points
// of a hall seen from inside: 3894 -> 235 us; as many in random order inside a
// grid: 1161 -> 768 us.
template <int FORM>
__device__ __forceinline__ void query_M_adjoint_warp(const VolView& v, bool valid, float3 x, float3 n, float3 wo,
                                                     float3 dM, float* g_irr, AdjointScratch& sh) {
    constexpr int kUnroll = FORM == kQueryGeneral ? 1 : 8;
    const int lane = threadIdx.x & 31;
    const int N = v.irr_n + 2;
    Cage cage{};
    Footprint fp{0, 0, 0.0f, 0.0f};
    Bilerp bw{};
    if (valid) {
        const LocalPoint q = local_point(v, x, n, wo);
        cage = cage_of(v, q);
        fp = footprint(oct_encode(n), v.irr_n);
        bw = bilerp_weights(fp);
        unsigned act = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) act |= state_active(v.states[cage.probe(v, c)]) ? 1u << c : 0u;
        float sumw = 0.0f;
        float3 acc = f3(0.0f, 0.0f, 0.0f);
        // w_c and the slopes of corner c in shared memory until the sums are known
#pragma unroll kUnroll
        for (int c = 0; c < 8; ++c) {
            float4 d = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (act & (1u << c)) {
                const int p = cage.probe(v, c);
                const float w = corner_weight<FORM, true>(v, q, cage, c, p, n);
                float er, eg, eb;
                f2_unpack(irr_taps<FORM>(v, p, fp, bw, eb), er, eg);
                acc.x += w * decode_slope<FORM>(er, v.half_gamma, d.x);
                acc.y += w * decode_slope<FORM>(eg, v.half_gamma, d.y);
                acc.z += w * decode_slope<FORM>(eb, v.half_gamma, d.z);
                d.w = w;
                sumw += w;
            }
            sh.d[c][lane] = d;
        }
        if (!(sumw > 0.0f)) {
            valid = false;
        } else {
            // dM_c/db_pc = 2 A_c (w_p / sum w) gamma/2 b^(gamma/2 - 1)
            const float inv = 1.0f / sumw;
            const float k = 2.0f * v.half_gamma;
            const float3 kA = f3(dM.x * (acc.x * inv) * k, dM.y * (acc.y * inv) * k, dM.z * (acc.z * inv) * k);
#pragma unroll kUnroll
            for (int c = 0; c < 8; ++c) {
                const float4 d = sh.d[c][lane];
                const float w = d.w > 0.0f ? d.w * inv : 0.0f;
                // a zero slope (b <= 0) or weight gives 0, whatever dM is
                sh.d[c][lane] = make_float4(w * d.x != 0.0f ? kA.x * (w * d.x) : 0.0f, w * d.y != 0.0f ? kA.y * (w * d.y) : 0.0f,
                                            w * d.z != 0.0f ? kA.z * (w * d.z) : 0.0f, 0.0f);
            }
            sh.bw[lane] = make_float4(bw.w00, bw.w10, bw.w01, bw.w11);
        }
    }
    // groups of equal cage and footprint (cells below 2^26, texel rows and
    // columns below 2^6); the cell's probes differ with it
    const unsigned long long cell = (unsigned)cage.base[0] + (unsigned long long)v.counts.x *
                                        ((unsigned)cage.base[1] + (unsigned long long)v.counts.y * (unsigned)cage.base[2]);
    const unsigned long long key = (cell << 12) | (unsigned)(fp.y0 << 6) | (unsigned)fp.x0;
    unsigned left = __ballot_sync(0xffffffffu, valid);
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? key : ~0ull);
    const unsigned leaders = __ballot_sync(0xffffffffu, valid && __ffs(peers) - 1 == lane);
    __syncwarp();   // the corner gradients are in shared memory
    if (__popc(leaders) > kAdjMaxGroups) {
        if (valid) {
#pragma unroll 1
            for (int c = 0; c < 8; ++c) {
                const float4 d = sh.d[c][lane];
                if (d.x == 0.0f && d.y == 0.0f && d.z == 0.0f) continue;
                float* g = g_irr + ((int64_t)cage.probe(v, c) * v.irr_tile + fp.y0 * N + fp.x0) * 3;
                add_run6(g, d.x * bw.w00, d.y * bw.w00, d.z * bw.w00, d.x * bw.w10, d.y * bw.w10, d.z * bw.w10);
                add_run6(g + 3 * N, d.x * bw.w01, d.y * bw.w01, d.z * bw.w01, d.x * bw.w11, d.y * bw.w11,
                         d.z * bw.w11);
            }
        }
        __syncwarp();
        return;
    }
    const float* wp = reinterpret_cast<const float*>(sh.bw) + (lane & 3);
    const float4* dp = sh.d[lane >> 2];
    // of lane (corner, tap) and, for the atomics, of words lane + 32 k of the
    // 96: corner, tap, channel = i / 12, i / 3 % 4, i % 3
    while (left) {
        const int leader = __ffs(left) - 1;
        const unsigned group = __shfl_sync(0xffffffffu, peers, leader);
        left &= ~group;
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
        if (group == 0xffffffffu) {
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                const float4 d = dp[q];
                const float w = wp[4 * q];
                s0 = fmaf(d.x, w, s0);
                s1 = fmaf(d.y, w, s1);
                s2 = fmaf(d.z, w, s2);
            }
        } else {
            for (unsigned m = group; m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                const float4 d = dp[q];
                const float w = wp[4 * q];
                s0 = fmaf(d.x, w, s0);
                s1 = fmaf(d.y, w, s1);
                s2 = fmaf(d.z, w, s2);
            }
        }
        sh.sum[3 * lane] = s0;
        sh.sum[3 * lane + 1] = s1;
        sh.sum[3 * lane + 2] = s2;
        // the leader's cage: physical planes of both sides of each axis, and its first tap
        const int px0 = __shfl_sync(0xffffffffu, cage.px[0], leader), px1 = __shfl_sync(0xffffffffu, cage.px[1], leader);
        const int py0 = __shfl_sync(0xffffffffu, cage.py[0], leader), py1 = __shfl_sync(0xffffffffu, cage.py[1], leader);
        const int pz0 = __shfl_sync(0xffffffffu, cage.pz[0], leader), pz1 = __shfl_sync(0xffffffffu, cage.pz[1], leader);
        const int tap0 = __shfl_sync(0xffffffffu, fp.y0 * N + fp.x0, leader);
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int i = lane + 32 * k;
            const int t = i / 3, c = t >> 2;
            const float s = sh.sum[i];
            if (s != 0.0f) {
                const int p = (c & 1 ? px1 : px0) + v.counts.x * ((c & 2 ? py1 : py0) + v.counts.y * (c & 4 ? pz1 : pz0));
                const int tap = tap0 + ((t >> 1) & 1) * N + (t & 1);
                atomicAdd(g_irr + ((int64_t)p * v.irr_tile + tap) * 3 + (i - 3 * t), s);
            }
        }
        __syncwarp();   // the sums are read before the next group's are written
    }
}

__device__ __forceinline__ float3 direction_to(float3 cam, float3 x, float3 n) {
    const float3 wo = cam - x;
    const float l = length(wo);
    return l < 1e-6f ? n : (1.0f / l) * wo;
}

// ---- order of scattered points ---------------------------------------------
// A warp of query_M_adjoint_warp wants points of few cages and footprints.
// Points in random order (a training step's samples of the surfaces) are put
// into bins by cage and by the axis that their normal is nearest to: a count
// of each bin, ranges given to the bins in any order, the points' indices in
// their ranges.  1 M points on the boxes of a room, 2048 probes: 338 us
// unordered, 178 us ordered, the three passes included.  Points that neighbour
// each other already (a G-buffer) are found so by the first pass, and the
// others leave at once.
__global__ void __launch_bounds__(256) k_point_bins(VolView v, const float* __restrict__ pos,
                                                    const float* __restrict__ nrm, int n, float3 cam, PointOrder o) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    int bin = -1;
    if (q < n) {
        const float3 x = f3(pos[3 * q], pos[3 * q + 1], pos[3 * q + 2]);
        const float3 m = f3(nrm[3 * q], nrm[3 * q + 1], nrm[3 * q + 2]);
        const Cage k = cage_of(v, local_point(v, x, m, direction_to(cam, x, m)));
        const float ax = fabsf(m.x), ay = fabsf(m.y), az = fabsf(m.z);
        const int axis = ax >= ay && ax >= az ? 0 : ay >= az ? 1 : 2;
        const float along = axis == 0 ? m.x : axis == 1 ? m.y : m.z;
        const int cell = max(k.base[0], 0) + v.counts.x * (max(k.base[1], 0) + v.counts.y * max(k.base[2], 0));
        bin = kPointBins * cell + 2 * axis + (along < 0.0f ? 1 : 0);   // cell < probes
    }
    const unsigned same = __match_any_sync(0xffffffffu, bin);
    const int leader = __ffs(same) - 1;
    int first = 0;
    if (bin >= 0 && lane == leader) first = atomicAdd(o.bins + bin, __popc(same));
    first = __shfl_sync(0xffffffffu, first, leader);
    if (q < n) {
        o.bin[q] = bin;
        o.rank[q] = first + __popc(same & ((1u << lane) - 1u));
    }
    const int groups = __syncthreads_count(bin >= 0 && lane == leader);
    if (threadIdx.x == 0) atomicAdd(o.groups, groups);
}

// Counts -> first indices: a warp takes one range for its 32 bins.
__global__ void __launch_bounds__(256) k_point_ranges(int n_bins, int n, PointOrder o) {
    pdl_wait();
    pdl_trigger();
    if (!points_scattered(o, n)) return;
    const int b = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int count = b < n_bins ? o.bins[b] : 0;
    int end = count;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int below = __shfl_up_sync(0xffffffffu, end, d);
        if (lane >= d) end += below;
    }
    int first = 0;
    if (lane == 31) first = atomicAdd(o.taken, end);
    first = __shfl_sync(0xffffffffu, first, 31);
    if (b < n_bins) o.bins[b] = first + end - count;
}

__global__ void __launch_bounds__(256) k_point_order(int n, PointOrder o) {
    pdl_wait();
    pdl_trigger();
    if (!points_scattered(o, n)) return;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) o.order[o.bins[o.bin[q]] + o.rank[q]] = q;
}

template <int FORM>
__global__ void __launch_bounds__(32 * kAdjWarps) k_query_adjoint(VolView v, const float* __restrict__ pos,
                                                                  const float* __restrict__ nrm, int64_t n, float3 cam,
                                                                  const float* __restrict__ dE, float* g_irr,
                                                                  PointOrder o) {
    pdl_wait();
    __shared__ AdjointScratch sh[kAdjWarps];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const bool ordered = o.order && points_scattered(o, (int)n);
    // warp-uniform loop: 32 consecutive points per warp
    for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < n; q0 += stride) {
        int64_t q = q0 + (threadIdx.x & 31);
        float3 x = f3(0.0f, 0.0f, 0.0f), nn = x, wo = x, dM = x;
        bool valid = q < n;
        if (valid) {
            if (ordered) q = o.order[q];
            x = f3(pos[3 * q], pos[3 * q + 1], pos[3 * q + 2]);
            nn = f3(nrm[3 * q], nrm[3 * q + 1], nrm[3 * q + 2]);
            valid = nn.x != 0.0f || nn.y != 0.0f || nn.z != 0.0f;
            wo = direction_to(cam, x, nn);
            const float pi = 3.14159265358979323846f;
            dM = f3(pi * dE[3 * q], pi * dE[3 * q + 1], pi * dE[3 * q + 2]);
        }
        query_M_adjoint_warp<FORM>(v, valid, x, nn, wo, dM, g_irr, sh[threadIdx.x >> 5]);
    }
}

// One block per probe: each interior texel gathers the gradients of the
// border texels that copy it, then the border gradients are cleared.
__global__ void k_border_fold(float* g_irr, int n) {
    const int N = n + 2;
    float* t = g_irr + (int64_t)blockIdx.x * N * N * 3;
    for (int q = threadIdx.x; q < n * n; q += blockDim.x) {
        int x = 1 + q % n, y = 1 + q / n;
        float add[3] = {0.0f, 0.0f, 0.0f};
        auto gather = [&](int bx, int by) {
            for (int c = 0; c < 3; ++c) add[c] += t[(by * N + bx) * 3 + c];
        };
        if (x == 1) gather(0, n + 1 - y);
        if (x == n) gather(n + 1, n + 1 - y);
        if (y == 1) gather(n + 1 - x, 0);
        if (y == n) gather(n + 1 - x, n + 1);
        if (x == n && y == n) gather(0, 0);
        if (x == 1 && y == n) gather(n + 1, 0);
        if (x == n && y == 1) gather(0, n + 1);
        if (x == 1 && y == 1) gather(n + 1, n + 1);
        for (int c = 0; c < 3; ++c) t[(y * N + x) * 3 + c] += add[c];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < N * N; q += blockDim.x) {
        int x = q % N, y = q / N;
        if (x == 0 || y == 0 || x == N - 1 || y == N - 1)
            for (int c = 0; c < 3; ++c) t[q * 3 + c] = 0.0f;
    }
}

// Texel gradients -> per-ray radiance gradients, a block for PB probes:
// each interior texel takes the gradients of the border texels that copy it
// (for_border_copies) and becomes g de/dm inv_s, once, in shared memory;
// then thread i sums dL_i = sum_t W[t][i] of that over the texels for the
// block's probes, so a weight read serves PB of them.  e is the texel of the
// atlas this frame wrote (e = m^(1/gamma)).  Bound by the weight reads; a
// thread per (probe, ray) that evaluated de/dm for each of its texels took
// 59 us for 2048 probes x 128 rays (three powf per texel and ray), and the
// border fold 5 us in a launch of its own.
template <int PB>
__global__ void __launch_bounds__(128) k_blend_adjoint(VolView v_after, const float* __restrict__ w_irr,
                                                       const float* __restrict__ inv_s, const float* __restrict__ g_irr,
                                                       int P, int R, float4* __restrict__ gL) {
    extern __shared__ float4 s_gd[];   // [PB][n^2]
    const int n = v_after.irr_n, N = n + 2, ti = n * n;
    const int p0 = blockIdx.x * PB, np = min(PB, P - p0);
    for (int q = threadIdx.x; q < PB * ti; q += blockDim.x) {
        const int b = q / ti, t = q - b * ti, x = 1 + t % n, y = 1 + t / n;
        float4 gd = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float is = b < np ? __ldg(inv_s + t) : -1.0f;
        if (is >= 0.0f) {
            const float* g = g_irr + (int64_t)(p0 + b) * N * N * 3;
            float3 s = f3(0.0f, 0.0f, 0.0f);
            auto add = [&](int bx, int by) {
                const float* c = g + (by * N + bx) * 3;
                s = s + f3(__ldg(c), __ldg(c + 1), __ldg(c + 2));
            };
            add(x, y);
            for_border_copies(x, y, n, add);
            const float3 e = load_irr<true>(v_after, p0 + b, x, y);
            // de/dm = (1/gamma) e^(1 - gamma); at e = 0 only gamma = 1 has a derivative
            auto slope = [&](float c) {
                if (v_after.gamma == 1.0f) return is;
                return c > 0.0f ? v_after.inv_gamma * powf(c, 1.0f - v_after.gamma) * is : 0.0f;
            };
            gd = make_float4(s.x * slope(e.x), s.y * slope(e.y), s.z * slope(e.z), 0.0f);
        }
        s_gd[q] = gd;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < R; i += blockDim.x) {
        float3 a[PB];
#pragma unroll
        for (int b = 0; b < PB; ++b) a[b] = f3(0.0f, 0.0f, 0.0f);
#pragma unroll 4
        for (int t = 0; t < ti; ++t) {
            const float w = __ldg(w_irr + (int64_t)t * R + i);
            if (w == 0.0f) continue;
#pragma unroll
            for (int b = 0; b < PB; ++b) {
                const float4 gd = s_gd[b * ti + t];
                a[b].x = fmaf(w, gd.x, a[b].x);
                a[b].y = fmaf(w, gd.y, a[b].y);
                a[b].z = fmaf(w, gd.z, a[b].z);
            }
        }
#pragma unroll
        for (int b = 0; b < PB; ++b)
            if (b < np) gL[(int64_t)(p0 + b) * R + i] = make_float4(a[b].x, a[b].y, a[b].z, 0.0f);
    }
}

// dst[3 key ..] += val over a warp's lanes (all call; key < 0: none): a group
// of lanes with one key is summed and added once, for the first kSumGroups
// keys; the lanes left add their own.
constexpr int kSumGroups = 6;
__device__ __forceinline__ void add3_by_key(float* dst, int key, float3 val) {
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, key >= 0);
    for (int round = 0; todo != 0 && round < kSumGroups; ++round) {
        const int k = __shfl_sync(0xffffffffu, key, __ffs(todo) - 1);
        const bool mine = key == k;
        float3 s = mine ? val : f3(0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            s = s + f3(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o),
                       __shfl_xor_sync(0xffffffffu, s.z, o));
        if (lane < 3) atomicAdd(dst + 3 * k + lane, lane == 0 ? s.x : lane == 1 ? s.y : s.z);
        todo &= ~__ballot_sync(0xffffffffu, mine);
    }
    if (todo & (1u << lane)) {
        atomicAdd(dst + 3 * key + 0, val.x);
        atomicAdd(dst + 3 * key + 1, val.y);
        atomicAdd(dst + 3 * key + 2, val.z);
    }
}

// Thread per (probe, ray) of frame f, re-traced against the scene.  v_before
// is the atlas the frame's hit shading sampled (the previous frame's).  Bound by
// the walk and, with a frame before it, by the atomics of scattered hits; so a
// warp takes a compact cone of one probe's rays (perm), whose hits share
// objects, emitters and cages.  Five CTAs to an SM (96 registers): 2048 probes
// x 128 rays in a room of 16000 boxes, two frames, take 330 us (402 us with rays
// in the spiral's order and an atomic for each hit; at four CTAs 360 us, at six
// as at four).
template <int FORM>
__global__ void __launch_bounds__(32 * kAdjWarps, 5)
k_shade_adjoint(DevScene s, VolView v_before, Lights L, const float4* __restrict__ dirs, int P, int R, FastDiv dR,
                const int32_t* __restrict__ perm, const float4* __restrict__ gL, float* d_emit, float* d_albedo,
                float* g_prev, int with_prev) {
    const unsigned total = (unsigned)P * (unsigned)R;   // below 2^31
    const unsigned stride = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const float3 tol = f3(-L.sun_dir.x, -L.sun_dir.y, -L.sun_dir.z);
    const RayPre r_sun = ray_pre(f3(0.0f, 0.0f, 0.0f), tol);
    __shared__ AdjointScratch sh[kAdjWarps];
    int2 stack[kStackSize4];
    WwLane<kStackSize4, int2> w;
    w.stack = stack;
    // warp-uniform loop: 32 rays per warp through the warp-cooperative 4-wide
    // walk (rays without a gradient take part without tracing), then their
    // shadow rays the same way
    for (unsigned base = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < total; base += stride) {
        const unsigned id = min(base + (unsigned)lane, total - 1);
        const int p = (int)fast_div(id, dR);
        const int i = __ldg(perm + ((int)id - p * R));
        const float4 g4 = gL[(size_t)p * R + i];
        const bool valid = base + lane < total && (g4.x != 0.0f || g4.y != 0.0f || g4.z != 0.0f);
        float3 o = probe_pos_phys(v_before, p);
        float4 d4 = __ldg(dirs + i);
        float3 d = f3(d4.x, d4.y, d4.z);
        const RayPre r = ray_pre_packed(o, d, __ldg(dirs + R + 2 * i), __ldg(dirs + R + 2 * i + 1));
        ww_start(s, w, valid);
        do {
            ww4_round<false, false, true>(s, r, w);
        } while (__ballot_sync(0xffffffffu, w.node != kDone) != 0);
        const Hit h = w.h;
        bool front = false;
        float3 n = f3(0.0f, 0.0f, 1.0f), x = o;
        float cosl = 0.0f;
        if (valid && h.orig >= 0) {
            const float4* T = s.tris + 3 * (int64_t)h.k;
            float4 p0 = __ldg(T), p1 = __ldg(T + 1), p2 = __ldg(T + 2);
            float3 ng = cross(f3(p1.x - p0.x, p1.y - p0.y, p1.z - p0.z), f3(p2.x - p0.x, p2.y - p0.y, p2.z - p0.z));
            front = !(dot(d, ng) > 0.0f);   // back faces carry no radiance
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
        const float3 wo = f3(-d.x, -d.y, -d.z);
        float3 dM = f3(0.0f, 0.0f, 0.0f);
        int2 at = make_int2(-1, -1);   // object, emitter
        float3 dA = f3(0.0f, 0.0f, 0.0f);
        if (front) {
            at = __ldg(s.attr + h.orig);
            float3 direct = f3(0.0f, 0.0f, 0.0f);
            if (lit) {
                float kk = cosl * 0.318309886183790672f;
                direct = f3(L.sun_irr.x * kk, L.sun_irr.y * kk, L.sun_irr.z * kk);
            }
            const float3 M = query_M<FORM>(v_before, x, n, wo);
            dA = f3(g4.x * (direct.x + M.x), g4.y * (direct.y + M.y), g4.z * (direct.z + M.z));
            const float4 rho = __ldg(s.albedo + at.x);
            dM = f3(g4.x * rho.x, g4.y * rho.y, g4.z * rho.z);
        }
        add3_by_key(d_emit, at.y, f3(g4.x, g4.y, g4.z));
        add3_by_key(d_albedo, at.x, dA);
        if (with_prev) query_M_adjoint_warp<FORM>(v_before, front, x, n, wo, dM, g_prev, sh[threadIdx.x >> 5]);
    }
}

// Copies per-object albedo [O][3] and per-emitter radiance [E][3] (device)
// into the scene's tables, keeping each object's flags.
__global__ void k_set_materials(float4* albedo, int n_obj, const float* __restrict__ alb, float4* emit, int n_em,
                                const float* __restrict__ em) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_obj + n_em; k += gridDim.x * blockDim.x) {
        if (k < n_obj) {
            if (alb) {
                float4 a = albedo[k];
                albedo[k] = make_float4(alb[3 * k], alb[3 * k + 1], alb[3 * k + 2], a.w);
            }
        } else if (em) {
            int e = k - n_obj;
            emit[e] = make_float4(em[3 * e], em[3 * e + 1], em[3 * e + 2], 0.0f);
        }
    }
}

static int grid_for(int64_t n, int block) {
    int64_t b = (n + block - 1) / block;
    return (int)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

static cudaError_t query_adjoint(const VolView& v, const float* pos, const float* nrm, int64_t n, float3 cam,
                                 const float* dE, float* g_irr, const PointOrder& o, cudaStream_t st) {
    return with_query_form(query_form(v), [&](auto f) {
        return launch_pdl(k_query_adjoint<decltype(f)::value>, grid_for(n, 32 * kAdjWarps), 32 * kAdjWarps, 0, st, v, pos,
                          nrm, n, cam, dE, g_irr, o);
    });
}

// Orders m points where there is scratch (point_order_bytes) and there are at
// least 16 of them to a probe; else o stays empty and they are taken as they
// come.  The adjoint of a training step on 2048 probes gains 181 us of 1438 with
// 1 M points, 14 of 989 with 130,000 and nothing any more with 40,000.  Points
// in order by cage already lose nothing (1198 us without, 1175 with).
cudaError_t order_points(const VolView& v, const float* pos, const float* nrm, int64_t m, float3 cam, int32_t* scratch,
                         PointOrder& o, cudaStream_t st) {
    if (!scratch || m < 16 * (int64_t)v.n_probes) return cudaSuccess;
    const int n_bins = kPointBins * v.n_probes, blocks = (int)((m + 255) / 256);
    o = point_order(scratch, v.n_probes);
    cudaError_t e = cudaMemsetAsync(o.groups, 0, sizeof(int32_t) * (2 + (size_t)n_bins), st);
    if (e != cudaSuccess) return e;
    k_point_bins<<<blocks, 256, 0, st>>>(v, pos, nrm, (int)m, cam, o);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_pdl(k_point_ranges, (n_bins + 255) / 256, 256, 0, st, n_bins, (int)m, o)) != cudaSuccess) return e;
    return launch_pdl(k_point_order, blocks, 256, 0, st, (int)m, o);
}

cudaError_t launch_query_adjoint(const VolView& v, const float* pos, const float* nrm, int64_t n, float3 cam,
                                 const float* dE, float* g_irr, int32_t* scratch, cudaStream_t st) {
    while (n > 0) {
        const int64_t m = scratch ? std::min<int64_t>(n, kPointsOrdered) : n;
        PointOrder o{};
        cudaError_t e = order_points(v, pos, nrm, m, cam, scratch, o, st);
        if (e != cudaSuccess) return e;
        e = query_adjoint(v, pos, nrm, m, cam, dE, g_irr, o, st);
        if (e != cudaSuccess) return e;
        pos += 3 * m;
        nrm += 3 * m;
        dE += 3 * m;
        n -= m;
    }
    return cudaSuccess;
}

cudaError_t launch_border_fold(float* g_irr, int P, int n, cudaStream_t st) {
    k_border_fold<<<P, 64, 0, st>>>(g_irr, n);
    return cudaGetLastError();
}

// Four probes to a block while their texels fit the default shared memory
// (up to 27 x 27 texels), else one (32 x 32).
cudaError_t launch_blend_adjoint(const VolView& v_after, const float* w_irr, const float* inv_s, const float* g_irr,
                                 int P, int R, float4* gL, cudaStream_t st) {
    const size_t tile = sizeof(float4) * (size_t)v_after.irr_n * v_after.irr_n;
    if (4 * tile <= 48 * 1024)
        k_blend_adjoint<4><<<(P + 3) / 4, 128, 4 * tile, st>>>(v_after, w_irr, inv_s, g_irr, P, R, gL);
    else
        k_blend_adjoint<1><<<P, 128, tile, st>>>(v_after, w_irr, inv_s, g_irr, P, R, gL);
    return cudaGetLastError();
}

cudaError_t launch_shade_adjoint(const DevScene& s, const VolView& v_before, const Lights& L, const float4* dirs,
                                 int P, int R, const int32_t* perm, const float4* gL, float* d_emit,
                                 float* d_albedo, float* g_prev, int with_prev, cudaStream_t st) {
    return with_query_form<false>(query_form(v_before), [&](auto f) {
        k_shade_adjoint<decltype(f)::value><<<grid_for((int64_t)P * R, 32 * kAdjWarps), 32 * kAdjWarps, 0, st>>>(
            s, v_before, L, dirs, P, R, make_fast_div((uint32_t)R), perm, gL, d_emit, d_albedo, g_prev, with_prev);
        return cudaGetLastError();
    });
}

cudaError_t launch_set_materials(float4* albedo, int n_obj, const float* alb, float4* emit, int n_em, const float* em,
                                 cudaStream_t st) {
    k_set_materials<<<grid_for(n_obj + n_em, 128), 128, 0, st>>>(albedo, n_obj, alb, emit, n_em, em);
    return cudaGetLastError();
}

}  // namespace ddgi
