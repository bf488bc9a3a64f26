// Adjoint of the ray caster: dL/d(table entries) and dL/d(voxel values) from
// dL/d(image), for front-to-back "over" with early termination and for MIP.
//
// Composite, per ray (samples k = 0..n-1 executed, T_k the transmittance
// before sample k, a_k and c_k the sample's alpha and colour):
//     C = sum_k T_k a_k c_k,   A = 1 - prod_k (1 - a_k)
//     dC/dc_k = T_k a_k,  dC/da_k = T_k (c_k - R_k),  dA/da_k = T_k P_k
// with R_k the colour composited behind sample k starting from transmittance 1
// and P_k the transmittance behind it: (R_k, P_k) is the "over" composite of
// the samples after k, an associative product, so nothing divides by 1 - a.
// The forward march is recomputed chunk by chunk instead of storing samples:
// the first pass keeps the transmittance at the start of every 32-sample chunk;
// the reverse pass recomputes each chunk from its checkpoint, one sample per
// lane, and gets (R_k, P_k) from a warp suffix scan carried from the chunks
// behind.  Table gradients are collected ray by ray in a histogram per warp in shared
// memory, added up per warp in device memory, and summed over the blocks in FP64 by a final
// kernel; voxel gradients are scattered through the trilinear weights with FP32 atomics.
// MIP: the image is TF(max v); the gradient reaches the first maximal sample.
#include <algorithm>

#include "vr_device.cuh"
#include "vr_ff.cuh"
#include "vr_tma.cuh"

namespace vr {

namespace {

constexpr int kAdjThreads = 128;
constexpr int kAdjWarps = kAdjThreads / 32;
constexpr int kAdjMaxChunks = 320;  // 32-sample transmittance checkpoints per ray
constexpr int kAdjKeep = 6;         // chunks whose samples the forward pass keeps for the reverse pass
constexpr int kDevTooManySegments = 2;
constexpr int kAdjCrowd = 8;        // samples on one table interval that are reduced by the whole warp

// Tables of up to kAdjTF entries and the default brick edge are compiled in (FAST): the
// table's arrays are S entries apart, S = 0 standing for its length.
constexpr int kAdjTF = 256;
template <int S> __device__ __forceinline__ int stride(int n) { return S ? S : n; }

struct TFGrad {
    int i;
    float w;
    float4 rgba, slope;
};

template <int S>
__device__ __forceinline__ TFGrad tf_eval(const float* __restrict__ tab, int n, float vmin,
                                          float inv_range, float val) {
    TFGrad r;
    const float u0 = (val - vmin) * inv_range;
    const bool inside = u0 > 0.f && u0 < 1.f;
    const float u = fminf(fmaxf(u0, 0.f), 1.f);
    const float x = u * (float)(n - 1);
    r.i = min((int)x, n - 2);
    r.w = x - (float)r.i;
    const int d = stride<S>(n);
    const float* t = tab + r.i;
    const float4 a = make_float4(t[0], t[d], t[2 * d], t[3 * d]);
    const float4 b = make_float4(t[1], t[d + 1], t[2 * d + 1], t[3 * d + 1]);
    const float4 up = make_float4(b.x - a.x, b.y - a.y, b.z - a.z, b.w - a.w);
    r.rgba = make_float4(fmaf(r.w, up.x, a.x), fmaf(r.w, up.y, a.y), fmaf(r.w, up.z, a.z), fmaf(r.w, up.w, a.w));
    const float s = inside ? (float)(n - 1) * inv_range : 0.f;
    r.slope = make_float4(up.x * s, up.y * s, up.z * s, up.w * s);
    return r;
}

// Opacity alone, of the table above.
template <int S>
__device__ __forceinline__ float tf_alpha(const float* __restrict__ tab, int n, float vmin, float inv_range,
                                          float val) {
    float x;
    const int i = tf_node(n, vmin, inv_range, val, x);
    const float w = x - (float)i;
    const float* t = tab + 3 * stride<S>(n) + i;
    const float a = t[0], b = t[1];
    return fmaf(w, b - a, a);
}

// Scatter dv to the 8 voxels of the sample at slot coordinate g of brick b.
__device__ __forceinline__ void scatter_voxels(float* __restrict__ dvol, const VolDev& v, int bx, int by,
                                               int bz, float gx, float gy, float gz, float dv) {
    if (dv == 0.f) return;
    const float fx0 = floorf(gx), fy0 = floorf(gy), fz0 = floorf(gz);
    const float fx = gx - fx0, fy = gy - fy0, fz = gz - fz0;
    // slot index s <-> cube index b*B + s - 1, clamped to the cube like the ghost layer
    const int x0 = bx * v.B + (int)fx0 - 1, y0 = by * v.B + (int)fy0 - 1, z0 = bz * v.B + (int)fz0 - 1;
    const int xl = min(max(x0, 0), v.nx - 1), yl = min(max(y0, 0), v.ny - 1), zl = min(max(z0, 0), v.nz - 1);
    const int dx = min(max(x0 + 1, 0), v.nx - 1) - xl;  // 0 where both clamp to the same voxel, else 1
    const long long dy = min(max(y0 + 1, 0), v.ny - 1) > yl ? v.nx : 0;
    const long long dz = min(max(z0 + 1, 0), v.nz - 1) > zl ? (long long)v.nx * v.ny : 0;
    float* p = dvol + ((long long)zl * v.ny + yl) * v.nx + xl;
    const float wz[2] = {(1.f - fz) * dv, fz * dv};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float* q = p + (c & 1 ? dy : 0) + (c >> 1 ? dz : 0);
        const float w = wz[c >> 1] * (c & 1 ? fy : 1.f - fy);
        if (dx && (reinterpret_cast<uintptr_t>(q) & 7) == 0) {  // an aligned x-pair in one reduction
            asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(q), "f"(w * (1.f - fx)), "f"(w * fx)
                         : "memory");
        } else {
            atomicAdd(q, w * (1.f - fx));
            atomicAdd(q + dx, w * fx);
        }
    }
}

// Adds w gc to one entry of a table gradient.
__device__ __forceinline__ void add_entry(float4* g, float w, float4 gc) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(g), "f"(w * gc.x), "f"(w * gc.y),
                 "f"(w * gc.z), "f"(w * gc.w)
                 : "memory");
}
__device__ __forceinline__ void add_tf(float4* g, const TFGrad& t, float4 gc) {
    add_entry(g + t.i, 1.f - t.w, gc);
    add_entry(g + t.i + 1, t.w, gc);
}

// One sample a lane (act) into the warp's histogram: wk and ga are shared by the entries t.i
// and t.i + 1 with weights 1 - t.w and t.w.  The lanes of one interval are added up first: by
// a reduction over the warp where there are at least kAdjCrowd of them (regions of one value:
// 256^3 with all below 3 sigma set to 0 and a fifth of the opacity, 23.5 ms a step, and 30.2 one
// lane at a time; 6 the same, 4 costs 6 % on noise), else by the group's first lane, one mate
// at a time (noise: 7.80 ms a step, and 7.93 with the lanes taking turns at the entries).  Each
// interval then has one writer; lower entries are written before upper ones.
__device__ __forceinline__ void collect_sample(float2* __restrict__ hist, const TFGrad& t, bool act, int lane,
                                               float wk, float ga) {
    constexpr unsigned int FULL = 0xffffffffu;
    const unsigned int same = __match_any_sync(FULL, t.i);
    const float w1 = t.w, w0 = 1.f - t.w;
    float c0 = w0 * wk, c1 = w1 * wk, a0 = w0 * ga, a1 = w1 * ga;
    const bool crowd = act && __popc(same) >= kAdjCrowd;
    for (unsigned int left = __ballot_sync(FULL, crowd); left;) {
        const int first = __ffs(left) - 1;
        const unsigned int group = __shfl_sync(FULL, same, first);
        const bool in = (group >> lane) & 1u;
        float4 v = in ? make_float4(c0, a0, c1, a1) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            v.x += __shfl_xor_sync(FULL, v.x, off);
            v.y += __shfl_xor_sync(FULL, v.y, off);
            v.z += __shfl_xor_sync(FULL, v.z, off);
            v.w += __shfl_xor_sync(FULL, v.w, off);
        }
        if (lane == first) {
            hist[t.i].x += v.x;
            hist[t.i].y += v.y;
            hist[t.i + 1].x += v.z;
            hist[t.i + 1].y += v.w;
        }
        __syncwarp();
        left &= ~group;
    }
    // the others: a group's first lane adds up its mates
    const bool lead = act && !crowd && lane == __ffs(same) - 1;
    unsigned int mates = lead ? same & (same - 1) : 0u;
    const int rounds = __reduce_max_sync(FULL, __popc(mates));
    for (int q = 0; q < rounds; ++q) {
        const int src = mates ? __ffs(mates) - 1 : lane;
        const float sw = __shfl_sync(FULL, w1, src), sk = __shfl_sync(FULL, wk, src), sg = __shfl_sync(FULL, ga, src);
        if (mates) {
            c0 = fmaf(1.f - sw, sk, c0);
            c1 = fmaf(sw, sk, c1);
            a0 = fmaf(1.f - sw, sg, a0);
            a1 = fmaf(sw, sg, a1);
        }
        mates &= mates - 1;
    }
    // no two first lanes share an interval: lower entries, then upper ones
    if (lead) {
        hist[t.i].x += c0;
        hist[t.i].y += a0;
    }
    __syncwarp();
    if (lead) {
        hist[t.i + 1].x += c1;
        hist[t.i + 1].y += a1;
    }
    __syncwarp();
}

// One warp per ray, its lanes on 32 consecutive samples (a chunk).  A warp
// claims a tile of 32 pixels, sets up their rays once (one lane each, float-float)
// into shared memory and then walks them.  Composite: the forward pass keeps
// the transmittance at the start of every chunk (in the registers of lane chunk
// mod 32) and finds the termination sample by a ballot on a warp prefix product of
// (1 - a); the reverse pass recomputes each chunk from its checkpoint and gets what is
// behind every sample from a warp suffix scan of "over", carried from chunk to chunk.
// The scan composites the scalar s = sum_c dL/dC_c c (over the colour channels) and the
// transmittance, two values instead of four: dL/da_k needs the colour behind a sample
// only through that sum.  MIP: a warp maximum per chunk keeps the first
// maximal sample.  Sample positions: the float-float ray from the set-up, one
// float-float anchor per chunk, lane offsets in FP32, each lane
// reading the brick that holds its sample (the ghost layer makes any brick
// within half a voxel give the same value, and keeps the corners inside the slot).
//
// Table gradient.  A float atomicAdd in shared memory is a compare-and-swap loop,
// repeated while lanes meet on an entry; eight a sample (4 channels x 2 entries) took
// 30 % of the kernel.  A ray is collected in a histogram of its warp instead, two values an
// entry (dL/dc_k = dL/dC T_k a_k: one weight T_k a_k for all three channels, and dL/da_k),
// without atomics: lanes whose samples fall between the same two entries are found by
// __match_any_sync and added up in registers first (collect_sample).  Everything is FP32, so
// a term keeps its 24 bits however small the transmittance before it is (histograms in fixed
// point, with integer atomics, were 4 % faster over the step and lost the entries that are
// reached only behind others; float atomics into the histograms were 13 % slower).  After a
// ray, the entries touched go to the warp's gradient in device memory, a reduction of four
// floats each: no copy of the table's gradient takes shared memory from the L1 cache (one a
// warp there made the MIP gradient a third slower), and no sum runs over more rays than a warp's.
//
// Bound by L1 data wavefronts (86 % busy) and the voxel reductions in L2 (70 %), with issue
// slots at 55 % (8 views): two passes over a chunk took some 1100 warp instructions before the
// anchors of a ray's chunks were made together, the default brick edge and table stride
// compiled in, the voxel addresses taken from one base and aligned x-pairs reduced
// together.  16 views of 512 x 512 on 256^3 FP32, forward and backward (one seed): 11.85 -> 7.73 ms.  Six CTAs an SM and kAdjKeep = 4 instead of five and 6: the same.
struct RaySetup {
    float o_hi[3], o_lo[3], e_hi[3], e_lo[3];
    int k0, k1;
    float4 g;  // dL/dI of the pixel
};

__device__ __forceinline__ unsigned int ord_enc_f(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Brick (bx, by, bz) and slot coordinate g of sample k + lane of the ray.
struct LaneSample {
    int bx, by, bz;
    float gx, gy, gz;
    long long base;
};

// brick index along one axis of the float-float position p (clamped to the grid)
// and the slot coordinate of p in it
__device__ __forceinline__ int anchor_axis(ff p, const VolDev& v, int nb, float& g) {
    const int b = min(max(((int)floorf(p.hi)) >> v.log2B, 0), nb - 1);
    g = __fadd_rn(__fsub_rn(p.hi, (float)(b << v.log2B)), p.lo) + 0.5f;
    return b;
}

// Brick index and slot coordinate of one sample.
struct __align__(16) SampleAnchor {
    float gx, gy, gz;
    int bx, by, bz;
};

__device__ __forceinline__ void sample_anchor(const RaySetup& r, int k, const VolDev& v, SampleAnchor& A) {
    const ff fk = ff_of_int(k);  // exact for any sample index
    A.bx = anchor_axis(ff_add(ff{r.o_hi[0], r.o_lo[0]}, ff_mul(ff{r.e_hi[0], r.e_lo[0]}, fk)), v, v.nbx, A.gx);
    A.by = anchor_axis(ff_add(ff{r.o_hi[1], r.o_lo[1]}, ff_mul(ff{r.e_hi[1], r.e_lo[1]}, fk)), v, v.nby, A.gy);
    A.bz = anchor_axis(ff_add(ff{r.o_hi[2], r.o_lo[2]}, ff_mul(ff{r.e_hi[2], r.e_lo[2]}, fk)), v, v.nbz, A.gz);
}

// This lane's sample of chunk c.  The float-float anchors of 32 chunks are made at once, a
// chunk a lane, and kept in shared memory (anchors: the 32 of chunks 32 group ..), instead
// of by every lane for every chunk in both passes.  All lanes take part; those past the
// ray's end get a sample outside the cube, to be ignored.
__device__ __forceinline__ LaneSample lane_sample(const RaySetup& r, int c, int lane, float3 e32, const VolDev& v,
                                                  SampleAnchor* anchors, int& group) {
    if (c >> 5 != group) {
        group = c >> 5;
        __syncwarp();
        sample_anchor(r, r.k0 + 32 * (32 * group + lane), v, anchors[lane]);
        __syncwarp();
    }
    const SampleAnchor A = anchors[c & 31];
    const float fl = (float)lane;
    const float gx = fmaf(fl, e32.x, A.gx), gy = fmaf(fl, e32.y, A.gy), gz = fmaf(fl, e32.z, A.gz);
    const float invB = 1.0f / (float)v.B;
    LaneSample s;
    s.bx = min(max(A.bx + (int)floorf((gx - 0.5f) * invB), 0), v.nbx - 1);
    s.by = min(max(A.by + (int)floorf((gy - 0.5f) * invB), 0), v.nby - 1);
    s.bz = min(max(A.bz + (int)floorf((gz - 0.5f) * invB), 0), v.nbz - 1);
    s.gx = gx - (float)((s.bx - A.bx) << v.log2B);
    s.gy = gy - (float)((s.by - A.by) << v.log2B);
    s.gz = gz - (float)((s.bz - A.bz) << v.log2B);
    // a cube in core: brick b is slot b
    s.base = (long long)((s.bz * v.nby + s.by) * v.nbx + s.bx) * v.slot_elems;
    return s;
}

template <typename T, int MODE, bool FAST>
__global__ void __launch_bounds__(kAdjThreads, 5)
k_adjoint(const __grid_constant__ AdjParams P) {
    constexpr unsigned int FULL = 0xffffffffu;
    // dynamic, by the size of the table: the table, channel-major, and a histogram per warp
    extern __shared__ __align__(16) float s_dyn[];
    constexpr int S = FAST ? kAdjTF : 0, BR = FAST ? kFastBrick : 0;
    const int ntf = P.tf.n, sd = stride<S>(ntf);
    const Anchor slot0{0.f, 0.f, 0.f, 0};  // fetches from the slot's first voxel
    float* s_tf = s_dyn;
    __shared__ RaySetup s_ray[kAdjWarps][32];
    __shared__ SampleAnchor s_anchor[kAdjWarps][32];
    __shared__ float2 s_keep[kAdjWarps][MODE == VR_COMPOSITE ? kAdjKeep * 32 : 1];
    for (int i = threadIdx.x; i < ntf; i += blockDim.x) {
        const float4 t = P.tf.tab[i];
        s_tf[i] = t.x;
        s_tf[sd + i] = t.y;
        s_tf[2 * sd + i] = t.z;
        s_tf[3 * sd + i] = t.w;
    }
    if (MODE == VR_COMPOSITE)
        for (int i = threadIdx.x; i < 2 * kAdjWarps * sd; i += blockDim.x) s_dyn[4 * sd + i] = 0.f;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2* hist = reinterpret_cast<float2*>(s_dyn + 4 * sd) + warp * sd;
    float4* g_tf = P.tf_partials + (size_t)(blockIdx.x * kAdjWarps + warp) * ntf;  // this warp's gradient
    float2* keep = s_keep[warp];
    SampleAnchor* anchors = s_anchor[warp];
    const int tiles_per_cam = P.tiles_x * P.tiles_y;
    const int total = tiles_per_cam * P.ncams;
    const T* __restrict__ pool = static_cast<const T*>(P.vol.pool);
    const float ert = P.ert;

    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(P.work, 1);
        item = __shfl_sync(FULL, item, 0);
        if (item >= total) break;
        const int cam = item / tiles_per_cam;
        const int tile = item - cam * tiles_per_cam;
        const int ty = tile / P.tiles_x, tx = tile - ty * P.tiles_x;
        {  // this lane's ray of the tile
            const int px = tx * kTileW + (lane % kTileW);
            const int py = ty * kTileH + (lane / kTileW);
            bool ok = px < P.width && py < P.height;
            Ray r;
            float4 gI = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ok) {
                gI = P.dimg[((long long)cam * P.height + py) * P.width + px];
                ok = (gI.x != 0.f || gI.y != 0.f || gI.z != 0.f || gI.w != 0.f) &&
                     make_ray(P.cams[cam], px, py, P.vol, ff{P.step_hi, P.step_lo}, r);
            }
            RaySetup& rs = s_ray[warp][lane];
            if (ok) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    rs.o_hi[a] = r.o[a].hi;
                    rs.o_lo[a] = r.o[a].lo;
                    rs.e_hi[a] = r.e[a].hi;
                    rs.e_lo[a] = r.e[a].lo;
                }
                rs.g = gI;
            }
            rs.k0 = ok ? r.k0 : 0;
            rs.k1 = ok ? r.k1 : 0;
        }
        __syncwarp();
        unsigned int pending = __ballot_sync(FULL, s_ray[warp][lane].k1 > s_ray[warp][lane].k0);
        while (pending) {
            const int who = __ffs(pending) - 1;
            pending &= pending - 1;
            const RaySetup r = s_ray[warp][who];
            const float3 e32 = make_float3(r.e_hi[0], r.e_hi[1], r.e_hi[2]);
            const float4 gI = r.g;
            int group = -1;

            if (MODE == VR_MIP) {
                unsigned int best = ord_enc_f(-INFINITY);
                float m = -INFINITY;
                int kmax = -1;
                for (int k = r.k0; k < r.k1; k += 32) {
                    const bool act = k + lane < r.k1;
                    float v = -INFINITY;
                    const LaneSample ls = lane_sample(r, (k - r.k0) >> 5, lane, e32, P.vol, anchors, group);
                    if (act) {
                        v = fetch_near<T, BR>(pool + ls.base, P.vol, slot0, ls.gx, ls.gy, ls.gz);
                    }
                    const unsigned int e = act ? ord_enc_f(v) : 0u;
                    const unsigned int cmax = __reduce_max_sync(FULL, e);
                    if (cmax > best) {  // strictly greater: the first maximal sample is kept
                        best = cmax;
                        const int src = __ffs(__ballot_sync(FULL, act && e == cmax)) - 1;
                        m = __shfl_sync(FULL, v, src);
                        kmax = k + src;
                    }
                }
                if (kmax < 0) continue;
                if (lane == 0) {
                    const TFGrad t = tf_eval<S>(s_tf, ntf, P.tf.vmin, P.tf.inv_range, m);
                    add_tf(g_tf, t, gI);
                    if (P.dvol) {
                        SampleAnchor ls;
                        sample_anchor(r, kmax, P.vol, ls);
                        const float dv = gI.x * t.slope.x + gI.y * t.slope.y + gI.z * t.slope.z + gI.w * t.slope.w;
                        scatter_voxels(P.dvol, P.vol, ls.bx, ls.by, ls.bz, ls.gx, ls.gy, ls.gz, dv);
                    }
                }
                continue;
            }

            // ---- composite, forward: transmittance checkpoints per chunk, termination by ballot
            int nch = 0, n_last = 0;
            float ck0 = 0.f, ck[(kAdjMaxChunks - 1) / 32];  // chunks lane, 32 + lane, ...
            {
                float Tr = 1.f;
                bool overflow = false;
                for (int k = r.k0; k < r.k1; k += 32) {
                    if (nch == kAdjMaxChunks) {
                        overflow = true;
                        break;
                    }
                    if (lane == (nch & 31)) {
                        if (nch < 32) ck0 = Tr;
                        else ck[(nch >> 5) - 1] = Tr;
                    }
                    const int n = min(32, r.k1 - k);
                    const bool act = lane < n;
                    float q = 1.f, v = 0.f;
                    const LaneSample ls = lane_sample(r, nch, lane, e32, P.vol, anchors, group);
                    if (act) {
                        v = fetch_near<T, BR>(pool + ls.base, P.vol, slot0, ls.gx, ls.gy, ls.gz);
                        q = 1.f - tf_alpha<S>(s_tf, ntf, P.tf.vmin, P.tf.inv_range, v);
                    }
                    float incl = q;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const float t = __shfl_up_sync(FULL, incl, off);
                        if (lane >= off) incl *= t;
                    }
                    if (nch < kAdjKeep) keep[nch * 32 + lane] = make_float2(v, incl);
                    ++nch;
                    const float Tout = Tr * incl;
                    const unsigned int done = __ballot_sync(FULL, act && 1.f - Tout >= ert);
                    if (done) {
                        n_last = __ffs(done);
                        break;
                    }
                    n_last = n;
                    Tr = __shfl_sync(FULL, Tout, n - 1);
                }
                if (overflow) {
                    if (lane == 0) atomicExch(P.status, kDevTooManySegments);
                    continue;
                }
            }
            __syncwarp();
            const bool collect = fabsf(gI.x) + fabsf(gI.y) + fabsf(gI.z) < INFINITY;  // NaN: false
            int e_lo = ntf, e_hi = 0;  // entries touched by this lane's samples
            // ---- reverse: chunks back to front, suffix "over" scan within a chunk
            float Rc = 0.f, Pc = 1.f;
            for (int c = nch - 1; c >= 0; --c) {
                const int n = c == nch - 1 ? n_last : 32;
                const bool act = lane < n;
                const float ckT = __shfl_sync(FULL, c < 32 ? ck0 : ck[(c >> 5) - 1], c & 31);
                TFGrad t;
                t.i = -1;
                LaneSample ls;
                if (c >= kAdjKeep || P.dvol) ls = lane_sample(r, c, lane, e32, P.vol, anchors, group);
                float a = 0.f, s = 0.f, incl = 1.f;
                if (act) {
                    float v;
                    if (c < kAdjKeep) {
                        const float2 kv = keep[c * 32 + lane];
                        v = kv.x;
                        incl = kv.y;
                    } else {
                        v = fetch_near<T, BR>(pool + ls.base, P.vol, slot0, ls.gx, ls.gy, ls.gz);
                    }
                    t = tf_eval<S>(s_tf, ntf, P.tf.vmin, P.tf.inv_range, v);
                    a = t.rgba.w;
                    s = gI.x * t.rgba.x + gI.y * t.rgba.y + gI.z * t.rgba.z;
                }
                const float q = 1.f - a;
                if (c >= kAdjKeep) {
                    incl = q;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const float u = __shfl_up_sync(FULL, incl, off);
                        if (lane >= off) incl *= u;
                    }
                }
                float excl = __shfl_up_sync(FULL, incl, 1);
                if (lane == 0) excl = 1.f;
                const float Tin = ckT * excl;
                // inclusive suffix of (A, B) = (a s, 1 - a) under (A1, B1) o (A2, B2) = (A1 + B1 A2, B1 B2)
                float A = a * s, Bq = q;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const float oa = __shfl_down_sync(FULL, A, off), ob = __shfl_down_sync(FULL, Bq, off);
                    if (lane + off < 32) {
                        A = fmaf(Bq, oa, A);
                        Bq *= ob;
                    }
                }
                // behind sample `lane`: the suffix after it, then the chunks behind this one
                float xa = __shfl_down_sync(FULL, A, 1), xb = __shfl_down_sync(FULL, Bq, 1);
                if (lane == 31) {
                    xa = 0.f;
                    xb = 1.f;
                }
                const float R = fmaf(xb, Rc, xa), Pt = xb * Pc;
                // carry for the chunk in front: this whole chunk over the carry
                const float ha = __shfl_sync(FULL, A, 0), hb = __shfl_sync(FULL, Bq, 0);
                Rc = fmaf(hb, Rc, ha);
                Pc *= hb;
                const float wk = Tin * a;
                const float ga = gI.w * Tin * Pt + Tin * (s - R);
                if (collect) {
                    collect_sample(hist, t, act, lane, wk, ga);
                    if (act) {
                        e_lo = min(e_lo, t.i);
                        e_hi = max(e_hi, t.i + 1);
                    }
                } else if (act) {
                    add_tf(g_tf, t, make_float4(gI.x * wk, gI.y * wk, gI.z * wk, ga));
                }
                if (act) {
                    if (P.dvol) {
                        const float dv = wk * (gI.x * t.slope.x + gI.y * t.slope.y + gI.z * t.slope.z) + ga * t.slope.w;
                        scatter_voxels(P.dvol, P.vol, ls.bx, ls.by, ls.bz, ls.gx, ls.gy, ls.gz, dv);
                    }
                }
            }
            if (collect) {  // the histogram, over the entries touched, to the warp's partial
                e_lo = __reduce_min_sync(FULL, e_lo);
                e_hi = __reduce_max_sync(FULL, e_hi);
                for (int e = e_lo + lane; e <= e_hi; e += 32) {
                    const float2 h = hist[e];
                    if (h.x != 0.f || h.y != 0.f) {
                        hist[e] = make_float2(0.f, 0.f);
                        add_entry(g_tf + e, 1.f, make_float4(gI.x * h.x, gI.y * h.x, gI.z * h.x, h.y));
                    }
                }
            }
            __syncwarp();
        }
        __syncwarp();  // the tile's ray set-ups are read before the next tile overwrites them
    }
}

// Final reduction of the table gradients of the warps, nblocks x kAdjWarps x nval: a block's
// in FP32, over the blocks in FP64 (the only FP64 arithmetic on the gradient path; all rows in
// FP64 took 58 us for 3040 x 1024).
// A block per 32 values, its warps on interleaved blocks' rows (a thread a value, serial over
// the rows, took 121 us for 760 x 1024: four blocks in all).
constexpr int kReduceWarps = 32;
__global__ void __launch_bounds__(kReduceWarps * 32)
k_tfgrad_reduce(const float* __restrict__ partials, int nblocks, int nval, float* __restrict__ out) {
    __shared__ double s_acc[kReduceWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    double acc = 0.0;
    if (i < nval) {
#pragma unroll 4
        for (int b = warp; b < nblocks; b += kReduceWarps) {
            const float* p = partials + (size_t)b * kAdjWarps * nval + i;
            float v = p[0];
#pragma unroll
            for (int w = 1; w < kAdjWarps; ++w) v += p[(size_t)w * nval];
            acc += (double)v;
        }
    }
    s_acc[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && i < nval) {
        for (int w = 1; w < kReduceWarps; ++w) acc += s_acc[w][lane];
        out[i] = (float)acc;
    }
}

template <typename T>
void* adj_t(int mode, bool fast) {
    if (mode == VR_MIP)
        return fast ? reinterpret_cast<void*>(&k_adjoint<T, VR_MIP, true>)
                    : reinterpret_cast<void*>(&k_adjoint<T, VR_MIP, false>);
    return fast ? reinterpret_cast<void*>(&k_adjoint<T, VR_COMPOSITE, true>)
                : reinterpret_cast<void*>(&k_adjoint<T, VR_COMPOSITE, false>);
}

// The kernel for p and its dynamic shared memory: the table, and a histogram a warp.
void* adj_pick(const AdjParams& p, vr_dtype dt, size_t& smem) {
    const bool fast = p.vol.B == kFastBrick && p.tf.n <= kAdjTF;
    smem = (size_t)(fast ? kAdjTF : p.tf.n) * sizeof(float) * (4 + (p.mode == VR_COMPOSITE ? 2 * kAdjWarps : 0));
    void* f = dt == VR_F32   ? adj_t<float>(p.mode, fast)
              : dt == VR_F16 ? adj_t<__half>(p.mode, fast)
                             : adj_t<__nv_bfloat16>(p.mode, fast);
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess ? f : nullptr;
}

}  // namespace

int adjoint_warps() { return kAdjWarps; }

int adjoint_blocks_per_sm(const AdjParams& p, vr_dtype dt) {
    size_t smem;
    void* f = adj_pick(p, dt, smem);
    int n = 0;
    if (!f || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, kAdjThreads, smem) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

cudaError_t launch_adjoint(const AdjParams& p, vr_dtype dt, int grid, cudaStream_t s) {
    size_t smem;
    void* f = adj_pick(p, dt, smem);
    if (!f) return cudaGetLastError();
    void* args[] = {const_cast<AdjParams*>(&p)};
    return cudaLaunchKernel(f, dim3(grid), dim3(kAdjThreads), args, smem, s);
}

cudaError_t launch_tfgrad_reduce(const float4* partials, int nblocks, int ntf, float* out, cudaStream_t s) {
    const int nval = 4 * ntf;
    k_tfgrad_reduce<<<(nval + 31) / 32, kReduceWarps * 32, 0, s>>>(reinterpret_cast<const float*>(partials), nblocks,
                                                                   nval, out);
    return cudaGetLastError();
}

}  // namespace vr
