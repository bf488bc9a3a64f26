// Image-order ray marcher: one thread per ray, one warp per 8 x 4 pixel tile,
// tiles handed out by a persistent scheduler (one atomic counter per launch).
//
// Per ray (the discretisation of include/vr.h, vr_render): float-float ray
// set-up and box interval; brick-by-brick traversal; inside a brick the samples
// are re-anchored in float-float every kAnchorSpan samples and stepped in FP32
// relative to the anchor's voxel, so each position is within 13 u (u = 2^-24)
// voxels of exact at the 0.5-voxel step; trilinear fetch from the ghosted brick
// (x-neighbour pairs with one load each when the store's shifted copy is kept);
// transfer-function lookup from shared memory; front-to-back "over" with early
// termination, or maximum-intensity projection.
#include "vr_device.cuh"

namespace vr {

namespace {

constexpr int kSegCap = 1 << 20;  // a brick segment is cut only where the ray leaves the brick
// Samples fetched together per step.  The marcher waits on its gathers, so more
// loads in flight beat more resident warps: with the register count left free
// (launch bound 256 x 2: at most 128 registers, two CTAs per SM), 4 measured fastest for single loads (3: +2 %, 6: +2 %,
// 2: +9 %; capping registers at 64 for more warps cost 30 %), and 6 with the
// paired loads, which need fewer registers per sample (4: +7 %, 3: +13 %,
// 8: +15 %; survey composite over the orbit).
constexpr int kMarchUnroll = 4;
constexpr int kMarchUnrollPaired = 6;

// Tables of up to kMarchTF entries are kept with the rises of their intervals, and the
// default brick edge is compiled in (kFormFast); other tables and edges take the general form.
//
// Bound by L1 wavefronts on sparse views (profile: 72-79 %) and by the instructions of 16
// warps an SM on dense ones: a sample took about 130 warp instructions on the small FP32
// view, lanes that wait for their neighbours included.  With constant slot offsets, no
// clamps, rises and a termination without branches it takes 111: 128^3 FP32 at 512 x 512
// 89.6 -> 77.1 us, 1721 x 1721 x 1025 FP32 at 3000 x 3000 3.27 -> 2.83 ms, survey FP16
// 0.440 -> 0.412 ms, the same images bit for bit.  (The times of a composite move with the seed
// of the cube's noise by some 15 %: the two figures of a comparison share a seed and a run, those
// of different comparisons here need not.)
constexpr int kMarchTF = 256;

// Asks L2 for what a sample some way ahead reads (both slabs; the offset is kept in the
// slot, so past the brick's end this asks in vain).  A sparse view's rays share few cache
// lines and a third of their requests go to DRAM, longer than six samples in flight cover:
// survey FP16 0.439 -> 0.405 ms, and nothing lost where the lines are shared (1721 x 1721 x
// 1025 at 3000 x 3000 3.136 and 3.139 ms).  30 samples ahead, four rows, or into L1: the same;
// two or three positions a span: 0.414 to 0.424 ms.  (In the layered composite it cost 4-8 %.)
constexpr float kPrefetchAhead = 18.f;  // samples, from a span's anchor

template <typename T, int BR, bool PAIRED>
__device__ __forceinline__ void prefetch_near(const T* slot, const T* slot1, const VolDev& v, const Anchor& A,
                                              float3 e) {
    float fx, fy, fz;
    const int o = near_offset<T, BR>(v, A, fmaf(kPrefetchAhead, e.x, A.qx), fmaf(kPrefetchAhead, e.y, A.qy),
                                     fmaf(kPrefetchAhead, e.z, A.qz), fx, fy, fz);
    const T* p = (PAIRED && (o & 1) ? slot1 : slot) + o;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p + SlotGeom<T, BR>::slab(v)));
}

template <typename T, int MODE, bool PAIRED, MarchForm FORM>
__global__ void __launch_bounds__(256, 2)
k_march(const __grid_constant__ MarchParams P) {
    constexpr bool FAST = FORM == kFormFast;
    constexpr int U = PAIRED ? kMarchUnrollPaired : kMarchUnroll;
    constexpr int BR = FAST ? kFastBrick : 0, S = FAST ? kMarchTF : kMaxTF;
    __shared__ float s_tf[(FAST ? 8 : 4) * S];
    fill_table<S, FAST>(s_tf, P.tf);
    __syncthreads();

    const int lane = threadIdx.x & 31;
    const int tiles_per_cam = P.tiles_x * P.tiles_y;
    const int total = tiles_per_cam * P.ncams;
    const T* __restrict__ pool = static_cast<const T*>(P.vol.pool);
    const T* __restrict__ pool1 = static_cast<const T*>(P.vol.pool1);
    const float ert = P.ert;
    unsigned long long my_samples = 0;

    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(P.work, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= total) break;
        const int cam = item / tiles_per_cam;
        const int tile = item - cam * tiles_per_cam;
        const int ty = tile / P.tiles_x, tx = tile - ty * P.tiles_x;
        const int px = tx * P.tile_w + (lane % P.tile_w);
        const int py = ty * P.tile_h + (lane / P.tile_w);
        if (px >= P.width || py >= P.height) continue;  // ragged edge tile; the lane
                                                        // rejoins at the next shuffle
        Ray r;
        const bool hit = make_ray(P.cams[cam], px, py, P.vol, ff{P.step_hi, P.step_lo}, r);
        float c0 = 0.f, c1 = 0.f, c2 = 0.f, Tr = 1.f, m_ = -INFINITY;
        if (hit) {
            const float3 e32 = make_float3(r.e[0].hi, r.e[1].hi, r.e[2].hi);
            int k = r.k0;
            bool done = false;
            while (k < r.k1 && !done) {
                Seg s;
                seg_begin(r, k, P.vol, e32, kSegCap, s);
                if (MODE == VR_COMPOSITE && brick_transparent(P.vol, P.tf, s.brick)) {
                    k += s.n;  // opacity 0 throughout: (C, T) would not change
                    continue;
                }
                const T* slot = pool + s.base;
                const T* slot1 = PAIRED ? pool1 + s.base : nullptr;
                int j = 0, executed = 0;  // samples of this segment done, and up to the termination
                while (j < s.n && !done) {
                    // sub-anchor at sample k + j; U samples fetched together (more loads
                    // in flight), then composited in order; a fetch past the span
                    // repeats its last sample
                    const Anchor A = anchor_at(r, k + j, P.vol, s);
                    const int m = min(kAnchorSpan, s.n - j);
                    prefetch_near<T, BR, PAIRED>(slot, slot1, P.vol, A, e32);
                    for (int i = 0; i < m && !done; i += U) {
                        float v[U];
#pragma unroll
                        for (int q = 0; q < U; ++q) {
                            const float fi = (float)min(i + q, m - 1);
                            const float qx = fmaf(fi, e32.x, A.qx), qy = fmaf(fi, e32.y, A.qy),
                                        qz = fmaf(fi, e32.z, A.qz);
                            v[q] = PAIRED ? fetch_near_pair<T, BR>(slot, slot1, P.vol, A, qx, qy, qz)
                                          : fetch_near<T, BR>(slot, P.vol, A, qx, qy, qz);
                        }
#pragma unroll
                        for (int q = 0; q < U; ++q) {
                            if (MODE == VR_MIP) {
                                m_ = fmaxf(m_, v[q]);  // a repeated sample changes nothing
                            } else {
                                // past the span or the termination: opacity 0, nothing changes
                                const bool on = i + q < m && !done;
                                if (FORM == kFormGuarded && !on) break;
                                const float4 c = tf_lookup<S, FAST>(s_tf, P.tf.n, P.tf.vmin, P.tf.inv_range, v[q]);
                                const float a = on ? c.w : 0.f;
                                const float w = Tr * a;
                                c0 = fmaf(w, c.x, c0);
                                c1 = fmaf(w, c.y, c1);
                                c2 = fmaf(w, c.z, c2);
                                Tr = Tr * (1.f - a);
                                if (on && 1.f - Tr >= ert) {
                                    executed = j + i + q + 1;
                                    done = true;
                                }
                            }
                        }
                    }
                    j += m;
                }
                my_samples += (unsigned long long)(done ? executed : s.n);
                k += s.n;
            }
        }
        const long long pix = ((long long)cam * P.height + py) * P.width + px;
        if (MODE == VR_MIP) {
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            if (m_ > -INFINITY) o = tf_lookup<S, FAST>(s_tf, P.tf.n, P.tf.vmin, P.tf.inv_range, m_);
            P.out_rgba[pix] = o;
            if (P.out_max) P.out_max[pix] = m_;
        } else {
            P.out_rgba[pix] = make_float4(c0, c1, c2, 1.f - Tr);
        }
    }
    if (P.samples) {
        unsigned long long s = my_samples;
        for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
        if (lane == 0 && s) atomicAdd(P.samples, s);
    }
}

template <typename T, int MODE, bool PAIRED>
void* kernel_ptr(MarchForm form) {
    if (MODE == VR_COMPOSITE && form == kFormGuarded)
        return reinterpret_cast<void*>(&k_march<T, VR_COMPOSITE, PAIRED, kFormGuarded>);
    return form == kFormFast ? reinterpret_cast<void*>(&k_march<T, MODE, PAIRED, kFormFast>)
                             : reinterpret_cast<void*>(&k_march<T, MODE, PAIRED, kFormGeneral>);
}

// Paired loads only for the composite: its rays stop in a front shell that stays in
// the caches, where halving the gathers pays (survey frame -11 %).  MIP rays cross the
// whole cube, and reading both copies there measured 34 % slower.
template <typename T>
void* pick_mode(int mode, bool paired, MarchForm form) {
    if (mode == VR_MIP) return kernel_ptr<T, VR_MIP, false>(form);
    if constexpr (sizeof(T) == 2) {
        if (paired) return kernel_ptr<T, VR_COMPOSITE, true>(form);
    }
    return kernel_ptr<T, VR_COMPOSITE, false>(form);
}

void* pick(vr_dtype dt, const MarchParams& p) {
    const bool paired = p.vol.pool1 != nullptr;
    const MarchForm form = march_form(p, kMarchTF);
    if (dt == VR_F32) return pick_mode<float>(p.mode, paired, form);
    if (dt == VR_F16) return pick_mode<__half>(p.mode, paired, form);
    return pick_mode<__nv_bfloat16>(p.mode, paired, form);
}

}  // namespace

int march_blocks_per_sm(const MarchParams& p, vr_dtype dt, int block) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pick(dt, p), block, 0) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

cudaError_t launch_march(const MarchParams& p, vr_dtype dt, int grid, int block, cudaStream_t s) {
    void* args[] = {const_cast<MarchParams*>(&p)};
    return cudaLaunchKernel(pick(dt, p), dim3(grid), dim3(block), args, 0, s);
}

}  // namespace vr
