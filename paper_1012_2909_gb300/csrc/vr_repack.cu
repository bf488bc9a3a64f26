// Repack of a linear float32 cube (x fastest) into the ghosted brick store, with
// conversion to the storage type (round to nearest even), the store's copy shifted by
// one element when it is kept, and the per-brick minimum / maximum of the stored
// values (ghost layer included), which bound every trilinear sample taken inside the
// brick.
#include <algorithm>

#include "vr_internal.cuh"

namespace vr {

namespace {

__device__ __forceinline__ unsigned int ord_enc(float f) {
    const unsigned int u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

template <typename T> __device__ __forceinline__ T to_store(float f);
template <> __device__ __forceinline__ float to_store<float>(float f) { return f; }
template <> __device__ __forceinline__ __half to_store<__half>(float f) { return __float2half_rn(f); }
template <> __device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(float f) {
    return __float2bfloat16_rn(f);
}
template <typename T> __device__ __forceinline__ float widen(T v);
template <> __device__ __forceinline__ float widen<float>(float v) { return v; }
template <> __device__ __forceinline__ float widen<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float widen<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}

__device__ __forceinline__ unsigned int bits(__half v) { return __half_as_ushort(v); }
__device__ __forceinline__ unsigned int bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }

__device__ __forceinline__ __half2 pack2(__half a, __half b) { return __halves2half2(a, b); }
__device__ __forceinline__ __nv_bfloat162 pack2(__nv_bfloat16 a, __nv_bfloat16 b) { return __halves2bfloat162(a, b); }

// Running minimum and maximum of the stored values, a word at a time (NaN ignored, as fminf).
template <typename T> struct Range {
    decltype(pack2(T(), T())) mn, mx;
    __device__ __forceinline__ Range() : mn(pack2(to_store<T>(INFINITY), to_store<T>(INFINITY))),
                                         mx(pack2(to_store<T>(-INFINITY), to_store<T>(-INFINITY))) {}
    __device__ __forceinline__ void add(T a, T b) {
        const auto p = pack2(a, b);
        mn = __hmin2(mn, p);
        mx = __hmax2(mx, p);
    }
    __device__ __forceinline__ float least() const { return fminf(widen<T>(mn.x), widen<T>(mn.y)); }
    __device__ __forceinline__ float most() const { return fmaxf(widen<T>(mx.x), widen<T>(mx.y)); }
};
template <> struct Range<float> {
    float mn = INFINITY, mx = -INFINITY;
    __device__ __forceinline__ void add(float a) {
        mn = fminf(mn, a);
        mx = fmaxf(mx, a);
    }
    __device__ __forceinline__ float least() const { return mn; }
    __device__ __forceinline__ float most() const { return mx; }
};

// grid: (nbx * nby, rows, layers of bricks); block: row_words x `lines` threads, rounded
// up to whole warps.  Block (b, lz, l) writes plane lz of the slot of brick (b % nbx,
// b / nbx, bz0 + l), and of its shifted copy.
//
// Bound by DRAM: 4 bytes read and sizeof(T) (twice, with the copy) written per voxel.
// A thread makes one 32-bit word of a row, two 16-bit voxels or one float, and goes
// down the plane in that column, so its clamped source columns are found once and a
// word costs few instructions.  Loads and stores of a warp are consecutive words
// whatever the source's alignment (a row starts one voxel before the brick, so wider
// loads would never be aligned); kRepackUnroll rows' loads are in flight, and the rows of
// threads in a block are chosen so that its trips end near the slot's last row (blocks of
// kRepackThreads whatever the brick went far past it in small ones: 512^3 FP16 in bricks of
// 8, 16, 32, 64 voxels 7.9, 1.86, 0.51, 0.29 ms a load, now 1.36, 0.49, 0.38, 0.26).  The copy's
// word (voxels x + 1, x + 2) is made from the same registers and the next lane's, in
// place of a device-to-device copy at a 2-byte offset afterwards.  Neighbouring bricks
// read the ghost planes and row ends again, so the loads go through L2 as usual: with
// streaming loads the survey cube (1024 x 1024 x 2048, 16-bit with the copy: 18.0 GB)
// read 10.9 GB instead of 8.6.  That cube in 3.09 ms, 5.82 TB/s; before, 16 launches
// with an element a thread took 5.2 ms and the offset copy came on top (load and first
// frame 15.4 -> 10.6 ms).  kRepackUnroll = 2, 8: the same, +10 %.
constexpr int kRepackUnroll = 4;
constexpr int kRepackThreads = 288;  // threads of a block, about

template <typename T, bool COPY>
__global__ void __launch_bounds__(512)
k_repack(const float* __restrict__ src, long long src_z0, int bz0, VolDev v, T* __restrict__ pool,
         T* __restrict__ pool1, unsigned int* __restrict__ minmax, int nbricks, int row_words, int lines) {
    constexpr int VPW = 4 / (int)sizeof(T);  // voxels per word
    constexpr int U = kRepackUnroll;
    const int bx = blockIdx.x % v.nbx, by = blockIdx.x / v.nbx, bz = bz0 + blockIdx.z;
    const int lz = blockIdx.y, lane = threadIdx.x & 31;
    const int bid = (bz * v.nby + by) * v.nbx + bx;
    const long long base = (long long)v.table[bid] * v.slot_elems + (long long)lz * v.rows * v.pitch;
    unsigned int* dst = reinterpret_cast<unsigned int*>(pool + base);
    unsigned int* dst1 = COPY ? reinterpret_cast<unsigned int*>(pool1 + base) : nullptr;
    const int gz = min(max(bz * v.B + lz - 1, 0), v.nz - 1);
    const float* plane = src + (long long)(gz - src_z0) * v.ny * v.nx;
    // this thread's line of the block's `lines` rows and its word of the row; a row is a
    // whole number of voxel words and padding words (rows is even, padding columns are 0)
    const int line = threadIdx.x / row_words, word = threadIdx.x - line * row_words;
    const int lx = word * VPW, x0 = bx * v.B - 1 + lx, y0 = by * v.B - 1;
    const bool mine = line < lines, real = mine && lx < v.rows;
    const int c0 = min(max(x0, 0), v.nx - 1), c1 = min(max(x0 + 1, 0), v.nx - 1);
    // lane 31 loads the voxel after its word itself
    const bool third = COPY && lane == 31 && lx + VPW < v.rows;
    const int c2 = min(max(x0 + 2, 0), v.nx - 1);
    Range<T> range;
    for (int ly0 = line; ly0 - line < v.rows; ly0 += lines * U) {  // the same trips for every lane
        float f[U][VPW], f2[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            // rows past the slot's last one repeat it
            const int ly = min(ly0 + u * lines, v.rows - 1);
            const float* row = plane + (long long)min(max(y0 + ly, 0), v.ny - 1) * v.nx;
            f[u][0] = real ? __ldg(row + c0) : 0.f;
            if (VPW == 2) f[u][VPW - 1] = real ? __ldg(row + c1) : 0.f;
            f2[u] = third ? __ldg(row + c2) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ly = ly0 + u * lines;
            const bool put = mine && ly < v.rows;
            if constexpr (VPW == 2) {
                const T a = to_store<T>(f[u][0]), b = to_store<T>(f[u][1]);
                if (real) range.add(a, b);  // a repeated row adds nothing new
                const unsigned int lo = bits(a), hi = bits(b);
                if (put) dst[ly * row_words + word] = lo | (hi << 16);
                if (COPY) {
                    const unsigned int next = __shfl_down_sync(0xffffffffu, lo, 1);
                    const unsigned int x2 = lane == 31 ? bits(to_store<T>(f2[u])) : next;
                    if (put) dst1[ly * row_words + word] = hi | (lx + VPW < v.pitch ? x2 << 16 : 0u);
                }
            } else {
                if (real) range.add(f[u][0]);
                if (put) dst[ly * row_words + word] = __float_as_uint(f[u][0]);
            }
        }
    }
    float mn = range.least(), mx = range.most();
    for (int off = 16; off > 0; off >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    if (lane == 0) {
        atomicMin(&minmax[bid], ord_enc(mn));
        atomicMax(&minmax[nbricks + bid], ord_enc(mx));
    }
}

template <typename T>
cudaError_t repack_t(const float* src, long long src_z0, int bz0, int nlayers, const VolDev& v, void* pool,
                     void* pool1, unsigned int* minmax, cudaStream_t s) {
    const int nbricks = v.nbx * v.nby * v.nbz;
    const int row_words = v.pitch * (int)sizeof(T) / 4;  // 8 .. 260
    // the most rows of threads that fit, in as many trips, spread evenly over the trips: a trip
    // goes past the slot's rows by fewer than kRepackUnroll rows a trip
    const int most = std::max(1, kRepackThreads / row_words), trips = (v.rows - 1) / (kRepackUnroll * most) + 1;
    const int lines = (v.rows - 1) / (kRepackUnroll * trips) + 1;
    const int block = (row_words * lines + 31) / 32 * 32;
    for (int l = 0; l < nlayers; l += 65535) {  // a grid's z limit
        const dim3 grid(v.nbx * v.nby, v.rows, std::min(nlayers - l, 65535));
        if (sizeof(T) == 2 && pool1)
            k_repack<T, sizeof(T) == 2><<<grid, block, 0, s>>>(src, src_z0, bz0 + l, v, static_cast<T*>(pool),
                                                              static_cast<T*>(pool1), minmax, nbricks, row_words,
                                                              lines);
        else
            k_repack<T, false><<<grid, block, 0, s>>>(src, src_z0, bz0 + l, v, static_cast<T*>(pool), nullptr, minmax,
                                                      nbricks, row_words, lines);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_repack(const float* src, long long src_z0, int bz0, int nlayers, const VolDev& v, vr_dtype dt,
                          void* pool, void* pool1, unsigned int* minmax, cudaStream_t s) {
    if (dt == VR_F32) return repack_t<float>(src, src_z0, bz0, nlayers, v, pool, pool1, minmax, s);
    if (dt == VR_F16) return repack_t<__half>(src, src_z0, bz0, nlayers, v, pool, pool1, minmax, s);
    return repack_t<__nv_bfloat16>(src, src_z0, bz0, nlayers, v, pool, pool1, minmax, s);
}

}  // namespace vr
