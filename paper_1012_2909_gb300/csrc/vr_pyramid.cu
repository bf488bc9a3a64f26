// Image pyramid of a render: the paper's high-resolution static renders are cut
// into tiles and shown at several zoom levels (Sec. 3); this is the render half
// of that path.  Level l+1 halves level l (rounding up) and its pixel is the
// mean of the in-level pixels of its 2 x 2 block (premultiplied RGBA).
//
// One CTA owns a 32 x 32 tile of its input level and derives up to five levels from it
// (tiles are aligned to 32 input pixels, so the children of every pixel of a level stay
// inside the CTA), writing every level once.  The host repeats the pass on the last level
// written until 1 x 1 is reached; each pass reads 1/1024 of the previous input.  In a
// tiled layout a first launch zeroes the pixels of edge tiles that lie past their level.
#include <algorithm>

#include "vr_internal.cuh"

namespace vr {

namespace {

constexpr int kPyrTile = 32;
constexpr int kPyrPassLevels = 5;  // 32 -> 16 -> 8 -> 4 -> 2 -> 1
constexpr int kPyrThreads = 256;

struct PyrLevel {
    int w, h;
    long long off;  // float4 offset of the level in the output
};

struct PyrParams {
    const float4* in;
    int in_w, in_h, in_tlog2;  // input level; tile log2, -1 = row-major
    float4* out;
    int tlog2;                 // output layout, -1 = row-major
    int nlev;                  // levels written by this pass
    PyrLevel lev[kPyrPassLevels];
};

__device__ __forceinline__ long long pix_index(int x, int y, int w, int tlog2) {
    if (tlog2 < 0) return (long long)y * w + x;
    const int m = (1 << tlog2) - 1;
    const int tx = (w + m) >> tlog2;
    return (((long long)(y >> tlog2) * tx + (x >> tlog2)) << (2 * tlog2)) + ((y & m) << tlog2) + (x & m);
}

// Mean of the in-level pixels of a 2 x 2 block: load(i, j) is pixel (2 gx + i, 2 gy + j).
template <typename F>
__device__ __forceinline__ float4 block_mean(F load, int gx, int gy, int pw, int ph) {
    float4 v[4];
    bool in[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        in[k] = 2 * gx + (k & 1) < pw && 2 * gy + (k >> 1) < ph;
        v[k] = in[k] ? load(k & 1, k >> 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int n = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!in[k]) continue;
        acc.x += v[k].x;
        acc.y += v[k].y;
        acc.z += v[k].z;
        acc.w += v[k].w;
        ++n;
    }
    const float inv = n == 4 ? 0.25f : (n == 2 ? 0.5f : 1.f);
    return make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
}

// Bound by DRAM: 16 bytes read per input pixel and written per output pixel.  A thread
// makes one pixel of the first level straight from its four input pixels, so that all of
// the input's loads are in flight at once and the input does not pass through shared
// memory (4 KB a CTA instead of 20: eight CTAs an SM); the four small levels that follow
// are made there.  8000 x 8000 in 256 x 256 tiles: 0.335 ms
// (with a clear of the whole output) -> 0.231 ms, 5.9 TB/s.
__global__ void __launch_bounds__(kPyrThreads) k_pyramid(const __grid_constant__ PyrParams P) {
    constexpr int kHalf = kPyrTile / 2;
    static_assert(kPyrThreads == kHalf * kHalf, "a thread per pixel of the first level");
    __shared__ float4 buf_a[kHalf * kHalf];
    __shared__ float4 buf_b[(kHalf / 2) * (kHalf / 2)];
    const int bx = blockIdx.x, by = blockIdx.y;
    {
        const int x = threadIdx.x % kHalf, y = threadIdx.x / kHalf;
        const int gx = bx * kHalf + x, gy = by * kHalf + y;
        const PyrLevel L = P.lev[0];
        if (gx < L.w && gy < L.h) {
            const float4 r = block_mean(
                [&](int i, int j) { return __ldg(P.in + pix_index(2 * gx + i, 2 * gy + j, P.in_w, P.in_tlog2)); }, gx,
                gy, P.in_w, P.in_h);
            buf_a[threadIdx.x] = r;
            P.out[L.off + pix_index(gx, gy, L.w, P.tlog2)] = r;
        }
    }
    float4* src = buf_a;
    float4* dst = buf_b;
    int side = kHalf;
    for (int k = 1; k < P.nlev; ++k) {
        __syncthreads();
        const int half = side >> 1;
        const PyrLevel L = P.lev[k];
        if ((int)threadIdx.x < half * half) {
            const int x = threadIdx.x % half, y = threadIdx.x / half;
            const int gx = bx * half + x, gy = by * half + y;
            if (gx < L.w && gy < L.h) {
                const float4 r = block_mean([&](int i, int j) { return src[(2 * y + j) * side + 2 * x + i]; }, gx, gy,
                                            P.lev[k - 1].w, P.lev[k - 1].h);
                dst[threadIdx.x] = r;
                P.out[L.off + pix_index(gx, gy, L.w, P.tlog2)] = r;
            }
        }
        float4* t = src;
        src = dst;
        dst = t;
        side = half;
    }
}

// Zeroes the pixels of edge tiles past their level: per level the strip to the right of
// its rows, then the rows below it.  (Clearing the whole output first, 341 MB for
// 8000 x 8000, took 50 us; the padding in 256 x 256 tiles is 16 MB.)
constexpr int kPyrMaxLevels = 20;  // 2^20 pixels a side
struct PadParams {
    float4* out;
    int tlog2, nlev;
    PyrLevel lev[kPyrMaxLevels];
    long long end[kPyrMaxLevels];  // padding pixels of the levels up to and with this one
};

__global__ void __launch_bounds__(256) k_pyramid_pad(const __grid_constant__ PadParams P) {
    const long long total = P.end[P.nlev - 1], m = (1LL << P.tlog2) - 1;
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < total; i += gridDim.x * 256LL) {
        int l = 0;
        while (i >= P.end[l]) ++l;
        const PyrLevel L = P.lev[l];
        const long long k = i - (l ? P.end[l - 1] : 0);
        const long long pw = (L.w + m) & ~m, strip = pw - L.w;
        const bool right = k < strip * L.h;
        const int y = (int)(right ? k / strip : L.h + (k - strip * L.h) / pw);
        const int x = (int)(right ? L.w + k % strip : (k - strip * L.h) % pw);
        P.out[L.off + pix_index(x, y, L.w, P.tlog2)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

}  // namespace

// Level sizes and float4 offsets of levels 1.. for the layout (tlog2 < 0:
// row-major); returns the total float4 count.
long long pyramid_levels(int w, int h, int tlog2, std::vector<int>& ws, std::vector<int>& hs,
                         std::vector<long long>& offs) {
    ws.clear();
    hs.clear();
    offs.clear();
    long long total = 0;
    while (w > 1 || h > 1) {
        w = (w + 1) / 2;
        h = (h + 1) / 2;
        ws.push_back(w);
        hs.push_back(h);
        offs.push_back(total);
        if (tlog2 < 0) {
            total += (long long)w * h;
        } else {
            const long long t = 1LL << tlog2;
            total += ((w + t - 1) / t) * ((h + t - 1) / t) * t * t;
        }
    }
    return total;
}

cudaError_t launch_pyramid(const float4* in, int w, int h, int tlog2, float4* out, cudaStream_t s) {
    std::vector<int> ws, hs;
    std::vector<long long> offs;
    const long long total = pyramid_levels(w, h, tlog2, ws, hs, offs);
    if (ws.empty()) return cudaSuccess;
    if (tlog2 >= 0) {
        PadParams Q;
        Q.out = out;
        Q.tlog2 = tlog2;
        Q.nlev = (int)ws.size();
        long long pad = 0;
        for (size_t l = 0; l < ws.size(); ++l) {
            const long long next = l + 1 < ws.size() ? offs[l + 1] : total;
            pad += next - offs[l] - (long long)ws[l] * hs[l];
            Q.lev[l] = PyrLevel{ws[l], hs[l], offs[l]};
            Q.end[l] = pad;
        }
        if (pad > 0) {
            k_pyramid_pad<<<(int)std::min<long long>((pad + 255) / 256, 152 * 8), 256, 0, s>>>(Q);
            cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    PyrParams P;
    P.in = in;
    P.in_w = w;
    P.in_h = h;
    P.in_tlog2 = -1;
    P.out = out;
    P.tlog2 = tlog2;
    size_t done = 0;
    while (done < ws.size()) {
        P.nlev = (int)std::min<size_t>(kPyrPassLevels, ws.size() - done);
        for (int k = 0; k < P.nlev; ++k) P.lev[k] = PyrLevel{ws[done + k], hs[done + k], offs[done + k]};
        const dim3 grid((unsigned)((P.in_w + kPyrTile - 1) / kPyrTile), (unsigned)((P.in_h + kPyrTile - 1) / kPyrTile));
        k_pyramid<<<grid, kPyrThreads, 0, s>>>(P);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        done += (size_t)P.nlev;
        const size_t last = done - 1;
        P.in = out + offs[last];
        P.in_w = ws[last];
        P.in_h = hs[last];
        P.in_tlog2 = tlog2;
    }
    return cudaSuccess;
}

}  // namespace vr
