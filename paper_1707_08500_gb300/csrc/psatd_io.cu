// Moves between global arrays and the padded-box arenas of a plan (the data
// layout of Sec. 3.2 / Fig. 2a of arXiv:1707.08500): scatter fills every
// local cell of every box -- valid cells and guard images -- from the
// periodic global grid; gather writes each box's valid cells back to it.
// Pure copies, one CTA per (field, subdomain, z plane).  A thread keeps one
// column (16 bytes of it where both sides allow) and steps down the rows, kRows
// of them in flight: bound by HBM, or by the L2 for the guard cells that a
// scatter reads again.  A row per warp and one load in flight took 0.73 ms for
// four fields into and six out of 64 boxes of 96^3 (2.7 TB/s); this takes
// 0.336 ms (5.9 TB/s).
#include <cuda_runtime.h>

#include <cstdint>

#include "psatd_internal.h"
#include "psatd_io.h"
#include "psatd_launch.cuh"

namespace psatd {

namespace {

constexpr int kIoThreads = 256;

// 16-byte vector of T
template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; };
template <> struct Vec16<double> { using type = double2; };

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

__device__ __forceinline__ int wrap(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

constexpr int kRows = 4;   // rows in flight per thread

// Copy `rows` rows of `cols` elements of VT (one element, or 16 bytes): row y
// from in + gy ild + gx, to out + y old + x, where gy = wrap(gy0 + y, ny) and
// gx = wrap(gx0 + x, nx) (a gather passes ranges that do not wrap).  ild, old,
// gx0 and nx count elements of VT.  Loads through the L2 (__ldcg): the kernel
// ahead may still be writing the source when this block starts (see
// wait_for_previous_launch), and guard cells are read again by other blocks, not
// by this one.
// WIDE: rows may be wider than half the block; they go in the number of equal
// parts that keeps most threads at work (one row of 130 would idle half the
// block, one of 320 give its last 64 elements a step of their own: six FP64
// arrays of 640 x 64 x 20 gathered in 28.3 us whole, 20.9 in parts, with the
// device idle before).  In its own kernel: the search costs boxes of 24^3 6%.
template <bool WIDE, typename VT>
__device__ __forceinline__ void copy_rows(const VT* in, int64_t ild, int gx0, int nx, int gy0, int ny, VT* out, int64_t old,
                                          int cols, int rows) {
    int ct = min(cols, kIoThreads), rs = kIoThreads / ct;   // columns and rows of one step of the block
    if (WIDE && cols > kIoThreads / 2) {
        int parts = (cols + ct - 1) / ct;
        for (int n = parts + 1, end = parts + 6; n <= end; ++n) {
            const int c = (cols + n - 1) / n, r = kIoThreads / c;
            if (n * rs < parts * r) { parts = n; ct = c; rs = r; }
        }
    }
    const int y0 = int(threadIdx.x) / ct, x0 = int(threadIdx.x) - y0 * ct;
    if (y0 >= rs) return;
    for (int x = x0; x < cols; x += ct) {
        const VT* src = in + wrap(gx0 + x, nx);
        int gy = wrap(gy0 + y0, ny);
        VT* dst = out + int64_t(y0) * old + x;
        for (int y = y0; y < rows; y += kRows * rs) {
            VT v[kRows];
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                if (y + k * rs < rows) v[k] = __ldcg(src + int64_t(gy) * ild);
                gy += rs;
                if (gy >= ny) gy = rs <= ny ? gy - ny : gy % ny;
            }
#pragma unroll
            for (int k = 0; k < kRows; ++k, dst += int64_t(rs) * old)
                if (y + k * rs < rows) *dst = v[k];
        }
    }
}

template <typename T, bool WIDE>
__global__ void __launch_bounds__(kIoThreads) k_scatter(IoArgs a) {
    wait_for_previous_launch();
    const int64_t item = blockIdx.x;
    const int f = int(item / a.planes_local);
    const int64_t p = item - int64_t(f) * a.planes_local;
    const int s = __ldg(a.plane_sub_local + p);
    const IoDesc& d = a.desc[s];
    const int z = int(p - d.zstart_local);
    const int Lx = d.L[0], Ly = d.L[1];
    const int gz = wrap(d.org[2] + z, a.gn[2]);
    const T* in = static_cast<const T*>(a.in[f]) + int64_t(gz) * a.gn[1] * a.gn[0];
    T* out = static_cast<T*>(a.out[f]) + d.field_off + int64_t(z) * Ly * Lx;
    // 16-byte pieces where they start on 16-byte boundaries on both sides (a
    // piece then never straddles the periodic edge)
    constexpr int V = 16 / int(sizeof(T));
    using V16 = typename Vec16<T>::type;
    if (d.org[0] % V == 0 && a.gn[0] % V == 0 && Lx % V == 0 && aligned16(in) && aligned16(out))
        copy_rows<WIDE>(reinterpret_cast<const V16*>(in), int64_t(a.gn[0] / V), d.org[0] / V, a.gn[0] / V, d.org[1], a.gn[1],
                  reinterpret_cast<V16*>(out), int64_t(Lx / V), Lx / V, Ly);
    else
        copy_rows<WIDE>(in, int64_t(a.gn[0]), d.org[0], a.gn[0], d.org[1], a.gn[1], out, int64_t(Lx), Lx, Ly);
}

template <typename T, bool WIDE>
__global__ void __launch_bounds__(kIoThreads) k_gather(IoArgs a) {
    wait_for_previous_launch();
    const int64_t item = blockIdx.x;
    const int f = int(item / a.planes_valid);
    const int64_t p = item - int64_t(f) * a.planes_valid;
    const int s = __ldg(a.plane_sub_valid + p);
    const IoDesc& d = a.desc[s];
    const int zv = int(p - d.zstart_valid);
    const int Lx = d.L[0], Ly = d.L[1];
    const T* in = static_cast<const T*>(a.in[f]) + d.field_off + (int64_t(zv + d.g[2]) * Ly + d.g[1]) * Lx + d.g[0];
    T* out = static_cast<T*>(a.out[f]) + (int64_t(d.lo[2] + zv) * a.gn[1] + d.lo[1]) * a.gn[0] + d.lo[0];
    constexpr int V = 16 / int(sizeof(T));
    using V16 = typename Vec16<T>::type;
    if (d.n[0] % V == 0 && Lx % V == 0 && a.gn[0] % V == 0 && aligned16(in) && aligned16(out))
        copy_rows<WIDE>(reinterpret_cast<const V16*>(in), int64_t(Lx / V), 0, d.n[0] / V, 0, d.n[1], reinterpret_cast<V16*>(out),
                  int64_t(a.gn[0] / V), d.n[0] / V, d.n[1]);
    else
        copy_rows<WIDE>(in, int64_t(Lx), 0, d.n[0], 0, d.n[1], out, int64_t(a.gn[0]), d.n[0], d.n[1]);
}

}  // namespace

cudaError_t launch_io(bool scatter, bool f64, const IoArgs& a, cudaStream_t st) {
    const int64_t items = int64_t(a.nfields) * (scatter ? a.planes_local : a.planes_valid);
    if (items <= 0) return cudaSuccess;
    if (items > 2147483647) return cudaErrorInvalidConfiguration;
    const bool wide = a.widest > kIoThreads / 2;
    auto pick = [&](auto t) -> void (*)(IoArgs) {
        using T = decltype(t);
        return scatter ? (wide ? k_scatter<T, true> : k_scatter<T, false>) : (wide ? k_gather<T, true> : k_gather<T, false>);
    };
    // Crowded SMs (see overlap_pays) cost more than the overlap gains once a
    // block's plane is large: gathers of six arrays, overlapped / not, 520 x 64 x
    // 20 in FP64 (260 KB a plane) 23.9 / 14.5 us, three of 96 x 200 x 64 (150 KB)
    // 14.0 / 10.4, but one of eight boxes of 96^3 in FP32 (36 KB) 4.0 / 6.2.
    const bool overlap = a.plane_bytes <= 96 * 1024 || overlap_pays(items);
    return launch_maybe_overlapped(overlap, f64 ? pick(double()) : pick(float()), dim3(unsigned(items)), kIoThreads, 0, st, a);
}

}  // namespace psatd
