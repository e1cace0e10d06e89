// Kernels of one lattice x store combination, selected at compile time by
// ELBM_D (2 or 3) and ELBM_ST (elbm::StoreKind).  Built once per combination so
// the eight variants compile in parallel.
//
//   init_kernel          f = f^eq, g = g^eq of (rho, u, T)              (Eqs. 27eq, geq_i)
//   fields_kernel        rho, u, T of the current populations           (Eqs. density..E)
//   totals_kernel        FP64 totals of the current state (per-CTA partials)
//   stats_kernel         turbulence statistics of the current state (per-CTA partials)
//   moments_kernel       two-pass schedule, pass 1: Q~_aaa field        (Eq. anomalya)
//   collide_kernel       two-pass schedule, pass 2: pull, collide, store (Eqs. fLBGK, gLBGK)
//   moments64_kernel, collide64_kernel  the two passes in FP64 (the default of D3Q27 FP64, and of
//                        D2Q9 FP64 grids beyond the strips and tiles)
//   fused2d_row_kernel, fused2d_split_kernel  D2Q9 step of a small grid: strips of 30 nodes (FP64:
//                        four warps share a strip's arithmetic)
//   fused2d_kernel       D2Q9 one-kernel step: tile + halo moments in shared memory
//   march2d_kernel, march2d_pair_kernel  D2Q9 row march (the latter: 16-bit stores, two nodes a thread)
//   ensemble2d_kernel, ensemble_march2d_kernel  persistent steps of an ensemble
//   fused3d_kernel       D3Q27 one-kernel step: xy tile + halo marching along z, the pulled
//                        populations of each plane prefetched into shared memory with
//                        cp.async one plane ahead; on the single store in place, after
//                        aa_edges_kernel
//   fused3d_tma_kernel   the same with tensor copies
//   fused3d_reread_kernel  D3Q27 one-kernel step without the shared-memory plane buffers:
//                        the populations of a plane are gathered twice (moments of the
//                        next plane, then the collision), the second time from L2
//   aa_moments_kernel, aa_collide_kernel  two passes on the single store
//
// Layout: element [i * N + n] holds the pair (f_i, g_i) of direction i at node n.
// Streaming is "pull": the pair of direction i at node x is read from x - c_i of the
// source store and the post-collision pair is written at x in the destination store
// (ping-pong), so every store is coalesced and no two threads write one element.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <cstring>
#include <type_traits>

#include "elbm_internal.h"
#include "elbm_node.cuh"
#include "elbm_pair.cuh"

#ifndef ELBM_D
#error "ELBM_D must be defined (2 or 3)"
#endif
#ifndef ELBM_ST
#error "ELBM_ST must be defined (elbm::StoreKind)"
#endif

namespace elbm {
namespace {

constexpr int kD = ELBM_D;
constexpr int kST = ELBM_ST;
using Cd = Codec<kST>;
using P = typename Cd::P;
using R = typename Cd::R;
constexpr int Q = Lat<kD>::Q;
constexpr bool DEV = Cd::DEV;

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long node_index(const KParams& p, int x, int y, int z) {
    return (long long)x + (long long)p.nx * ((long long)y + (long long)p.ny * (long long)z);
}

// Source nodes of the pull at node (x, y, z): direction i = a + 3b + 9c is read at
// (xs[a], ys[b], zs[c]) = (x - c_x, y - c_y, z - c_z) with ghosts resolved by map_axis.
// Node indices fit in 32 bits (N <= 2^31); only the per-direction plane offset
// i * N needs 64 bits, and it is the same for every thread.
struct PullRows {
    int row[3][3];   // node index of (0, ys[b], zs[c])
    int xs[3];
    unsigned gmask;  // bit i: direction i is pulled from beyond a fixed-state face
};

// Fixed-state faces (D2Q9): is coordinate v of axis a beyond a fixed face, and the
// ghost values there (the fixed state's equilibria as raw stored values, its Q~).
__device__ __forceinline__ bool beyond_fixed(const KParams& p, int a, int v, int n) {
    return (v < 0 && p.fix_lo[a]) || (v >= n && p.fix_hi[a]);
}
__device__ __forceinline__ void fixed_pair(const KParams& p, int i, R& f, R& g) {
    if constexpr (sizeof(R) == 8) {
        f = p.fixd[i][0];
        g = p.fixd[i][1];
    } else {
        f = p.fixf[i].x;
        g = p.fixf[i].y;
    }
}
__device__ __forceinline__ R fixed_Q(const KParams& p, int a) {
    if constexpr (sizeof(R) == 8) return p.fixQd[a];
    else return p.fixQf[a];
}

// Directions of node (x, y) whose pull source lies beyond a fixed-state face (D2Q9;
// bit i for direction i): their pairs are the fixed state's, not a stored node's.
// FIX = false: a kernel compiled for grids without fixed faces (always 0).
template <bool FIX = true>
__device__ __forceinline__ unsigned fixed_mask(const KParams& p, int x, int y) {
    unsigned m = 0u;
    if constexpr (kD == 2 && FIX) {
        if (p.has_fixed) {
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    if (beyond_fixed(p, 0, x + 1 - a, p.nx) || beyond_fixed(p, 1, y + 1 - b, p.ny))
                        m |= 1u << (a + 3 * b);
        }
    }
    return m;
}

// With PULL = false every direction is read at the node itself (no streaming);
// that form is used once, to collide the initial state.
template <bool PULL = true>
__device__ __forceinline__ void pull_rows(const KParams& p, int x, int y, int z, PullRows& r) {
    r.xs[0] = PULL ? map_axis(x + 1, p.nx, p.per_x) : x;
    r.xs[1] = x;
    r.xs[2] = PULL ? map_axis(x - 1, p.nx, p.per_x) : x;
    int ys[3] = {PULL ? map_axis(y + 1, p.ny, p.per_y) : y, y, PULL ? map_axis(y - 1, p.ny, p.per_y) : y};
    int zs[3] = {z, z, z};
    if (kD == 3 && PULL) {
        zs[0] = map_axis(z + 1, p.nz, p.per_z);
        zs[2] = map_axis(z - 1, p.nz, p.per_z);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            r.row[b][c] = p.nx * (ys[b] + p.ny * zs[c]);
    r.gmask = PULL ? fixed_mask(p, x, y) : 0u;
}

// Address of the pair of direction i pulled by node r in store s.
__device__ __forceinline__ const P* src_ptr(const KParams& p, const P* __restrict__ s, const PullRows& r, int i) {
    const int a = i % 3, b = (i / 3) % 3, c = (kD == 3) ? i / 9 : 1;
    return (s + (size_t)i * (size_t)p.N) + (unsigned)(r.row[b][c] + r.xs[a]);
}

__device__ __forceinline__ void gather(const KParams& p, const P* __restrict__ src, const PullRows& r,
                                       R* f, R* g) {
#pragma unroll
    for (int i = 0; i < Q; ++i) Cd::dec(*src_ptr(p, src, r, i), f[i], g[i]);
    if (r.gmask) {   // sources beyond a fixed-state face (the load above read a clamped node)
#pragma unroll
        for (int i = 0; i < Q; ++i)
            if ((r.gmask >> i) & 1u) fixed_pair(p, i, f[i], g[i]);
    }
}

// The post-collision pairs C(X_n)_i of node n as stored: in place (p.aa = 0), or in the AA
// single-store layouts (p.aa = 1: direction i at opp(i) of the node; p.aa = 2: direction i
// pushed to the node's neighbour n + c_i, periodic).
__device__ __forceinline__ void load_local(const KParams& p, const P* __restrict__ pop, long long n, R* f,
                                           R* g) {
    if (p.aa == 0) {
#pragma unroll
        for (int i = 0; i < Q; ++i) Cd::dec(pop[(size_t)i * (size_t)p.N + (size_t)n], f[i], g[i]);
    } else if (p.aa == 1) {
#pragma unroll
        for (int i = 0; i < Q; ++i) Cd::dec(pop[(size_t)(Q - 1 - i) * (size_t)p.N + (size_t)n], f[i], g[i]);
    } else {
        const int x = (int)(n % p.nx), y = (int)((n / p.nx) % p.ny), z = (int)(n / ((long long)p.nx * p.ny));
        PullRows r;
        pull_rows(p, x, y, z, r);   // the pull source of opp(i) is n + c_i
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int k = Q - 1 - i, a = k % 3, b = (k / 3) % 3, c = (kD == 3) ? k / 9 : 1;
            Cd::dec(*((pop + (size_t)i * (size_t)p.N) + (unsigned)(r.row[b][c] + r.xs[a])), f[i], g[i]);
        }
    }
}

__device__ __forceinline__ void store_node(const KParams& p, P* __restrict__ dst, long long n, const R* f,
                                           const R* g) {
    const unsigned nn = (unsigned)n;
#pragma unroll
    for (int i = 0; i < Q; ++i) (dst + (size_t)i * (size_t)p.N)[nn] = Cd::enc(f[i], g[i]);
}

// Totals of one node: rho, rho u_x, rho u_y, rho u_z, rho E.
__device__ __forceinline__ void node_totals(const Moments<R>& m, R rE, R v[5]) {
    v[0] = m.rho;
    v[1] = m.rho * m.ux;
    v[2] = m.rho * m.uy;
    v[3] = m.rho * m.uz;
    v[4] = rE;
}

// Per-thread running sum of the node totals over the planes of a z segment:
// Kahan-compensated in FP64; in FP32 a plain sum (at most p.tz terms of per-node
// values that are themselves FP32 results), which saves the registers of the
// compensation terms.
struct Acc5 {
    R s[5], c[5];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int k = 0; k < 5; ++k) s[k] = c[k] = R(0);
    }
    __device__ __forceinline__ void add(const R v[5]) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if constexpr (sizeof(R) == 8) {
                const R y = v[k] - c[k];
                const R t = s[k] + y;
                c[k] = (t - s[k]) - y;
                s[k] = t;
            } else {
                s[k] += v[k];
            }
        }
    }
    __device__ __forceinline__ void total(R out[5]) {
#pragma unroll
        for (int k = 0; k < 5; ++k) out[k] = s[k] - c[k];
    }
};

// Block-wide FP64 sum of 5 values per thread of a block of at most MAXT threads; out[0..4].  The
// values go through shared memory, so that one warp per value adds them on full warps: 60 FP64
// warp instructions for 256 threads, where a shuffle tree in every warp takes 240.
template <int MAXT>
__device__ __forceinline__ void block_sum5(const double v[5], double* __restrict__ out) {
    __shared__ double red[5][MAXT];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthreads = blockDim.x * blockDim.y * blockDim.z, lane = tid & 31;
#pragma unroll
    for (int k = 0; k < 5; ++k) red[k][tid] = v[k];
    __syncthreads();
    for (int k = tid >> 5; k < 5; k += nthreads >> 5) {
        double t = red[k][lane];
        for (int j = lane + 32; j < nthreads; j += 32) t += red[k][j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) out[k] = t;
    }
}

// The same sum for kernels that reduce once per small tile: the sum within each warp runs
// in the arithmetic type T (an FP64 shuffle tree per 256-node tile costs more than the
// tile's whole update on GB300's narrow FP64 pipe), the sum of the warp partials in FP64.
// With T = double it is block_sum5.  An FP32 warp partial of 32 node values carries a
// relative rounding error of about 1e-7, below the rounding of the FP32 values summed.
template <typename T, int MAXT = 256>
__device__ __forceinline__ void block_sum5_warp(T v[5], double* __restrict__ out) {
    if constexpr (sizeof(T) == 8) {
        block_sum5<MAXT>(v, out);
    } else {
        __shared__ double red[32][5];
        const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
        const int nthreads = blockDim.x * blockDim.y * blockDim.z;
        const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < 5; ++k) red[warp][k] = (double)v[k];
        __syncthreads();
        if (tid < 5) {
            const int nw = (nthreads + 31) >> 5;
            double t = 0.0;
            for (int w = 0; w < nw; ++w) t += red[w][tid];
            out[tid] = t;
        }
    }
}

__device__ __forceinline__ void flag_if(bool bad, int* __restrict__ status) {
    // every thread of the warp reaches this call
    const unsigned any = __ballot_sync(0xffffffffu, bad);
    if (any && (threadIdx.x & 31) == 0 && status) atomicOr(status, 1);
}

// Asynchronous global -> shared copy of one pair (cp.async, bypasses registers).
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// Waits until at most N of this thread's most recent cp.async groups are still pending.
template <int N>
__device__ __forceinline__ void cp_async_wait_pending() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Programmatic dependent launch.  The step kernels are launched by launch_dependent: the next
// one's CTAs may be set up as soon as every CTA of this one has called launch_dependents, and
// wait for its end, with its writes visible, before they touch memory (wait_for_previous, in every
// CTA, so that the wait carries over from launch to launch).  Launched one after another
// without it, kernels start on a raster of about 2.05 us.  Most kernels call it late, a marching
// one when its column is done: CTAs set up beside a whole grid that is still running are
// spread unevenly (D2Q9 724^2, FP32: 22.6 us a step without dependent launches, 34.7 with early
// ones).  The pointers such a kernel reads are not const __restrict__: the compiler would load
// through the non-coherent path, which is for data that nobody writes while the grid exists, and a
// dependent grid exists while the one before it still writes.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void dependent_launch_point() {
    wait_for_previous();
    launch_dependents();
}

// ---------------------------------------------------------------------------
// initial state and field extraction
// ---------------------------------------------------------------------------
// Nodes n0 .. n0 + cnt - 1; the fields hold those nodes only (u component-major with
// stride cnt).
__global__ void init_kernel(const __grid_constant__ KParams p, const double* __restrict__ rho,
                            const double* __restrict__ u, const double* __restrict__ T,
                            P* __restrict__ pop, int* __restrict__ status, long long n0, long long cnt) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = n0 + k;
    bool bad = false;
    if (k < cnt) {
        const R r = (R)rho[k], t = (R)T[k];
        const R ux = (R)u[k], uy = (R)u[cnt + k], uz = kD == 3 ? (R)u[2 * cnt + k] : R(0);
        bad = !(r > R(0)) || !(t > R(0)) || !isfinite(r) || !isfinite(t) || !isfinite(ux) ||
              !isfinite(uy) || !isfinite(uz);
        R f[Q], g[Q];
        equilibria<kD, R>(r, ux, uy, uz, t, U_of_T(t, p), f, g);
        if constexpr (DEV) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                f[i] -= R(p.rest2[i].x);
                g[i] -= R(p.rest2[i].y);
            }
        }
        store_node(p, pop, n, f, g);
    }
    flag_if(bad, status);
}

// Nodes n0 .. n0 + cnt - 1 into fields of cnt nodes (u component-major with stride cnt).
__global__ void fields_kernel(const __grid_constant__ KParams p, const P* __restrict__ pop,
                              double* __restrict__ rho, double* __restrict__ u,
                              double* __restrict__ T, int* __restrict__ status, long long n0, long long cnt) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long n = n0 + k;
    bool bad = false;
    if (k < cnt) {
        R f[Q], g[Q];
        load_local(p, pop, n, f, g);
        Moments<R> m;
        node_moments<kD, R, false, DEV>(f, g, p, m);
        rho[k] = m.rho;
        u[k] = m.ux;
        u[cnt + k] = m.uy;
        if (kD == 3) u[2 * cnt + k] = m.uz;
        T[k] = m.T;
        bad = nonphysical(m);
    }
    flag_if(bad, status);
}

// Totals of the current state.  A work unit is a run of kTotThreads x kTotRun pairs of one
// direction's plane, read as it lies in memory, and CTA b takes units b, b + gridDim.x, ...: the
// device walks through the planes one after another.  A thread sums its share of F = sum f_i and
// G = sum g_i, and only at a plane's end turns F into the sums of rho and rho c_i f_i.  That is
// two additions per pair where a sum over each node's moments takes five or more, each of them
// compensated.  FP32-arithmetic stores: the sums are three-float ones (Tri2) throughout, so no
// FP64 instruction runs before a CTA's last warp; as an FP64 sum per node the FP64 pipe bounded
// it (256^3, FP32: 6.08 ms, now 0.56, which is 6.5 TB/s).  FP64 store: sums of kTotRun pairs as
// integers (FixedSum), compensated from there on (128^3: 0.65 ms, now 0.30; as FP64 sums 0.45).  Runs
// of 16 pairs and a plane's bounds tested on its last unit alone: with runs of 8, a 64-bit
// division a unit and five CTAs to an SM it waited for its own address arithmetic (256^3: FP32
// 0.64 ms, FP16 0.70, now 0.53).  Each CTA writes five sums and their five corrections.
constexpr int kTotRun = 16;   // pairs in flight per thread
constexpr int kTotThreads = 256;
constexpr int kTotCtas = sizeof(R) == 8 ? 1 : 3;   // per SM; FP64: what a thread does once takes the FP64 pipe
struct TotalsF64 {
    double F = 0, Fc = 0, G = 0, Gc = 0, s[5] = {}, c[5] = {};
    __device__ __forceinline__ void pairs(const R* f, const R* g) {
        add(F, Fc, f);
        add(G, Gc, g);
    }
    // s + c += the values of a run: their integer sum as its upper bits and its low 24, either exact
    static __device__ __forceinline__ void add(double& s, double& c, const R* v) {
        static_assert(kTotRun <= 27, "values that a sum of integers holds");
        int top = 0;
#pragma unroll
        for (int k = 0; k < kTotRun; ++k) top = FixedSum::top_of(top, v[k]);
        if (!FixedSum::usable(top)) {
#pragma unroll
            for (int k = 0; k < kTotRun; ++k) dd_add(s, c, v[k]);
            return;
        }
        top = (top >> 20) + 6;
        long long a = 0;
#pragma unroll
        for (int k = 0; k < kTotRun; ++k) a += FixedSum::fixed(v[k], top);
        const long long low = a & 0xffffff;
        dd_add(s, c, FixedSum::value(a - low, top));
        c += FixedSum::value(low, top);
    }
    __device__ __forceinline__ void plane_end(int i) {
        const double cx = cx_of(i), cy = cy_of(i), cz = cz_of<kD>(i);
        auto put = [&](int k, double x, double v, double vc) {
            dd_add(s[k], c[k], x * v);
            c[k] += x * vc;
        };
        put(0, 1.0, F, Fc);
        if (cx != 0.0) put(1, cx, F, Fc);
        if (cy != 0.0) put(2, cy, F, Fc);
        if (cz != 0.0) put(3, cz, F, Fc);
        put(4, 1.0, G, Gc);
        F = Fc = G = Gc = 0.0;
    }
    // this warp's sums and corrections, in its lane 0
    __device__ __forceinline__ void warp_total(int lane, double* out) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double v = __shfl_xor_sync(0xffffffffu, s[k], o);
                c[k] += __shfl_xor_sync(0xffffffffu, c[k], o);
                dd_add(s[k], c[k], v);
            }
            if (lane == 0) {
                out[k] = s[k];
                out[5 + k] = c[k];
            }
        }
    }
};
struct TotalsF32 {
    Tri2 a, t[3];   // (F, G); (rho, rho E), (rho u_x, rho u_y), (rho u_z, -)
    __device__ __forceinline__ TotalsF32() {
        a.zero();
#pragma unroll
        for (int k = 0; k < 3; ++k) t[k].zero();
    }
    __device__ __forceinline__ void pairs(const R* f, const R* g) {
#pragma unroll
        for (int k = 0; k < kTotRun; ++k) a.add(make_float2((float)f[k], (float)g[k]));
    }
    __device__ __forceinline__ void plane_end(int i) {
        t[0].add(a);
        // c_i F: products with -1, 0 and 1 are exact
        auto scaled = [&](float kx, float ky) {
            Tri2 m;
            m.s = make_float2(a.s.x * kx, a.s.x * ky);
            m.e1 = make_float2(a.e1.x * kx, a.e1.x * ky);
            m.e2 = make_float2(a.e2.x * kx, a.e2.x * ky);
            return m;
        };
        t[1].add(scaled((float)cx_of(i), (float)cy_of(i)));
        if (kD == 3) t[2].add(scaled((float)cz_of<kD>(i), 0.f));
        a.zero();
    }
    __device__ __forceinline__ void warp_total(int lane, double* out) {
#pragma unroll
        for (int k = 0; k < kD; ++k) t[k].warp_sum();
        if (lane == 0) {
            auto put = [&](int k, float a0, float e1, float e2) {
                out[k] = (double)a0;
                out[5 + k] = (double)e1 + (double)e2;
            };
            put(0, t[0].s.x, t[0].e1.x, t[0].e2.x);
            put(4, t[0].s.y, t[0].e1.y, t[0].e2.y);
            put(1, t[1].s.x, t[1].e1.x, t[1].e2.x);
            put(2, t[1].s.y, t[1].e1.y, t[1].e2.y);
            put(3, t[2].s.x, t[2].e1.x, t[2].e2.x);
        }
    }
};
__global__ void __launch_bounds__(kTotThreads, kTotCtas)
totals_kernel(const __grid_constant__ KParams p, const P* __restrict__ pop, double* __restrict__ partials, int units) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kWarps = kTotThreads / 32;
    __shared__ double part[kWarps][10];
    std::conditional_t<sizeof(R) == 8, TotalsF64, TotalsF32> tot;
    // unit `r` of direction i; the N nodes of a plane are at most 2^31
    int i = 0, r = (int)blockIdx.x;
    for (; r >= units && i < Q; ++i) r -= units;
    while (i < Q) {
        // the plane that holds direction i (swapped in the even AA layout)
        const P* __restrict__ b = pop + (size_t)(p.aa == 1 ? Q - 1 - i : i) * (size_t)p.N;
        const unsigned N = (unsigned)p.N;
        for (; r < units; r += (int)gridDim.x) {
            const unsigned n = (unsigned)r * (kTotThreads * kTotRun) + threadIdx.x;
            R f[kTotRun], g[kTotRun];
            if (r < units - 1) {
#pragma unroll
                for (int k = 0; k < kTotRun; ++k) Cd::dec(b[n + k * kTotThreads], f[k], g[k]);
            } else {
#pragma unroll
                for (int k = 0; k < kTotRun; ++k)
                    Cd::dec(n + k * kTotThreads < N ? b[n + k * kTotThreads] : Cd::enc(R(0), R(0)), f[k], g[k]);
            }
            tot.pairs(f, g);
        }
        tot.plane_end(i);
        for (; r >= units && i < Q; ++i) r -= units;
    }
    tot.warp_total(lane, part[warp]);
    __syncthreads();
    if (threadIdx.x < 5) {
        const int k = threadIdx.x;
        double a = 0.0, e = 0.0;
        for (int w = 0; w < kWarps; ++w) {
            dd_add(a, e, part[w][k]);
            e += part[w][5 + k];
        }
        if (DEV && blockIdx.x == 0 && (k == 0 || k == 4)) {   // N times the rest state's sums (no momentum)
            const double r = k == 0 ? (double)p.rest_rho : (double)p.rest_E, n = (double)p.N, v = r * n;
            dd_add(a, e, v);
            e += fma(r, n, -v);
        }
        partials[10 * blockIdx.x + k] = a;
        partials[10 * blockIdx.x + 5 + k] = e;
    }
}

// Turbulence statistics of the current state (one FP64 partial vector per CTA):
// sums of rho, rho^2, rho u.u, u.u, theta^2, T, T^2, (d u_x / d x)^2, |omega|^2, u_x^2
// and mu(T) |omega|^2, with the velocity gradient by second-order central differences
// (boundary nodes use the ghost values of the boundary map): dilatation
// theta = div u, vorticity omega = curl u, mu = mu0 (T/T0)^mu_exp (Eq. mu law).
//
// A CTA marches a 32 x 8 column over tz planes: each plane's velocities (tile and halo ring)
// go through shared memory, those of the planes below and above stay in registers, so the
// store is read once and a node's moments are computed 1.3 times (from seven reads and seven
// evaluations, 256^3 FP32 6.1 ms).  For the FP32-arithmetic stores the sums and their terms
// are unevaluated sums of floats: differences and products of FP32 values are exact as two
// floats, the viscosity law comes from pow_pos_df and the sums are Tri2 ones.  (With the law in
// FP64 that pipe bounded the kernel: 256^3 FP32 1.48 ms, without 0.79.)  Terms or sums that leave the range
// of floats, or fall so low that their second one does, show in the sums; elbm_turbulence_stats then asks for
// them in FP64 (WIDE, which FP64 stores always take).
constexpr int kStats = kStatsSums;
template <int DD, bool WIDE>
__global__ void __launch_bounds__(256, WIDE ? 1 : 2)
stats_kernel(const __grid_constant__ KParams p, const P* __restrict__ pop, double* __restrict__ partials, int tz,
             unsigned tiles_x, unsigned tiles_y) {
    constexpr int TX = 32, TY = 8, NT = TX * TY;
    __shared__ R us[2][DD][TY + 2][TX + 2];
    __shared__ double part[NT / 32][kStats];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + TX * ty;
    // columns in one dimension of the grid: the other two hold 65535 CTAs, and grids may be taller
    const unsigned row = blockIdx.x / tiles_x, seg = row / tiles_y;
    const int x0 = (int)(blockIdx.x - row * tiles_x) * TX, y0 = (int)(row - seg * tiles_y) * TY;
    const int zb = (int)seg * tz, ze = min(zb + tz, p.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < p.nx && y < p.ny;
    const int xl = min(x0 + TX, p.nx) - 1 - x0, yl = min(y0 + TY, p.ny) - 1 - y0;
    // halo ring: rows below and above, columns left and right; (hr, hc) its place in `us`
    int hx = 0, hy = 0, hr = 0, hc = 0;
    bool halo = false;
    if (tid < 2 * TX) {
        const int side = tid / TX;
        hc = tx + 1, hr = side ? yl + 2 : 0;
        hx = x, hy = map_axis(side ? y0 + yl + 1 : y0 - 1, p.ny, p.per_y);
        halo = tx <= xl;
    } else if (tid < 2 * TX + 2 * TY) {
        const int side = (tid - 2 * TX) / TY, k = (tid - 2 * TX) % TY;
        hr = k + 1, hc = side ? xl + 2 : 0;
        hy = y0 + k, hx = map_axis(side ? x0 + xl + 1 : x0 - 1, p.nx, p.per_x);
        halo = k <= yl;
    }
    struct Node {
        R u[3], rho, T;
    };
    auto node = [&](int nx_, int ny_, int nz_) {
        R f[Q], g[Q];
        load_local(p, pop, node_index(p, nx_, ny_, nz_), f, g);
        Moments<R> m;
        node_moments<kD, R, false, DEV>(f, g, p, m);
        return Node{{m.ux, m.uy, m.uz}, m.rho, m.T};
    };
    auto put = [&](int b, int r, int c, const Node& n) {
#pragma unroll
        for (int a = 0; a < DD; ++a) us[b][a][r][c] = n.u[a];
    };

    double acc[WIDE ? kStats : 1] = {};
    Tri2 t[6];   // not WIDE: the sums in pairs
#pragma unroll
    for (int k = 0; k < 6; ++k) t[k].zero();
    // bits of all that was squared: u_x, the other velocities, theta, d u_x / d x, omega
    unsigned any[5] = {};
    auto seen = [&](int k, float v) { any[k] |= __float_as_uint(v); };
    const float eh = (float)p.mu_exp;
    const Df mu_exp = {eh, WIDE ? 0.f : (float)(p.mu_exp - (double)eh)};
    // log2 T0 to a multiple of 2^-8, which the law's logarithms are taken from
    const float base = WIDE ? 0.f : rintf(log2f((float)p.T0) * 256.f) * 0x1p-8f;

    Node prev = {}, cur = {}, next = {};
    if (active) {
        if (DD == 3) prev = node(x, y, map_axis(zb - 1, p.nz, p.per_z));
        cur = node(x, y, zb);
        put(0, ty + 1, tx + 1, cur);
    }
    if (halo) put(0, hr, hc, node(hx, hy, zb));
    for (int z = zb; z < ze; ++z) {
        const int b = (z - zb) & 1;
        __syncthreads();   // plane z is in us[b]; us[b ^ 1] is free
        const int zn = map_axis(z + 1, p.nz, p.per_z);
        if (DD == 3 && active) {
            next = node(x, y, zn);
            if (z + 1 < ze) put(b ^ 1, ty + 1, tx + 1, next);
        }
        if (DD == 3 && halo && z + 1 < ze) put(b ^ 1, hr, hc, node(hx, hy, zn));
        if (active) {
            auto U = [&](int a, int r, int c) { return us[b][a][ty + 1 + r][tx + 1 + c]; };
            if constexpr (WIDE) {
                double G[3][3] = {};   // twice d u_a / d x_b
#pragma unroll
                for (int a = 0; a < DD; ++a) {
                    G[a][0] = (double)U(a, 0, 1) - U(a, 0, -1);
                    G[a][1] = (double)U(a, 1, 0) - U(a, -1, 0);
                    if (DD == 3) G[a][2] = (double)next.u[a] - prev.u[a];
                }
                const double theta = G[0][0] + G[1][1] + G[2][2];
                const double wx = G[2][1] - G[1][2], wy = G[0][2] - G[2][0], wz = G[1][0] - G[0][1];
                const double w2 = wx * wx + wy * wy + wz * wz;
                const double rho = cur.rho, T = cur.T, ux = cur.u[0], uy = cur.u[1], uz = cur.u[2];
                const double uu = ux * ux + uy * uy + uz * uz;
                acc[0] += rho;
                acc[1] = fma(rho, rho, acc[1]);
                acc[2] = fma(rho, uu, acc[2]);
                acc[3] += uu;
                acc[4] = fma(theta, theta, acc[4]);
                acc[5] += T;
                acc[6] = fma(T, T, acc[6]);
                acc[7] = fma(G[0][0], G[0][0], acc[7]);
                acc[8] += w2;
                acc[9] = fma(ux, ux, acc[9]);
                if (p.powlaw) acc[10] = fma(pow_pos(T * p.d_invT0, p.mu_exp), w2, acc[10]);
            } else {
                Df G[3][3];
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int k = 0; k < 3; ++k) G[a][k] = {0.f, 0.f};
#pragma unroll
                for (int a = 0; a < DD; ++a) {
                    G[a][0] = df_diff(U(a, 0, 1), U(a, 0, -1));
                    G[a][1] = df_diff(U(a, 1, 0), U(a, -1, 0));
                    if (DD == 3) G[a][2] = df_diff(next.u[a], prev.u[a]);
                }
                Df theta = df_add(G[0][0], G[1][1]);
                const Df wz = df_add(G[1][0], df_neg(G[0][1]));
                seen(0, cur.u[0]);
                seen(1, cur.u[1]);
                seen(3, G[0][0].h);
                seen(4, wz.h);
                float uu_rest = 0.f;
                Df w2 = df_sq(wz), uu = df_add(df_prod(cur.u[0], cur.u[0]), df_prod(cur.u[1], cur.u[1]), uu_rest);
                if (DD == 3) {
                    theta = df_add(theta, G[2][2]);
                    const Df wx = df_add(G[2][1], df_neg(G[1][2])), wy = df_add(G[0][2], df_neg(G[2][0]));
                    w2 = df_add(df_add(w2, df_sq(wx)), df_sq(wy));
                    seen(1, cur.u[2]);
                    seen(4, wx.h);
                    seen(4, wy.h);
                    uu = df_add(uu, df_prod(cur.u[2], cur.u[2]), uu_rest);
                }
                seen(2, theta.h);
                const Df r2 = df_prod(cur.rho, cur.rho), ruu = df_scale(uu, cur.rho), th2 = df_sq(theta);
                const Df T2 = df_prod(cur.T, cur.T), gxx = df_sq(G[0][0]), ux2 = df_prod(cur.u[0], cur.u[0]);
                t[0].add(make_float2(cur.rho, r2.h), make_float2(0.f, r2.l));
                t[1].add(make_float2(ruu.h, uu.h), make_float2(ruu.l, uu.l));
                t[1].e2 = add2(t[1].e2, make_float2(cur.rho * uu_rest, uu_rest));
                t[2].add(make_float2(th2.h, cur.T), make_float2(th2.l, 0.f));
                t[3].add(make_float2(T2.h, gxx.h), make_float2(T2.l, gxx.l));
                t[4].add(make_float2(w2.h, ux2.h), make_float2(w2.l, ux2.l));
                if (p.powlaw) {   // (T 2^-base)^mu_exp |omega|^2
                    Df y;
                    if (!pow_pos_df(cur.T, mu_exp, y, base)) y.h = y.l = __int_as_float(0x7fffffff);   // NaN: FP64 wanted
                    y = df_mul(y, w2);
                    t[5].add(make_float2(y.h, 0.f), make_float2(y.l, 0.f));
                }
            }
        }
        prev = cur;
        cur = next;
    }
    const int lane = tid & 31, warp = tid >> 5;
    if constexpr (WIDE) {
#pragma unroll
        for (int k = 0; k < kStats; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
            if (lane == 0) part[warp][k] = acc[k];
        }
    } else {
        // a sum of zero whose terms were not: they underflowed, FP64 wanted
        const float nan = __int_as_float(0x7fffffff);
        auto lost = [&](float& s, unsigned bits) {
            if (s == 0.f && (bits & 0x7fffffffu) != 0u) s = nan;
        };
        lost(t[1].s.x, any[0] | any[1]);
        lost(t[1].s.y, any[0] | any[1]);
        lost(t[2].s.x, any[2]);
        lost(t[3].s.y, any[3]);
        lost(t[4].s.x, any[4]);
        lost(t[4].s.y, any[0]);
        if (p.powlaw) lost(t[5].s.x, any[4]);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            t[k].warp_sum();
            if (lane == 0) {
                part[warp][2 * k] = (double)t[k].s.x + ((double)t[k].e1.x + (double)t[k].e2.x);
                if (k < 5) part[warp][2 * k + 1] = (double)t[k].s.y + ((double)t[k].e1.y + (double)t[k].e2.y);
            }
        }
    }
    __syncthreads();
    if (tid < kStats) {
        // theta, omega and d u_x / d x were summed as twice their values; the last sum lacks mu0, and (not
        // WIDE) has base for log2 T0, at the exponent in two floats
        const bool quad = tid == 4 || tid == 7 || tid == 8 || tid == 10;
        const int k = tid == 10 && !p.powlaw ? 8 : tid;
        double v = 0.0;
        for (int w = 0; w < NT / 32; ++w) v += part[w][k];
        if (quad) v *= 0.25;
        if (tid == 10) v *= p.mu0;
        if (tid == 10 && !WIDE && p.powlaw) v *= exp2(((double)mu_exp.h + mu_exp.l) * (base - log2(p.T0)));
        partials[(size_t)kStats * blockIdx.x + tid] = v;
    }
}

// ---------------------------------------------------------------------------
// two-pass schedule
// ---------------------------------------------------------------------------
// Pass 1: Q~_aaa at every node from the pulled (post-stream) populations.
template <bool PULL>
__global__ void moments_kernel(const __grid_constant__ KParams p, const P* src,
                               R* __restrict__ qf) {
    dependent_launch_point();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const int x = (int)(n % p.nx);
    const int y = (int)((n / p.nx) % p.ny);
    const int z = (int)(n / ((long long)p.nx * p.ny));
    PullRows r;
    pull_rows<PULL>(p, x, y, z, r);
    R f[Q], g[Q];
    gather(p, src, r, f, g);
    Moments<R> m;
    node_moments<kD, R, false, DEV>(f, g, p, m);
    qf[n] = anomaly(m.rho, m.ux, m.T);
    qf[p.N + n] = anomaly(m.rho, m.uy, m.T);
    if (kD == 3) qf[2 * p.N + n] = anomaly(m.rho, m.uz, m.T);
}

// Pass 2: pull, moments, derivative of Q~ from the field, collide, store.
template <bool PULL>
__global__ void collide_kernel(const __grid_constant__ KParams p, const P* src,
                               P* __restrict__ dst, const R* qf,
                               double* __restrict__ partials, int* __restrict__ status) {
    dependent_launch_point();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    R tot[5] = {0, 0, 0, 0, 0};
    bool bad = false;
    if (n < p.N) {
        const int x = (int)(n % p.nx);
        const int y = (int)((n / p.nx) % p.ny);
        const int z = (int)(n / ((long long)p.nx * p.ny));
        PullRows r;
        pull_rows<PULL>(p, x, y, z, r);
        R f[Q], g[Q];
        gather(p, src, r, f, g);
        Moments<R> m;
        node_moments<kD, R, true, DEV>(f, g, p, m);
        bad = nonphysical(m);
        const long long N = p.N;
        const int xm = map_axis(x - 1, p.nx, p.per_x), xp = map_axis(x + 1, p.nx, p.per_x);
        const int ym = map_axis(y - 1, p.ny, p.per_y), yp = map_axis(y + 1, p.ny, p.per_y);
        R qxm = qf[node_index(p, xm, y, z)], qxp = qf[node_index(p, xp, y, z)];
        R qym = qf[N + node_index(p, x, ym, z)], qyp = qf[N + node_index(p, x, yp, z)];
        if (kD == 2 && p.has_fixed) {
            if (beyond_fixed(p, 0, x - 1, p.nx)) qxm = fixed_Q(p, 0);
            if (beyond_fixed(p, 0, x + 1, p.nx)) qxp = fixed_Q(p, 0);
            if (beyond_fixed(p, 1, y - 1, p.ny)) qym = fixed_Q(p, 1);
            if (beyond_fixed(p, 1, y + 1, p.ny)) qyp = fixed_Q(p, 1);
        }
        const R Dx = dQ(p.deriv, m.ux, qxm, qf[n], qxp);
        const R Dy = dQ(p.deriv, m.uy, qym, qf[N + n], qyp);
        R Dz = R(0);
        if (kD == 3) {
            const int zm = map_axis(z - 1, p.nz, p.per_z), zp = map_axis(z + 1, p.nz, p.per_z);
            Dz = dQ(p.deriv, m.uz, qf[2 * N + node_index(p, x, y, zm)], qf[2 * N + n],
                    qf[2 * N + node_index(p, x, y, zp)]);
        }
        node_totals(m, m.rE, tot);
        collide<kD, R, DEV>(f, g, m, Dx, Dy, Dz, p);
        store_node(p, dst, n, f, g);
    }
    flag_if(bad, status);
    block_sum5_warp(tot, partials + 5 * blockIdx.x);
}

// The two passes in FP64.  The FP64 pipe bounds every FP64 kernel and the memory is idle (8 % of
// its rate), so the first pass computes the moments once and for all and hands them on, rather
// than have the second, or a halo, compute them again: rho, T, u and the flux part of q* go to
// the node's own pairs of the first planes of the destination store, which the same node's
// thread of the second pass reads before it writes there.  Q~, which neighbours read, goes to
// the Q~ field.  D3Q27 128^3: 3.39 -> 1.74 ms a step, from the re-read kernel, which computes the
// moments 2.3 times (both with the arithmetic of their time; with the sums and products in
// integers, FixedSum and FixedProd, 1.20 now, of which the traffic takes 0.46).
#if ELBM_ST == 0   // ST_F64
template <bool PULL>
__global__ void __launch_bounds__(kThreads1D)
moments64_kernel(const __grid_constant__ KParams p, const P* src, R* __restrict__ qf,
                 P* __restrict__ dst, double* __restrict__ partials, int* __restrict__ status) {
    wait_for_previous();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    R tot[5] = {0, 0, 0, 0, 0};
    bool bad = false;
    if (n < p.N) {
        const unsigned row = (unsigned)n / (unsigned)p.nx, x = (unsigned)n - row * (unsigned)p.nx;
        const unsigned z = row / (unsigned)p.ny, y = row - z * (unsigned)p.ny;
        PullRows r;
        pull_rows<PULL>(p, (int)x, (int)y, (int)z, r);
        R f[Q], g[Q];
        gather(p, src, r, f, g);
        Moments<R> m;
        node_moments<kD, R, true, DEV>(f, g, p, m);
        bad = nonphysical(m);
        node_totals(m, m.rE, tot);
        R dq[3];
        Relax<kD, R, DEV>::flux(m, dq);
        const R c = fma(R(-3), m.T, R(1));
        qf[n] = tot[1] * fma(-m.ux, m.ux, c);
        qf[p.N + n] = tot[2] * fma(-m.uy, m.uy, c);
        const size_t N = (size_t)p.N;
        dst[n] = Cd::enc(m.rho, m.T);
        dst[N + n] = Cd::enc(m.ux, m.uy);
        if (kD == 3) {
            qf[2 * p.N + n] = tot[3] * fma(-m.uz, m.uz, c);
            dst[2 * N + n] = Cd::enc(m.uz, dq[2]);
            dst[3 * N + n] = Cd::enc(dq[0], dq[1]);
        } else {
            dst[2 * N + n] = Cd::enc(dq[0], dq[1]);
        }
    }
    launch_dependents();
    flag_if(bad, status);
    block_sum5_warp(tot, partials + 5 * blockIdx.x);
}
constexpr int kThreads64 = 128;   // second pass: smaller CTAs, so that one's loads overlap another's arithmetic
// (registers capped at 128, D2Q9 102: uncapped 138 and 108 take a CTA from every SM, 96^3 409 -> 497 us)
template <bool PULL>
__global__ void __launch_bounds__(kThreads64, kD == 3 ? 4 : 5)
collide64_kernel(const __grid_constant__ KParams p, const P* src, P* __restrict__ dst, const R* qf) {
    wait_for_previous();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const unsigned row = (unsigned)n / (unsigned)p.nx, xu = (unsigned)n - row * (unsigned)p.nx;
    const int x = (int)xu, z = (int)(row / (unsigned)p.ny), y = (int)(row - (unsigned)z * (unsigned)p.ny);
    const long long N = p.N;
    PullRows r;
    pull_rows<PULL>(p, x, y, z, r);
    R rho, T, ux, uy, uz = R(0), dq[3] = {};
    Cd::dec(dst[n], rho, T);
    Cd::dec(dst[N + n], ux, uy);
    if (kD == 3) {
        Cd::dec(dst[2 * N + n], uz, dq[2]);
        Cd::dec(dst[3 * N + n], dq[0], dq[1]);
    } else {
        Cd::dec(dst[2 * N + n], dq[0], dq[1]);
    }
    const int xm = map_axis(x - 1, p.nx, p.per_x), xp = map_axis(x + 1, p.nx, p.per_x);
    const int ym = map_axis(y - 1, p.ny, p.per_y), yp = map_axis(y + 1, p.ny, p.per_y);
    R qxm = qf[node_index(p, xm, y, z)], qxp = qf[node_index(p, xp, y, z)];
    R qym = qf[N + node_index(p, x, ym, z)], qyp = qf[N + node_index(p, x, yp, z)];
    if (kD == 2 && p.has_fixed) {
        if (beyond_fixed(p, 0, x - 1, p.nx)) qxm = fixed_Q(p, 0);
        if (beyond_fixed(p, 0, x + 1, p.nx)) qxp = fixed_Q(p, 0);
        if (beyond_fixed(p, 1, y - 1, p.ny)) qym = fixed_Q(p, 1);
        if (beyond_fixed(p, 1, y + 1, p.ny)) qyp = fixed_Q(p, 1);
    }
    const R Dx = dQ(p.deriv, ux, qxm, qf[n], qxp);
    const R Dy = dQ(p.deriv, uy, qym, qf[N + n], qyp);
    R Dz = R(0);
    if (kD == 3) {
        const int zm = map_axis(z - 1, p.nz, p.per_z), zp = map_axis(z + 1, p.nz, p.per_z);
        Dz = dQ(p.deriv, uz, qf[2 * N + node_index(p, x, y, zm)], qf[2 * N + n],
                qf[2 * N + node_index(p, x, y, zp)]);
    }
    launch_dependents();
    Relax<kD, R, DEV> rx;
    rx.init(rho, T, ux, uy, uz, dq, Dx, Dy, Dz, p);
    const unsigned nn = (unsigned)n;
    auto in = [&](int i, R& f, R& g) {
        Cd::dec(*src_ptr(p, src, r, i), f, g);
        if (kD == 2 && ((r.gmask >> i) & 1u)) fixed_pair(p, i, f, g);
    };
    auto out = [&](int i, R f, R g) { (dst + (size_t)i * (size_t)N)[nn] = Cd::enc(f, g); };
    // (a finite sum rho has finite terms, and T those of rho E).  With one CTA to an SM a warp has its FP64
    // pipe to itself, and the chains of integers are longer: 24^3 24.5 us a step, in integers 26.3
    if (gridDim.x > (unsigned)p.sms && rx.usable() && finite64(rho) && finite64(T)) {
        rx.all(in, out);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            R f, g;
            in(i, f, g);
            out(i, rx.f(i, f, p), rx.g(i, g, p));
        }
    }
}
#endif

// ---------------------------------------------------------------------------
// AA single-store layout (periodic grids, two-pass schedule)
// ---------------------------------------------------------------------------
// One store A holds the post-collision state C(X_n) in one of two layouts that alternate
// with the step:
//   L0: C(X_n)_i(x) at A[opp(i)][x]          (swapped at the node)
//   L1: C(X_n)_i(x) at A[i][x + c_i]         (pushed to the neighbour, periodic wrap)
// A step from L0 pulls f_i(y) = C(X_n)_i(y - c_i) = A[opp(i)][y - c_i] and pushes the new
// C(X_n+1)_i(y) to A[i][y + c_i] (-> L1); a step from L1 reads f_i(y) = A[i][y] at the node
// itself and writes C(X_n+1)_i(y) to A[opp(i)][y] (-> L0).  In both, the slots a node
// writes are exactly the slots it read (for a step from L0, direction i's write target
// A[i][y + c_i] is direction opp(i)'s source), so with the Q~ field computed in a first pass
// every slot is read and written by one thread only.  A periodic map is a bijection; a
// clamped (zero-gradient) face would let two nodes read one slot that one of them writes.
__host__ __device__ constexpr int opp(int i) { return Q - 1 - i; }

// Address of direction j's pair in the row/column of direction k's pull source (PullRows of
// the node): a step from L0 reads A[opp(i)] at the source of i and writes A[i] at the
// source of opp(i).
__device__ __forceinline__ P* aa_ptr(const KParams& p, P* A, const PullRows& r, int j, int k) {
    const int a = k % 3, b = (k / 3) % 3, c = (kD == 3) ? k / 9 : 1;
    return (A + (size_t)j * (size_t)p.N) + (unsigned)(r.row[b][c] + r.xs[a]);
}

template <bool FROM_L1>
__device__ __forceinline__ void aa_gather(const KParams& p, P* A, const PullRows& r, long long n, R* f, R* g) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const P v = FROM_L1 ? A[(size_t)i * (size_t)p.N + (size_t)n] : *aa_ptr(p, A, r, opp(i), i);
        Cd::dec(v, f[i], g[i]);
    }
}
template <bool FROM_L1>
__device__ __forceinline__ void aa_store(const KParams& p, P* A, const PullRows& r, long long n, const R* f,
                                         const R* g) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const P v = Cd::enc(f[i], g[i]);
        if (FROM_L1) A[(size_t)opp(i) * (size_t)p.N + (size_t)n] = v;
        else *aa_ptr(p, A, r, i, opp(i)) = v;
    }
}

// Pass 1 of an AA step: Q~_aaa of every node from its post-stream populations.
template <bool FROM_L1>
__global__ void aa_moments_kernel(const __grid_constant__ KParams p, P* A, R* __restrict__ qf) {
    dependent_launch_point();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= p.N) return;
    const int x = (int)(n % p.nx), y = (int)((n / p.nx) % p.ny), z = (int)(n / ((long long)p.nx * p.ny));
    PullRows r;
    if (!FROM_L1) pull_rows(p, x, y, z, r);
    R f[Q], g[Q];
    aa_gather<FROM_L1>(p, A, r, n, f, g);
    Moments<R> m;
    node_moments<kD, R, false, DEV>(f, g, p, m);
    qf[n] = anomaly(m.rho, m.ux, m.T);
    qf[p.N + n] = anomaly(m.rho, m.uy, m.T);
    if (kD == 3) qf[2 * p.N + n] = anomaly(m.rho, m.uz, m.T);
}

// Pass 2 of an AA step: the same reads, the derivative of Q~ from the field, collision, and
// the writes into the slots just read.
// Two CTAs per SM (at most 128 registers) for the FP32-arithmetic stores: the L0 form holds
// the pull offsets for its pushed writes and would take 156 (FP32) / 182 (FP16) registers,
// one CTA of 8 warps per SM, which made it twice as slow as the L1 form (AA step at 256^3,
// FP32 6.1 -> 7.8 GLUPS, FP16 7.6 -> 10.7 with the cap, despite about 100 bytes of spills).
// FP64 keeps one CTA (the cap would spill 0.8 KB per thread).
constexpr int kAaMinBlocks = sizeof(R) == 4 ? 2 : 1;
template <bool FROM_L1>
__global__ void __launch_bounds__(kThreads1D, kAaMinBlocks)
aa_collide_kernel(const __grid_constant__ KParams p, P* A, const R* qf,
                                  double* __restrict__ partials, int* __restrict__ status) {
    dependent_launch_point();
    const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    R tot[5] = {0, 0, 0, 0, 0};
    bool bad = false;
    if (n < p.N) {
        const int x = (int)(n % p.nx), y = (int)((n / p.nx) % p.ny), z = (int)(n / ((long long)p.nx * p.ny));
        PullRows r;
        if (!FROM_L1) pull_rows(p, x, y, z, r);
        R f[Q], g[Q];
        aa_gather<FROM_L1>(p, A, r, n, f, g);
        Moments<R> m;
        node_moments<kD, R, true, DEV>(f, g, p, m);
        bad = nonphysical(m);
        const long long N = p.N;
        const int xm = map_axis(x - 1, p.nx, p.per_x), xp = map_axis(x + 1, p.nx, p.per_x);
        const int ym = map_axis(y - 1, p.ny, p.per_y), yp = map_axis(y + 1, p.ny, p.per_y);
        const R Dx = dQ(p.deriv, m.ux, qf[node_index(p, xm, y, z)], qf[n], qf[node_index(p, xp, y, z)]);
        const R Dy = dQ(p.deriv, m.uy, qf[N + node_index(p, x, ym, z)], qf[N + n], qf[N + node_index(p, x, yp, z)]);
        R Dz = R(0);
        if (kD == 3) {
            const int zm = map_axis(z - 1, p.nz, p.per_z), zp = map_axis(z + 1, p.nz, p.per_z);
            Dz = dQ(p.deriv, m.uz, qf[2 * N + node_index(p, x, y, zm)], qf[2 * N + n],
                    qf[2 * N + node_index(p, x, y, zp)]);
        }
        node_totals(m, m.rE, tot);
        collide<kD, R, DEV>(f, g, m, Dx, Dy, Dz, p);
        aa_store<FROM_L1>(p, A, r, n, f, g);
    }
    flag_if(bad, status);
    block_sum5_warp(tot, partials + 5 * blockIdx.x);
}

// ---------------------------------------------------------------------------
// fused schedules
// ---------------------------------------------------------------------------
constexpr int TX = 32;

// Halo ring of a TX x TY tile: 2*TX row nodes (they need Q~_yyy) and 2*TY column
// nodes (Q~_xxx).  Corners are never needed: the stencil uses axis neighbours only.
// Halo node h: [0,TX) row below, [TX,2TX) row above, then the left and right columns.
// Returns false for slots outside a ragged tile; (hx, hy) are mapped by the BCs and
// (sx, sy) is where its Q~ goes: qy[sy][sx] for rows, qx[sy][sx] for columns.
template <int TY>
__device__ __forceinline__ bool halo_node(const KParams& p, int h, int x0, int y0, int xl, int yl, int& hx,
                                          int& hy, int& sx, int& sy, int& axis) {
    if (h < TX) {
        hx = x0 + h; hy = map_axis(y0 - 1, p.ny, p.per_y); sx = h; sy = 0; axis = 1;
        return h <= xl;
    }
    if (h < 2 * TX) {
        const int k = h - TX;
        hx = x0 + k; hy = map_axis(y0 + yl + 1, p.ny, p.per_y); sx = k; sy = yl + 2; axis = 1;
        return k <= xl;
    }
    if (h < 2 * TX + TY) {
        const int k = h - 2 * TX;
        hx = map_axis(x0 - 1, p.nx, p.per_x); hy = y0 + k; sx = 0; sy = k; axis = 0;
        return k <= yl;
    }
    const int k = h - 2 * TX - TY;
    hx = map_axis(x0 + xl + 1, p.nx, p.per_x); hy = y0 + k; sx = xl + 2; sy = k; axis = 0;
    return k <= yl;
}

// D2Q9: one thread per node of a TX x TY tile.  Phase 1 pulls the populations into
// registers and puts Q~ of the tile and its halo ring into shared memory; phase 2
// collides and stores.  One launch per step, no intermediate field in HBM.  The tile
// body is shared by the per-lattice kernel and the persistent ensemble kernel;
// `partial` (may be null) receives the tile's totals.
template <int TY, bool CAL, bool ONE_WAIT>
__device__ __forceinline__ void fused2d_tile(const KParams& p, const P* __restrict__ src, P* __restrict__ dst,
                                             int bx, int by, double* __restrict__ partial,
                                             int* __restrict__ status) {
    __shared__ R qx[TY][TX + 2];
    __shared__ R qy[TY + 2][TX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = bx * TX, y0 = by * TY;
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < p.nx && y < p.ny;
    const int xl = min(x0 + TX, p.nx) - 1 - x0, yl = min(y0 + TY, p.ny) - 1 - y0;

    // ONE_WAIT: both gathers (the node's and its halo node's pairs) are issued before any
    // arithmetic, so the tile waits for memory once; the persistent ensemble kernel keeps
    // the node's gather and moments first, which needs fewer registers (64, no spills)
    const int h = tx + TX * ty;
    int hx = 0, hy = 0, sx = 0, sy = 0, axis = 0;
    const bool hv = h < 2 * TX + 2 * TY && halo_node<TY>(p, h, x0, y0, xl, yl, hx, hy, sx, sy, axis);
    // the unmapped halo coordinate is (x0 + sx - 1, y0 + sy) for columns and (x0 + sx, y0 + sy - 1)
    // for rows; beyond a fixed face the halo's Q~ is the fixed state's
    const bool hfixed = hv && p.has_fixed &&
                        (axis == 1 ? beyond_fixed(p, 1, y0 + sy - 1, p.ny) : beyond_fixed(p, 0, x0 + sx - 1, p.nx));
    R f[Q], g[Q];
    Moments<R> m;
    auto halo_q = [&](const R* hf, const R* hg) {
        Moments<R> hm;
        node_moments<kD, R, false, DEV, CAL>(hf, hg, p, hm);
        return anomaly(hm.rho, axis == 1 ? hm.uy : hm.ux, hm.T);
    };
    auto store_halo_q = [&](R q) {
        if (axis == 1) qy[sy][sx] = q;
        else qx[sy][sx] = q;
    };
    if constexpr (ONE_WAIT) {
        R hf[Q], hg[Q];
        if (active) {
            PullRows r;
            pull_rows(p, x, y, 0, r);
            gather(p, src, r, f, g);
        }
        if (hv && !hfixed) {
            PullRows r;
            pull_rows(p, hx, hy, 0, r);
            gather(p, src, r, hf, hg);
        }
        if (active) {
            node_moments<kD, R, true, DEV, CAL>(f, g, p, m);
            qx[ty][tx + 1] = anomaly(m.rho, m.ux, m.T);
            qy[ty + 1][tx] = anomaly(m.rho, m.uy, m.T);
        }
        if (hv) store_halo_q(hfixed ? fixed_Q(p, axis) : halo_q(hf, hg));
    } else {
        if (active) {
            PullRows r;
            pull_rows(p, x, y, 0, r);
            gather(p, src, r, f, g);
            node_moments<kD, R, true, DEV, CAL>(f, g, p, m);
            qx[ty][tx + 1] = anomaly(m.rho, m.ux, m.T);
            qy[ty + 1][tx] = anomaly(m.rho, m.uy, m.T);
        }
        if (hv) {
            R q;
            if (hfixed) {
                q = fixed_Q(p, axis);
            } else {
                PullRows r;
                pull_rows(p, hx, hy, 0, r);
                R hf[Q], hg[Q];
                gather(p, src, r, hf, hg);
                q = halo_q(hf, hg);
            }
            store_halo_q(q);
        }
    }
    if constexpr (ONE_WAIT) launch_dependents();
    __syncthreads();

    R tot[5] = {0, 0, 0, 0, 0};
    bool bad = false;
    if (active) {
        bad = nonphysical(m);
        const R Dx = dQ(p.deriv, m.ux, qx[ty][tx], qx[ty][tx + 1], qx[ty][tx + 2]);
        const R Dy = dQ(p.deriv, m.uy, qy[ty][tx], qy[ty + 1][tx], qy[ty + 2][tx]);
        if (partial) node_totals(m, m.rE, tot);
        collide<kD, R, DEV, CAL>(f, g, m, Dx, Dy, R(0), p);
        store_node(p, dst, node_index(p, x, y, 0), f, g);
    }
    flag_if(bad, status);
    if (partial) block_sum5_warp<R, TX * TY>(tot, partial);
    __syncthreads();   // the shared arrays are reused by the next tile of a persistent CTA
}

template <int TY, bool CAL>
__global__ void __launch_bounds__(TX * TY)
fused2d_kernel(const __grid_constant__ KParams p, const P* src, P* __restrict__ dst,
               double* __restrict__ partials, int* __restrict__ status) {
    wait_for_previous();
    fused2d_tile<TY, CAL, true>(p, src, dst, blockIdx.x, blockIdx.y, partials + 5 * (blockIdx.x + gridDim.x * blockIdx.y),
                     status);
}

// D2Q9 step of a small grid: a warp owns kRowW = 30 nodes of a row; its first and last lane hold
// the nodes at either end, for their Q~_xxx alone.  Nothing goes through shared memory but
// the totals: Q~_xxx of the x neighbours comes by shuffle, and of the two y neighbours only the
// upwind one is evaluated (both for the central derivative).  The pairs of all three nodes
// are requested before any arithmetic, so a warp waits for memory once.  A grid of a few
// thousand nodes is all latency, and in FP64 the arithmetic of a warp keeps its SM's pipe busy
// for about 16 cycles an instruction: one warp to a CTA spreads 3,200 nodes over 108 SMs
// where the 32 x 8 tiles used 25 (800 x 4, FP32: 3.4 us a step, this kernel 2.6).
constexpr int kRowSmem = 5 * 32 * (int)sizeof(R);   // its static shared memory, bytes
template <bool CAL, bool FIX>
__global__ void __launch_bounds__(32)
fused2d_row_kernel(const __grid_constant__ KParams p, const P* src, P* __restrict__ dst, int strips,
                   double* __restrict__ partials, int* __restrict__ status) {
    __shared__ R red[1][5][32];
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int y = warp / strips, x = (warp - y * strips) * kRowW - 1 + lane;
    const bool have = y < p.ny && x <= p.nx;                        // a node of the strip or an end
    const bool node = have && lane >= 1 && lane <= kRowW && x < p.nx;
    const int xc = map_axis(x, p.nx, p.per_x);
    const int yd = map_axis(y - 1, p.ny, p.per_y), yu = map_axis(y + 1, p.ny, p.per_y);
    auto request = [&](int yy, P pk[Q]) {
        PullRows r;
        pull_rows(p, xc, yy, 0, r);
#pragma unroll
        for (int i = 0; i < Q; ++i) pk[i] = *src_ptr(p, src, r, i);
    };
    auto decode = [&](const P pk[Q], int yy, R f[Q], R g[Q]) {
        const unsigned gm = fixed_mask<FIX>(p, xc, yy);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            Cd::dec(pk[i], f[i], g[i]);
            if ((gm >> i) & 1u) fixed_pair(p, i, f[i], g[i]);
        }
    };
    wait_for_previous();
    P pc[Q], pd[Q], pu[Q];
    if (have) request(y, pc);
    if (node) {
        request(yd, pd);
        request(yu, pu);
    }
    R f[Q], g[Q], qx = R(0);
    Moments<R> m;
    if (have) {
        decode(pc, y, f, g);
        node_moments<kD, R, true, DEV, CAL>(f, g, p, m);
        qx = FIX && p.has_fixed && beyond_fixed(p, 0, x, p.nx) ? fixed_Q(p, 0) : anomaly(m.rho, m.ux, m.T);
    }
    launch_dependents();
    const R qxm = __shfl_up_sync(0xffffffffu, qx, 1), qxp = __shfl_down_sync(0xffffffffu, qx, 1);
    R tot[5] = {0, 0, 0, 0, 0};
    bool bad = false;
    if (node) {
        bad = nonphysical(m);
        const R q0 = anomaly(m.rho, m.uy, m.T);
        auto neighbour_q = [&](const P pk[Q], int yy, int y_unmapped) {
            if (FIX && p.has_fixed && beyond_fixed(p, 1, y_unmapped, p.ny)) return fixed_Q(p, 1);
            R hf[Q], hg[Q];
            decode(pk, yy, hf, hg);
            Moments<R> hm;
            node_moments<kD, R, false, DEV, CAL>(hf, hg, p, hm);
            return anomaly(hm.rho, hm.uy, hm.T);
        };
        R Dy;
        if (p.deriv) {
            Dy = R(0.5) * (neighbour_q(pu, yu, y + 1) - neighbour_q(pd, yd, y - 1));
        } else {
            const bool up = m.uy > R(0);
            P pn[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) pn[i] = up ? pd[i] : pu[i];
            const R qn = neighbour_q(pn, up ? yd : yu, up ? y - 1 : y + 1);
            Dy = up ? q0 - qn : qn - q0;
        }
        const R Dx = dQ(p.deriv, m.ux, qxm, qx, qxp);
        node_totals(m, m.rE, tot);
        collide<kD, R, DEV, CAL>(f, g, m, Dx, Dy, R(0), p);
        store_node(p, dst, node_index(p, x, y, 0), f, g);
    }
    flag_if(bad, status);
    // totals of the warp: lane 4k + j adds eight of the 32 values of sum k
#pragma unroll
    for (int k = 0; k < 5; ++k) red[wb][k][lane] = tot[k];
    __syncwarp();
    const int k = lane >> 2, j = lane & 3;
    R t = R(0);
    if (k < 5) {
        const R* v = red[wb][k] + j;
        t = ((v[0] + v[4]) + (v[8] + v[12])) + ((v[16] + v[20]) + (v[24] + v[28]));
    }
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    if (k < 5 && j == 0) partials[5 * warp + k] = (double)t;
}

// The same strip in FP64, where one warp alone would take 10.5 us: an SM's quarter finishes an FP64
// warp instruction in 64 cycles, whatever lanes it has, and starts the next one only then, so
// a warp's instructions run one after another (measured: 64.6 cycles each at any degree of
// independence, 16.2 with four warps).  So four warps share a node's arithmetic: the moments
// of the node and of its two y neighbours; then the rates, the factors of either axis and the
// flux of q*; then one row of three directions each, and the totals.  63 FP64 instructions a warp on
// the average (800 x 4: 27,108 in 432 warps) instead of 205.
#if ELBM_ST == 0 && ELBM_D == 2
constexpr int kSplitSmem = 35 * 34 * (int)sizeof(double);   // its static shared memory, bytes
template <bool CAL, bool FIX>
__global__ void __launch_bounds__(128)
fused2d_split_kernel(const __grid_constant__ KParams p, const P* src, P* __restrict__ dst, int strips,
                     double* __restrict__ partials, int* __restrict__ status) {
    enum { RHO, TT_, UX, UY, RE, QXL, QX, QXR, QY, QD, QU, PX, GX, AX = GX + 3, PY = AX + 3, GY, SY = GY + 3, KK = SY + 3,
           WR, W1R, OMW, OMW1, HH, DX, DY, FX, FY, NV };
    static_assert(NV * 34 * sizeof(double) == kSplitSmem, "static shared memory");
    __shared__ double v[NV][34];   // column lane + 1 of a node; QXL and QXR are QX shifted by one
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5, col = lane + 1;
    const int y = blockIdx.x / strips, x = (blockIdx.x - y * strips) * kRowW - 1 + lane;
    const bool have = x <= p.nx;                                    // a node of the strip or an end
    const bool node = have && lane >= 1 && lane <= kRowW && x < p.nx;
    const int xc = map_axis(x, p.nx, p.per_x);
    // warps 0 and 3: the node's row; 1: the row below; 2: above
    const int yw = wb == 1 ? y - 1 : wb == 2 ? y + 1 : y, yy = map_axis(yw, p.ny, p.per_y);
    wait_for_previous();
    double f[Q], g[Q];
    Moments<double> m;
    if (wb == 0 || wb == 3 ? have : node) {
        PullRows r;
        pull_rows(p, xc, yy, 0, r);
        r.gmask = fixed_mask<FIX>(p, xc, yy);
        gather(p, src, r, f, g);
        if (wb == 3) {
            double rho, jx, jy, jz, P6[6];
            f_moments<kD, double, true, false>(f, p, rho, jx, jy, jz, P6);
            m.Pxx = P6[0];
            m.Pyy = P6[1];
            m.Pxy = P6[3];
        } else {
            node_moments<kD, double, false, false, CAL>(f, g, p, m);
            if (wb == 0) {
                v[RHO][col] = m.rho;
                v[TT_][col] = m.T;
                v[UX][col] = m.ux;
                v[UY][col] = m.uy;
                v[RE][col] = m.rE;
                const double q =
                    FIX && p.has_fixed && beyond_fixed(p, 0, x, p.nx) ? fixed_Q(p, 0) : anomaly(m.rho, m.ux, m.T);
                v[QX][col] = v[QXL][col + 1] = v[QXR][col - 1] = q;
                v[QY][col] = anomaly(m.rho, m.uy, m.T);
            } else {
                v[wb == 1 ? QD : QU][col] = FIX && p.has_fixed && beyond_fixed(p, 1, yw, p.ny)
                                                ? fixed_Q(p, 1)
                                                : anomaly(m.rho, m.uy, m.T);
            }
        }
    }
    __syncthreads();
    if (node) {
        m.rho = v[RHO][col];
        m.T = v[TT_][col];
        m.ux = v[UX][col];
        m.uy = v[UY][col];
        m.rE = v[RE][col];
        m.uz = 0.0;
        using Rx = Relax<kD, double, false, CAL>;
        if (wb == 0) {
            double k, omw, omw1, wr, w1r, h;
            Rx::rates(m.rho, m.T, p, k, omw, omw1, wr, w1r, h);
            v[KK][col] = k;
            v[WR][col] = wr;
            v[W1R][col] = w1r;
            v[OMW][col] = omw;
            v[OMW1][col] = omw1;
            v[HH][col] = h;
        } else if (wb < 3) {
            const double u = wb == 1 ? m.ux : m.uy, u2 = u * u, Pa = m.T + u2;
            double phi[3], ps[3];
            Rx::phi2(u, Pa, phi);
            Rx::psi2(u, u2, m.T, 2.5 * m.T, m.T * m.T, ps);
            const double U = U_of_T<double, CAL>(m.T, p);
            v[wb == 1 ? PX : PY][col] = Pa;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                v[(wb == 1 ? GX : GY) + a][col] = phi[a];
                v[(wb == 1 ? AX : SY) + a][col] = wb == 1 ? fma(U, phi[a], ps[a]) : ps[a];
            }
        } else {
            double dq[3];
            Rx::flux(m, dq);
            const double Dx = dQ(p.deriv, m.ux, v[QXL][col], v[QX][col], v[QXR][col]);
            const double Dy = dQ(p.deriv, m.uy, v[QD][col], v[QY][col], v[QU][col]);
            v[DX][col] = Dx;
            v[DY][col] = Dy;
            v[FX][col] = fma(m.ux, 0.5 * Dx, dq[0]);
            v[FY][col] = fma(m.uy, 0.5 * Dy, dq[1]);
        }
    }
    __syncthreads();
    launch_dependents();
    if (wb < 3) {   // row c_y = wb - 1
        if (node) {
            const double k = v[KK][col], omw = v[OMW][col], omw1 = v[OMW1][col];
            double X[3], Y[3];
            Relax<kD, double, false, CAL>::phi2(m.ux, fma(k, v[DX][col], v[PX][col]), X);
            Relax<kD, double, false, CAL>::phi2(m.uy, fma(k, v[DY][col], v[PY][col]), Y);
            const double wY = v[WR][col] * (wb == 0 ? Y[0] : wb == 1 ? Y[1] : Y[2]);
            const double A = v[W1R][col] * v[GY + wb][col], B = v[W1R][col] * v[SY + wb][col];
            const double hq = v[HH][col] * v[wb == 1 ? FX : FY][col];
            PullRows r;
            pull_rows(p, x, y, 0, r);
            r.gmask = fixed_mask<FIX>(p, x, y);
            const unsigned n = (unsigned)(x + p.nx * y);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int i = a + 3 * wb;
                double fi, gi;
                Cd::dec((src + (size_t)i * (size_t)p.N)[(unsigned)((wb == 0 ? r.row[0][1] : wb == 1 ? r.row[1][1] : r.row[2][1]) + r.xs[a])], fi, gi);
                if ((r.gmask >> i) & 1u) {
                    fi = p.fixd[i][0];
                    gi = p.fixd[i][1];
                }
                double go = fma(omw1, gi, fma(v[AX + a][col], A, v[GX + a][col] * B));
                // unit-speed directions: (+-1, 0) in the middle row, (0, +-1) in the outer ones
                if (wb == 1 ? a != 1 : a == 1) go = (wb == 1 ? a == 0 : wb == 0) ? go + hq : go - hq;
                (dst + (size_t)i * (size_t)p.N)[n] = Cd::enc(fma(omw, fi, X[a] * wY), go);
            }
        }
    } else {
        flag_if(node && nonphysical(m), status);
        // lane 4k + j adds eight of the 32 values of sum k: rho, rho u_x, rho u_y, rho u_z, rho E
        __syncwarp();
        v[QX][col] = node ? m.rho * m.ux : 0.0;
        v[QY][col] = node ? m.rho * m.uy : 0.0;
        v[QD][col] = node ? m.rho : 0.0;
        v[QU][col] = node ? m.rE : 0.0;
        __syncwarp();
        const int k = lane >> 2, j = lane & 3;
        const double* w = v[k == 0 ? QD : k == 1 ? QX : k == 2 ? QY : QU] + 1 + j;
        double t = ((w[0] + w[4]) + (w[8] + w[12])) + ((w[16] + w[20]) + (w[24] + w[28]));
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if (k < 5 && j == 0) partials[5 * blockIdx.x + k] = k == 3 ? 0.0 : t;
    }
}
#endif

// Persistent D2Q9 ensemble step: the tiles of all instances form one work list
// (instance k owns tiles [tile_start[k], tile_start[k+1]), tiles_x[k] per row); CTA
// b processes tiles b, b + gridDim.x, ...  Instance k's populations start at element
// offset[k] of both stores; its parameters are params[k].  No totals are kept.
template <int TY, bool CAL>
__global__ void __launch_bounds__(TX * TY)
ensemble2d_kernel(const EnsembleArgs a, const P* src, P* __restrict__ dst, int* __restrict__ status) {
    wait_for_previous();
    __shared__ int s_start[kMaxEnsemble + 1];
    __shared__ int s_tx[kMaxEnsemble];
    const int tid = threadIdx.x + TX * threadIdx.y;
    for (int k = tid; k <= a.n; k += TX * TY) s_start[k] = a.tile_start[k];
    for (int k = tid; k < a.n; k += TX * TY) s_tx[k] = a.tiles_x[k];
    __syncthreads();
    int k = 0;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        while (t >= s_start[k + 1]) ++k;   // t increases, so k only moves forward
        const int local = t - s_start[k];
        const int bx = local % s_tx[k], by = local / s_tx[k];
        const long long off = a.offset[k];
        fused2d_tile<TY, CAL, false>(a.params[k], src + off, dst + off, bx, by, nullptr, status);
    }
}

// Q~_zzz of the node (x, y, z) by a direct gather (used once per z segment).
template <bool CAL>
__device__ __forceinline__ R direct_anomaly_z(const KParams& p, const P* __restrict__ src, int x, int y, int z) {
    PullRows r;
    pull_rows(p, x, y, z, r);
    R f[Q], g[Q];
    gather(p, src, r, f, g);
    Moments<R> m;
    node_moments<kD, R, false, DEV, CAL>(f, g, p, m);
    return anomaly(m.rho, m.uz, m.T);
}

// D3Q27, pipelined.  A CTA owns a TX x TY column of nodes and marches along z over a
// segment of p.tz planes.  For every plane q it needs the pulled pairs of its TX*TY
// nodes and of the 2TX+2TY halo nodes; these are copied with cp.async into one of
// two shared-memory plane buffers, laid out [direction][slot].  Thread t copies and
// reads only its own slots (its node, and halo node t for t < 2TX+2TY), so the
// population buffers need no barrier: each thread waits for its own copies.  Only
// the Q~ arrays (double-buffered by plane parity) are shared, and one barrier per
// plane orders both of their hazards.  Per plane z:
//   wait for this thread's copies of plane z+1; barrier;
//   moments of plane z+1 (tile and halo) -> Q~ in shared memory, moments kept in
//       registers for the next iteration;
//   read the pairs of plane z from shared memory, prefetch plane z+2 into the same
//       slots;
//   collide plane z (moments and Q~ from the previous iteration, the rolling Q~_zzz
//       registers) and store.
// Every population leaves HBM once per step; the collision overlaps the prefetch.
template <int TY, int NB>
struct Pipe {
    static constexpr int NT = TX * TY;
    static constexpr int NH = 2 * TX + 2 * TY;
    static constexpr int NS = NT + NH;
    static constexpr size_t buf_bytes = (size_t)NB * Q * NS * sizeof(P);
    static constexpr size_t q_bytes = (size_t)2 * (TY * (TX + 2) + (TY + 2) * TX) * sizeof(R);
    static constexpr size_t smem_bytes = buf_bytes + q_bytes;
};

// Base of every direction plane of the source and destination stores, computed on the
// host: the kernel then forms each population address as one 32-bit node offset added
// to a base read from the parameter bank, instead of a 64-bit i * N product per access.
struct DirPlanes {
    const P* src[Q];
    P* dst[Q];
};
__device__ __forceinline__ const P* dir_src(const DirPlanes& pl, const PullRows& r, int i) {
    const int a = i % 3, b = (i / 3) % 3, c = (kD == 3) ? i / 9 : 1;
    return pl.src[i] + (unsigned)(r.row[b][c] + r.xs[a]);
}

// AA single store (src = dst): direction j's pair where direction k is pulled from.
__device__ __forceinline__ P* aa_slot(const DirPlanes& pl, const PullRows& r, int j, int k) {
    const int a = k % 3, b = (k / 3) % 3, c = (kD == 3) ? k / 9 : 1;
    return pl.dst[j] + (unsigned)(r.row[b][c] + r.xs[a]);
}

template <int TY, int NB>
struct PipeBytes {
    static constexpr size_t value = Pipe<TY, NB>::smem_bytes;
};

// Q~ of the nodes at the faces of the fused kernel's tiles and segments, where other CTAs of
// the in-place march read it: Q~_yyy in the first and last row of every tile, Q~_xxx in its first
// and last column, Q~_zzz in the first and last plane of every segment (30 % of the nodes with 32
// x 8 tiles).  The columns touch a line of 128 bytes in every 16 (FP32) or 32 nodes, so this reads
// about the whole store, at the memory's rate: 256^3 FP32 2.9 GB of DRAM reads from L0 (0.41 ms) and 4.1 from
// L1 (0.57), FP16 1.95 (0.28), of stores of 3.6 and 1.8 GB.  Rows and columns of a plane
// are adjacent CTAs, whose shared lines come from memory once.
struct AaEdges {
    int tx, ty, tz;               // tile and segment
    int nr, nc, ns;               // rows, columns, planes of the three sets
    unsigned br, bc;              // CTAs of a plane's rows and columns
};
template <bool FROM_L1>
__global__ void __launch_bounds__(kThreads1D)
aa_edges_kernel(const __grid_constant__ KParams p, const __grid_constant__ AaEdges e, P* A, R* __restrict__ qf) {
    wait_for_previous();
    // entry k of the set 0 | t - 1, t | 2 t - 1, 2 t | ... | n - 1
    auto member = [](int k, int t, int n) { return k % 2 == 0 ? k / 2 * t : min((k + 1) / 2 * t, n) - 1; };
    const unsigned per = e.br + e.bc, pz = blockIdx.x / per;
    int x, y, z = p.nz, comp;
    if (pz < (unsigned)p.nz) {
        unsigned k = blockIdx.x - pz * per;
        comp = k < e.br ? 1 : 0;
        k = (comp ? k : k - e.br) * kThreads1D + threadIdx.x;
        const unsigned w = comp ? p.nx : e.nc, line = k / w;
        if (comp) {
            x = (int)(k - line * w);
            y = member((int)line, e.ty, p.ny);
        } else {
            x = member((int)(k - line * w), e.tx, p.nx);
            y = (int)line;
        }
        if (line < (unsigned)(comp ? e.nr : p.ny)) z = (int)pz;
    } else {
        const long long k = (long long)(blockIdx.x - per * (unsigned)p.nz) * kThreads1D + threadIdx.x, line = k / p.nx;
        x = (int)(k - line * p.nx);
        const int q = (int)(line / p.ny);
        y = (int)(line - (long long)q * p.ny);
        if (q < e.ns) z = member(q, e.tz, p.nz);
        comp = 2;
    }
    if (z < p.nz) {
        const long long n = node_index(p, x, y, z);
        PullRows r;
        if (!FROM_L1) pull_rows(p, x, y, z, r);
        R f[Q], g[Q];
        aa_gather<FROM_L1>(p, A, r, n, f, g);
        Moments<R> m;
        node_moments<kD, R, false, DEV>(f, g, p, m);
        qf[(long long)comp * p.N + n] = anomaly(m.rho, comp == 0 ? m.ux : comp == 1 ? m.uy : m.uz, m.T);
    }
    launch_dependents();
}

// Store of a post-collision pair.  With ELBM_STCS the store is marked streaming (evict
// first), so that the step's writes do not push the planes prefetched ahead out of L2.
#ifndef ELBM_STCS
#define ELBM_STCS 1
#endif
__device__ __forceinline__ void store_pair(P* ptr, P v) {
    if constexpr (ELBM_STCS && sizeof(P) <= 8) __stcs(ptr, v);
    else *ptr = v;
}

// L2 prefetch of one box of a direction plane through the tensor-copy unit (no shared
// memory, no L1; a hint: boxes that leave the tensor are clipped).  x * element size
// must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int x, int y, int w) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];\n" ::"l"(
                     reinterpret_cast<unsigned long long>(map)),
                 "r"(x), "r"(y), "r"(w)
                 : "memory");
}

// AA = 1, 2: the same march in place on the AA single store (pl.src = pl.dst), from layout L0 or
// L1.  A node's slots are read and written by its own thread alone, so what the kernel may not do
// is read other CTAs' nodes: Q~ of the halo ring and of the planes on either side of the segment
// comes from qf, where aa_edges_kernel put it before.
template <int TY, int NB, int MINB, bool EARLY, int DD, bool CAL, int AA>
__global__ void __launch_bounds__(TX * TY, MINB)
fused3d_kernel(const __grid_constant__ KParams p, const __grid_constant__ DirPlanes pl,
               const P* src, double* __restrict__ partials, int* __restrict__ status,
               const __grid_constant__ CUtensorMap pmap, int pref, const R* qf) {
    using PP = Pipe<TY, NB>;
    static_assert(NB == 2, "plane z+2 is prefetched into the slots of plane z");
    static_assert(sizeof(R) == 4 && DD == 3, "the pipelined kernel is D3Q27 in FP32");
    constexpr int NT = PP::NT, NH = PP::NH, NS = PP::NS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    P* buf = reinterpret_cast<P*>(smem_raw);                       // [NB][Q][NS]
    R* qxs = reinterpret_cast<R*>(smem_raw + PP::buf_bytes);       // [2][TY][TX+2]
    R* qys = qxs + 2 * TY * (TX + 2);                              // [2][TY+2][TX]
    auto QX = [&](int b, int row, int col) -> R& { return qxs[(b * TY + row) * (TX + 2) + col]; };
    auto QY = [&](int b, int row, int col) -> R& { return qys[(b * (TY + 2) + row) * TX + col]; };

    wait_for_previous();
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + TX * ty;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zb = blockIdx.z * p.tz, ze = min(zb + p.tz, p.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < p.nx && y < p.ny;
    const int xl = min(x0 + TX, p.nx) - 1 - x0, yl = min(y0 + TY, p.ny) - 1 - y0;

    // this thread's halo node (if any) is fixed for the whole segment
    int hx = 0, hy = 0, hsx = 0, hsy = 0, haxis = 0;
    const bool has_halo = tid < NH && halo_node<TY>(p, tid, x0, y0, xl, yl, hx, hy, hsx, hsy, haxis);

    // copies of plane q (already mapped) into buffer sb
    auto issue_plane = [&](int q, int sb, bool with_halo) {
        P* bb = buf + (size_t)sb * Q * NS;
        if (active) {
            if constexpr (AA == 2) {
                const unsigned n = (unsigned)node_index(p, x, y, q);
#pragma unroll
                for (int i = 0; i < Q; ++i) cp_async<sizeof(P)>(bb + i * NS + tid, pl.src[i] + n);
            } else {
                PullRows r;
                pull_rows(p, x, y, q, r);
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    cp_async<sizeof(P)>(bb + i * NS + tid, AA ? aa_slot(pl, r, opp(i), i) : dir_src(pl, r, i));
            }
        }
        if (AA == 0 && with_halo && has_halo) {
            PullRows r;
            pull_rows(p, hx, hy, q, r);
#pragma unroll
            for (int i = 0; i < Q; ++i) cp_async<sizeof(P)>(bb + i * NS + NT + tid, dir_src(pl, r, i));
        }
        cp_async_commit();
    };
    // moments of the node in slot `slot` of buffer sb (the pressure tensor only for
    // tile nodes: halo nodes contribute Q~ alone)
    auto slot_moments = [&](int sb, int slot, Moments<R>& m, auto full) {
        const P* bb = buf + (size_t)sb * Q * NS + slot;
        if constexpr (DEV) {   // sums straight from the stored pairs
            node_moments_stored<kD, kST, decltype(full)::value, CAL>([&](int i) { return bb[i * NS]; }, p, m);
        } else {
            R f[Q], g[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) Cd::dec(bb[i * NS], f[i], g[i]);
            node_moments<kD, R, decltype(full)::value, DEV, CAL>(f, g, p, m);
        }
    };
    using Full = std::true_type;
    using Lite = std::false_type;
    // pref > 0: plane q's pulled source windows are prefetched into L2 `pref` planes
    // before their cp.async copies are issued (one tensor-prefetch box per direction,
    // issued by lanes of the last warp, which has no halo work), so that the copies of
    // the plane buffer find their lines in L2.  The box for direction i (pmap: TX x TY+2
    // pairs) covers the tile's own columns x0 .. x0 + TX - 1 and rows y0 - 1 - c_y ..
    // y0 + TY - c_y of source plane q - c_z.  The columns the pulls take beyond the tile
    // (x0 - 1 - c_x, x0 + TX - c_x) are left to the neighbouring tiles' boxes: a box
    // widened to them must start on a 16-byte boundary and then carries whole lines of
    // the neighbours' columns, which in FP32 cost 15 % more DRAM reads and 11 % of the step.
    const int pf_lane = tid - (NT - 32);
    auto prefetch_plane = [&](int q) {
        if (AA && pf_lane >= 0 && pf_lane < Q) {   // box TX x TY: the tile's rows where they are pulled from
            const int i = pf_lane, b = (i / 3) % 3, c = i / 9;
            if (AA == 2) tma_prefetch_3d(&pmap, x0, y0, i * p.nz + q);
            else tma_prefetch_3d(&pmap, x0, max(y0 + 1 - b, 0), opp(i) * p.nz + map_axis(q + 1 - c, p.nz, p.per_z));
            return;
        }
        if (pf_lane >= 0 && pf_lane < Q) {
            const int i = pf_lane, b = (i / 3) % 3, c = i / 9;
            // x0 is a multiple of TX (x0 * pair size a multiple of 16 bytes); rows clamped
            tma_prefetch_3d(&pmap, x0, max(y0 - b, 0), i * p.nz + map_axis(q + 1 - c, p.nz, p.per_z));
        }
    };

    Acc5 acc;
    acc.zero();
    bool bad = false;

    // prologue: Q~_zzz below the segment, planes zb and zb+1 in flight, moments of zb
    R qz_prev = R(0), qz_cur = R(0), qz_next = R(0);
    // AA: Q~ at this thread's node or halo node of a plane, from qf
    auto field_qz = [&](int q) { return qf[2 * p.N + node_index(p, x, y, map_axis(q, p.nz, p.per_z))]; };
    auto field_halo = [&](int q) { return qf[(haxis == 1 ? p.N : 0) + node_index(p, hx, hy, q)]; };
    const int zt = AA ? ze - 1 : ze;   // last plane whose pairs are needed
    if (active) {
        if constexpr (AA) qz_prev = field_qz(zb - 1);
        else qz_prev = direct_anomaly_z<CAL>(p, src, x, y, map_axis(zb - 1, p.nz, p.per_z));
    }
    for (int d = 2; d < 2 + pref && zb + d <= zt; ++d) prefetch_plane(map_axis(zb + d, p.nz, p.per_z));
    issue_plane(zb, 0, true);
    if (zb + 1 <= zt) issue_plane(map_axis(zb + 1, p.nz, p.per_z), 1 % NB, zb + 1 < ze);
    else cp_async_commit();
    Moments<R> m_cur, m_next;
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    if (active) {
        slot_moments(0, tid, m_cur, Full());
        QX(0, ty, tx + 1) = anomaly(m_cur.rho, m_cur.ux, m_cur.T);
        QY(0, ty + 1, tx) = anomaly(m_cur.rho, m_cur.uy, m_cur.T);
        qz_cur = anomaly(m_cur.rho, m_cur.uz, m_cur.T);
    }
    auto put_halo = [&](int b, R q) {
        if (haxis == 1) QY(b, hsy, hsx) = q;
        else QX(b, hsy, hsx) = q;
    };
    // Q~ of a halo node, below: the two forms round differently, and either kind of store keeps the bits that
    // it has had; the shorter one is also the faster in FP32 (256^3 1245 us a step, 1261 with the other).
    if (has_halo) {
        if constexpr (AA) {
            put_halo(0, field_halo(zb));
        } else {
            Moments<R> hm;
            slot_moments(0, NT + tid, hm, Lite());
            if constexpr (!DEV) put_halo(0, anomaly(hm.rho, haxis == 1 ? hm.uy : hm.ux, hm.T));
            else if (haxis == 1) QY(0, hsy, hsx) = anomaly(hm.rho, hm.uy, hm.T);
            else QX(0, hsy, hsx) = anomaly(hm.rho, hm.ux, hm.T);
        }
    }

    for (int z = zb; z < ze; ++z) {
        const int k = z - zb;
        const int bq = k & 1;               // Q~ buffer of plane z
        const int sz = k % NB;              // population buffer of plane z
        const int sn = (k + 1) % NB;        // ... of plane z+1
        const bool last = (z + 1 == ze);
        cp_async_wait_all();
        __syncthreads();

        // EARLY: plane z is read into registers and plane z+2 requested before the
        // moments of plane z+1, so the copy overlaps them too (both planes are live
        // in registers meanwhile, which only a one-CTA-per-SM launch affords)
        P pk[Q];   // the pulled pairs of plane z, as stored
        if (pref > 0 && z + 2 + pref <= zt) prefetch_plane(map_axis(z + 2 + pref, p.nz, p.per_z));
        if (EARLY) {
            if (active) {
                const P* bb = buf + (size_t)sz * Q * NS + tid;
#pragma unroll
                for (int i = 0; i < Q; ++i) pk[i] = bb[i * NS];
            }
            if (z + 2 <= zt) issue_plane(map_axis(z + 2, p.nz, p.per_z), sz, z + 2 < ze);
        }

        R halo_next = R(0);
        if (AA && !last && has_halo) halo_next = field_halo(z + 1);
        if (AA && last) {
            if (active) qz_next = field_qz(ze);
        } else if (active) {
            slot_moments(sn, tid, m_next, Full());
            qz_next = anomaly(m_next.rho, m_next.uz, m_next.T);
            if (!last) {
                QX(bq ^ 1, ty, tx + 1) = anomaly(m_next.rho, m_next.ux, m_next.T);
                QY(bq ^ 1, ty + 1, tx) = anomaly(m_next.rho, m_next.uy, m_next.T);
            }
        }
        if (!last && has_halo) {
            if constexpr (AA) {
                put_halo(bq ^ 1, halo_next);
            } else {
                Moments<R> hm;
                slot_moments(sn, NT + tid, hm, Lite());
                if constexpr (!DEV) put_halo(bq ^ 1, anomaly(hm.rho, haxis == 1 ? hm.uy : hm.ux, hm.T));
                else if (haxis == 1) QY(bq ^ 1, hsy, hsx) = anomaly(hm.rho, hm.uy, hm.T);
                else QX(bq ^ 1, hsy, hsx) = anomaly(hm.rho, hm.ux, hm.T);
            }
        }

        if (!EARLY) {
            if (active) {
                const P* bb = buf + (size_t)sz * Q * NS + tid;
#pragma unroll
                for (int i = 0; i < Q; ++i) pk[i] = bb[i * NS];
            }
            if (z + 2 <= zt) issue_plane(map_axis(z + 2, p.nz, p.per_z), sz, z + 2 < ze);
        }
        if (active) {
            bad |= nonphysical(m_cur);
            const R Dx = dQ(p.deriv, m_cur.ux, QX(bq, ty, tx), QX(bq, ty, tx + 1), QX(bq, ty, tx + 2));
            const R Dy = dQ(p.deriv, m_cur.uy, QY(bq, ty, tx), QY(bq, ty + 1, tx), QY(bq, ty + 2, tx));
            const R Dz = dQ(p.deriv, m_cur.uz, qz_prev, qz_cur, qz_next);
            R v[5];
            node_totals(m_cur, m_cur.rE, v);
            acc.add(v);
            // collide and store pair by pair, decoding each just before its update
            const unsigned n = (unsigned)node_index(p, x, y, z);
            PullRows w;   // AA from L0: the new pairs go to where opposite directions are pulled from
            if constexpr (AA == 1) pull_rows(p, x, y, z, w);
            auto out = [&](int i) { return AA == 0 ? pl.dst[i] + n : AA == 2 ? pl.dst[opp(i)] + n : aa_slot(pl, w, i, opp(i)); };
            Relax<kD, R, DEV, CAL> rx;
            rx.init(m_cur, Dx, Dy, Dz, p);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                R f, g;
                Cd::dec(pk[i], f, g);
                const float2 o = rx.fg(i, make_float2(f, g), p);
                store_pair(out(i), Cd::enc(o.x, o.y));
            }
        }
        m_cur = m_next;
        qz_prev = qz_cur;
        qz_cur = qz_next;
    }
    launch_dependents();
    cp_async_wait_all();
    flag_if(bad, status);
    R tot[5];
    acc.total(tot);
    block_sum5_warp(tot, partials + 5 * (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)));
}

// ---------------------------------------------------------------------------
// D3Q27 with tensor-copy (TMA) plane staging
// ---------------------------------------------------------------------------
// The tensor-copy engine (cp.async.bulk.tensor, the TMA unit) moves a box of a direction
// plane from global to shared memory; the copies of one plane count their bytes on an
// mbarrier, which the consuming threads wait on.
__device__ __forceinline__ unsigned smem_u32(const void* ptr) {
    return static_cast<unsigned>(__cvta_generic_to_shared(ptr));
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
// One arrival that also announces `bytes` of copies for the current phase.
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(bar),
                 "r"(bytes)
                 : "memory");
}
// One arrival, made when this thread's earlier cp.async copies have landed (counts as
// one of the arrivals the mbarrier was initialised with).
__device__ __forceinline__ void mbar_arrive_cp_async(unsigned bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}
// Waits for the phase of parity `parity` to complete, for at most about one second;
// false if it gave up.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try(bar, parity))
        if (global_ns() - t0 > 1000000000ull) return false;
    return true;
}
// Box {x, y, w} of a rank-3 tensor map into shared memory (128-byte aligned), completing
// on the mbarrier.  x * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int x, int y, int w,
                                            unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(w), "r"(bar)
        : "memory");
}

// Shared-memory plan of the TMA-staged kernel.  For every direction i the buffer of
// plane q holds a box of RB rows x BW columns of the SOURCE plane q - c_z: rows
// y0 - 1 - c_y ... y0 + TY - c_y and columns x0 - XO ... x0 + TX + XO - 1, so that node
// (x, y) of the tile and its halo ring finds its pulled pair of direction i at box row
// y - y0 + 1 and column x - x0 + XO - c_x (one box element per destination node and
// direction).  XO keeps the box's first column 16-byte aligned; each box starts on a
// 128-byte boundary (BOXP elements apart).
template <int TY>
struct Tma {
    static constexpr int XO = 16 / (int)sizeof(P);
    static constexpr int BW = TX + 2 * XO;
    static constexpr int RB = TY + 2;
    static constexpr int BOX = RB * BW;
    static constexpr int BOXP = ((BOX * (int)sizeof(P) + 127) / 128) * 128 / (int)sizeof(P);
    static constexpr unsigned plane_bytes = (unsigned)(Q * BOX * sizeof(P));   // bytes the 27 boxes deliver
    static constexpr size_t buf_bytes = (size_t)2 * Q * BOXP * sizeof(P);
    static constexpr size_t q_bytes = (size_t)2 * (TY * (TX + 2) + (TY + 2) * TX) * sizeof(R);
    static constexpr size_t smem_bytes = buf_bytes + q_bytes + 2 * sizeof(unsigned long long);
};

// D3Q27, pipelined on tensor copies.  The same march as fused3d_kernel (a TX x TY
// column over a z segment, two plane buffers, plane z+2 requested while plane z+1's
// moments and plane z's collision run), with a plane's arrival counted on one mbarrier.
// A CTA whose boxes lie inside the grid for every direction requests a plane as 27
// tensor copies (one box per direction, issued by six threads of each of warps 3..7)
// and one thread announces their bytes; a CTA at an x or y face, where a box would wrap
// around a periodic axis or clamp at a zero-gradient one, copies each pulled pair with
// cp.async into the same box positions (the boundary map resolves the source), and each
// thread arrives when its copies have landed.  Per plane z:
//   wait for plane z+1's phase; read the pairs of plane z into registers; barrier
//   (every thread has read plane z's buffer; the Q~ arrays are free); request plane
//   z+2 into plane z's buffer; moments of plane z+1 (tile and halo) -> Q~; collide
//   plane z and store.
// A wait that gives up (about one second) latches kStatusTimeoutBit, and the CTA stops
// after waiting, again bounded, for the copies it still has in flight.
// A selectable schedule: at 256^3 it runs level with fused3d_kernel (within 1 %).  It
// executes fewer instructions and waits far less at the plane barrier, but the boxes
// carry 11-19 % more pairs than the pulls use (corners, and the columns that keep the
// box 16-byte aligned) and the kernel draws 12-25 % more DRAM reads.
#ifndef ELBM_PREF_TMA
#define ELBM_PREF_TMA 0   // measured: FP32 11.16 -> 10.95 GLUPS with it at 256^3, FP16 19.3 -> 19.5
#endif
constexpr bool kPrefTma = ELBM_PREF_TMA;

template <int TY, int MINB, int DD, bool CAL>
__global__ void __launch_bounds__(TX * TY, MINB)
fused3d_tma_kernel(const __grid_constant__ KParams p, const __grid_constant__ DirPlanes pl,
                   const __grid_constant__ CUtensorMap tmap, const P* src,
                   double* __restrict__ partials, int* __restrict__ status) {
    using TT = Tma<TY>;
    static_assert(sizeof(R) == 4 && DD == 3, "the TMA-staged kernel is D3Q27 in FP32 arithmetic");
    constexpr int NT = TX * TY, NH = 2 * TX + 2 * TY, XO = TT::XO, BW = TT::BW, BOXP = TT::BOXP;
    static_assert(NT >= 96 + 5 * 32, "tensor copies are issued by warps 3..7");
    extern __shared__ __align__(128) unsigned char tma_smem[];   // tensor-copy destinations: 128-byte aligned
    P* buf = reinterpret_cast<P*>(tma_smem);                                // [2][Q][BOXP]
    R* qxs = reinterpret_cast<R*>(tma_smem + TT::buf_bytes);                // [2][TY][TX+2]
    R* qys = qxs + 2 * TY * (TX + 2);                                       // [2][TY+2][TX]
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(tma_smem + TT::buf_bytes + TT::q_bytes);
    auto QX = [&](int b, int row, int col) -> R& { return qxs[(b * TY + row) * (TX + 2) + col]; };
    auto QY = [&](int b, int row, int col) -> R& { return qys[(b * (TY + 2) + row) * TX + col]; };

    wait_for_previous();
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + TX * ty;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zb = blockIdx.z * p.tz, ze = min(zb + p.tz, p.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < p.nx && y < p.ny;
    const int xl = min(x0 + TX, p.nx) - 1 - x0, yl = min(y0 + TY, p.ny) - 1 - y0;
    const int nslot = (ty + 1) * BW + tx + XO;   // this node in a direction's box (before -c_x)
    // every box of this CTA inside the grid: columns x0 - XO .. x0 + TX + XO - 1, rows
    // y0 - 2 .. y0 + TY + 1 (the union over c_y)
    const bool boxed = x0 >= XO && x0 + TX + XO <= p.nx && y0 >= 2 && y0 + TY + 1 < p.ny;

    // this thread's halo node: its box position is the unmapped one, or, beyond a
    // zero-gradient face, that of the clamped node it copies (whose pairs the tile node
    // there already brings: such a halo thread copies nothing)
    int hx = 0, hy = 0, hsx = 0, hsy = 0, haxis = 0, hslot = 0;
    const bool has_halo = tid < NH && halo_node<TY>(p, tid, x0, y0, xl, yl, hx, hy, hsx, hsy, haxis);
    bool halo_copies = false;
    if (has_halo) {
        const int ux = haxis == 1 ? x0 + hsx : x0 + hsx - 1;
        const int uy = haxis == 1 ? y0 + hsy - 1 : y0 + hsy;
        const bool clamped = (ux < 0 || ux >= p.nx) ? !p.per_x : ((uy < 0 || uy >= p.ny) ? !p.per_y : false);
        halo_copies = !clamped;
        hslot = ((clamped ? hy : uy) - y0 + 1) * BW + ((clamped ? hx : ux) - x0 + XO);
    }

    unsigned issued = 0u;   // planes requested per buffer: buffer 0 in the low half, 1 in the high
    auto issue_plane = [&](int q, int sb) {
        const unsigned bar = smem_u32(&bars[sb]);
        issued += sb ? 0x10000u : 1u;
        P* bb = buf + (size_t)sb * Q * BOXP;
        if (boxed) {
            if (tid == 0) mbar_expect_tx(bar, TT::plane_bytes + p.inject_tx);
            const int w = (tid >> 5) - 3, lane = tid & 31;
            if (w >= 0 && lane < 6 && 6 * w + lane < Q) {
                const int i = 6 * w + lane;
                const int b = (i / 3) % 3, c = i / 9;
                const int zs = map_axis(q + 1 - c, p.nz, p.per_z);   // q - c_z
                tma_load_3d(smem_u32(bb + (size_t)i * BOXP), &tmap, x0 - XO, y0 - b, i * p.nz + zs, bar);
            }
        } else {
            if (active) {
                PullRows r;
                pull_rows(p, x, y, q, r);
#pragma unroll
                for (int i = 0; i < Q; ++i) cp_async<sizeof(P)>(bb + i * BOXP + nslot - cx_of(i), dir_src(pl, r, i));
            }
            if (halo_copies) {
                PullRows r;
                pull_rows(p, hx, hy, q, r);
#pragma unroll
                for (int i = 0; i < Q; ++i) cp_async<sizeof(P)>(bb + i * BOXP + hslot - cx_of(i), dir_src(pl, r, i));
            }
            mbar_arrive_cp_async(bar);
        }
    };
    auto slot_moments = [&](int sb, int slot, Moments<R>& m, auto full) {
        const P* bb = buf + (size_t)sb * Q * BOXP + slot;
        if constexpr (DEV) {   // sums straight from the stored pairs
            node_moments_stored<kD, kST, decltype(full)::value, CAL>([&](int i) { return bb[i * BOXP - cx_of(i)]; },
                                                                       p, m);
        } else {
            R f[Q], g[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) Cd::dec(bb[i * BOXP - cx_of(i)], f[i], g[i]);
            node_moments<kD, R, decltype(full)::value, DEV, CAL>(f, g, p, m);
        }
    };
    using Full = std::true_type;
    using Lite = std::false_type;

    if (tid == 0) {
        mbar_init(smem_u32(&bars[0]), boxed ? 1 : NT);
        mbar_init(smem_u32(&bars[1]), boxed ? 1 : NT);
    }
    __syncthreads();

    Acc5 acc;
    acc.zero();
    bool bad = false, late = false;

    // prologue: Q~_zzz below the segment, planes zb and zb+1 in flight, moments of zb
    R qz_prev = R(0), qz_cur = R(0), qz_next = R(0);
    if (active) qz_prev = direct_anomaly_z<CAL>(p, src, x, y, map_axis(zb - 1, p.nz, p.per_z));
    // L2 prefetch of the plane after the two in flight, by lanes of the last warp, one
    // staging box per direction (ELBM_PREF_TMA, off by default)
    const int pf_lane = tid - (NT - 32);
    auto prefetch_plane = [&](int q) {
        if (kPrefTma && pf_lane >= 0 && pf_lane < Q) {
            const int i = pf_lane, b = (i / 3) % 3, c = i / 9;
            tma_prefetch_3d(&tmap, max(x0 - XO, 0), max(y0 - b, 0), i * p.nz + map_axis(q + 1 - c, p.nz, p.per_z));
        }
    };
    if (zb + 2 <= ze) prefetch_plane(map_axis(zb + 2, p.nz, p.per_z));
    issue_plane(zb, 0);
    issue_plane(map_axis(zb + 1, p.nz, p.per_z), 1);
    Moments<R> m_cur, m_next;
    late |= !mbar_wait(smem_u32(&bars[0]), 0);
    if (active) {
        slot_moments(0, nslot, m_cur, Full());
        QX(0, ty, tx + 1) = anomaly(m_cur.rho, m_cur.ux, m_cur.T);
        QY(0, ty + 1, tx) = anomaly(m_cur.rho, m_cur.uy, m_cur.T);
        qz_cur = anomaly(m_cur.rho, m_cur.uz, m_cur.T);
    }
    if (has_halo) {
        Moments<R> hm;
        slot_moments(0, hslot, hm, Lite());
        if (haxis == 1) QY(0, hsy, hsx) = anomaly(hm.rho, hm.uy, hm.T);
        else QX(0, hsy, hsx) = anomaly(hm.rho, hm.ux, hm.T);
    }

    bool gave_up = false;
    for (int z = zb; z < ze; ++z) {
        const int k = z - zb;
        const int sz = k & 1, sn = sz ^ 1;   // buffers (and Q~ arrays) of planes z and z+1
        const bool last = (z + 1 == ze);
        late |= !mbar_wait(smem_u32(&bars[sn]), ((k + 1) >> 1) & 1);
        P pk[Q];   // the pulled pairs of plane z, as stored
        if (active) {
            const P* bb = buf + (size_t)sz * Q * BOXP + nslot;
#pragma unroll
            for (int i = 0; i < Q; ++i) pk[i] = bb[i * BOXP - cx_of(i)];
        }
        if (__syncthreads_or(late)) {
            gave_up = true;
            break;
        }
        if (z + 3 <= ze) prefetch_plane(map_axis(z + 3, p.nz, p.per_z));
        if (z + 2 <= ze) issue_plane(map_axis(z + 2, p.nz, p.per_z), sz);

        if (active) {
            slot_moments(sn, nslot, m_next, Full());
            qz_next = anomaly(m_next.rho, m_next.uz, m_next.T);
            if (!last) {
                QX(sn, ty, tx + 1) = anomaly(m_next.rho, m_next.ux, m_next.T);
                QY(sn, ty + 1, tx) = anomaly(m_next.rho, m_next.uy, m_next.T);
            }
        }
        if (!last && has_halo) {
            Moments<R> hm;
            slot_moments(sn, hslot, hm, Lite());
            if (haxis == 1) QY(sn, hsy, hsx) = anomaly(hm.rho, hm.uy, hm.T);
            else QX(sn, hsy, hsx) = anomaly(hm.rho, hm.ux, hm.T);
        }
        if (active) {
            bad |= nonphysical(m_cur);
            const R Dx = dQ(p.deriv, m_cur.ux, QX(sz, ty, tx), QX(sz, ty, tx + 1), QX(sz, ty, tx + 2));
            const R Dy = dQ(p.deriv, m_cur.uy, QY(sz, ty, tx), QY(sz, ty + 1, tx), QY(sz, ty + 2, tx));
            const R Dz = dQ(p.deriv, m_cur.uz, qz_prev, qz_cur, qz_next);
            R v[5];
            node_totals(m_cur, m_cur.rE, v);
            acc.add(v);
            const unsigned n = (unsigned)node_index(p, x, y, z);
            Relax<kD, R, DEV, CAL> rx;
            rx.init(m_cur, Dx, Dy, Dz, p);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                R f, g;
                Cd::dec(pk[i], f, g);
                const float2 o = rx.fg(i, make_float2(f, g), p);
                store_pair(pl.dst[i] + n, Cd::enc(o.x, o.y));
            }
        }
        m_cur = m_next;
        qz_prev = qz_cur;
        qz_cur = qz_next;
    }
    launch_dependents();
    if (gave_up) {
        // the last phase of each buffer may still have copies in flight
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const unsigned n = b ? issued >> 16 : issued & 0xffffu;
            if (n) mbar_wait(smem_u32(&bars[b]), (n - 1) & 1);
        }
        if (tid == 0) atomicOr(status, kStatusTimeoutBit);
    }
    cp_async_wait_all();
    flag_if(bad, status);
    R tot[5];
    acc.total(tot);
    block_sum5_warp(tot, partials + 5 * (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)));
}

// D3Q27 without plane buffers: for plane z it computes Q~ of plane z+1 (tile + halo)
// from a first gather, then gathers plane z again (an L2 hit) to collide it.
template <int TY, bool CAL>
__global__ void __launch_bounds__(TX * TY, 2)
fused3d_reread_kernel(const __grid_constant__ KParams p, const P* src, P* __restrict__ dst,
                      double* __restrict__ partials, int* __restrict__ status) {
    wait_for_previous();
    __shared__ R qx[2][TY][TX + 2];
    __shared__ R qy[2][TY + 2][TX];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + TX * ty;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zb = blockIdx.z * p.tz, ze = min(zb + p.tz, p.nz);
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < p.nx && y < p.ny;
    const int xl = min(x0 + TX, p.nx) - 1 - x0, yl = min(y0 + TY, p.ny) - 1 - y0;
    int hx = 0, hy = 0, hsx = 0, hsy = 0, haxis = 0;
    const bool has_halo = tid < 2 * TX + 2 * TY && halo_node<TY>(p, tid, x0, y0, xl, yl, hx, hy, hsx, hsy, haxis);

    // Q~ of the tile and its halo in plane z -> buffer b; returns Q~_zzz of (x, y, z)
    auto plane_moments = [&](int z, int b, bool with_xy) -> R {
        R qz = R(0);
        if (active) {
            PullRows r;
            pull_rows(p, x, y, z, r);
            R f[Q], g[Q];
            gather(p, src, r, f, g);
            Moments<R> m;
            node_moments<kD, R, false, DEV, CAL>(f, g, p, m);
            if (with_xy) {
                qx[b][ty][tx + 1] = anomaly(m.rho, m.ux, m.T);
                qy[b][ty + 1][tx] = anomaly(m.rho, m.uy, m.T);
            }
            qz = anomaly(m.rho, m.uz, m.T);
        }
        if (with_xy && has_halo) {
            PullRows r;
            pull_rows(p, hx, hy, z, r);
            R f[Q], g[Q];
            gather(p, src, r, f, g);
            Moments<R> m;
            node_moments<kD, R, false, DEV, CAL>(f, g, p, m);
            if (haxis == 1) qy[b][hsy][hsx] = anomaly(m.rho, m.uy, m.T);
            else qx[b][hsy][hsx] = anomaly(m.rho, m.ux, m.T);
        }
        return qz;
    };

    Acc5 acc;
    acc.zero();
    bool bad = false;
    R qz_prev = plane_moments(map_axis(zb - 1, p.nz, p.per_z), 0, false);
    R qz_cur = plane_moments(zb, 0, true);
    for (int z = zb; z < ze; ++z) {
        const int b = (z - zb) & 1;
        const bool last = (z + 1 == ze);
        __syncthreads();   // buffer b^1 is free (collision of z-1 is done)
        const R qz_next = plane_moments(map_axis(z + 1, p.nz, p.per_z), b ^ 1, !last);
        __syncthreads();   // buffer b complete for plane z
        if (active) {
            PullRows r;
            pull_rows(p, x, y, z, r);
            R f[Q], g[Q];
            gather(p, src, r, f, g);
            Moments<R> m;
            node_moments<kD, R, true, DEV, CAL>(f, g, p, m);
            bad |= nonphysical(m);
            const R Dx = dQ(p.deriv, m.ux, qx[b][ty][tx], qx[b][ty][tx + 1], qx[b][ty][tx + 2]);
            const R Dy = dQ(p.deriv, m.uy, qy[b][ty][tx], qy[b][ty + 1][tx], qy[b][ty + 2][tx]);
            const R Dz = dQ(p.deriv, m.uz, qz_prev, qz_cur, qz_next);
            R v[5];
            node_totals(m, m.rE, v);
            acc.add(v);
            collide<kD, R, DEV, CAL>(f, g, m, Dx, Dy, Dz, p);
            store_node(p, dst, node_index(p, x, y, z), f, g);
        }
        qz_prev = qz_cur;
        qz_cur = qz_next;
    }
    launch_dependents();
    flag_if(bad, status);
    R tot[5];
    acc.total(tot);
    block_sum5_warp(tot, partials + 5 * (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)));
}

// ---------------------------------------------------------------------------
// D2Q9, row march
// ---------------------------------------------------------------------------
// The two-dimensional form of the pipelined D3Q27 kernel: a CTA of W threads owns a
// strip of W nodes of a row and marches along y over a segment of rows [y0, ye); the
// row plays the part of the plane.  For every row it needs the pulled pairs of its W
// nodes and of the two nodes at the strip's ends (the halo of the x derivative);
// they are copied with cp.async into one of two shared-memory row buffers one row ahead
// ([direction][slot], slot 0 the left end, 1..W the strip, W+1 or the ragged end + 1
// the right end).  Each thread copies and reads only its own slots; the Q~_xxx row
// (double-buffered by row parity) is the only shared array, so one barrier per row
// orders it.  Q~_yyy of the rows below, at and above the current one rolls in registers.
// Per row y: wait for this thread's copies of row y+1; barrier; read row y's pairs into
// registers and request row y+2 into their slots; moments of row y+1 (strip and ends)
// -> Q~ (registers kept for the next row); collide row y and store.  Every population
// leaves HBM once per step; a segment re-reads about two rows (the row below it and
// the row above it).
template <int W, int NB = 2>
struct March2 {
    static constexpr int NS = W + 2;
    static constexpr int NBUF = NB;   // row buffers: rows y (collide), y+1 (moments), up to y+NB-1 in flight
    static constexpr size_t buf_bytes = (size_t)NB * Q * NS * sizeof(P);
    static constexpr size_t q_bytes = (size_t)2 * NS * sizeof(R);
    static constexpr size_t smem_bytes = buf_bytes + q_bytes;
};

// Per-direction plane bases of one lattice's stores: from the kernel parameters (one
// lattice), or formed from the instance's base (ensemble).
struct PlanesParam {
    const DirPlanes* pl;
    const P* base;
    __device__ __forceinline__ const P* s(int i) const { return pl->src[i]; }
    __device__ __forceinline__ P* d(int i) const { return pl->dst[i]; }
};
struct PlanesBase {
    const P* src;
    P* dst;
    size_t N;
    const P* base;
    __device__ __forceinline__ const P* s(int i) const { return src + (size_t)i * N; }
    __device__ __forceinline__ P* d(int i) const { return dst + (size_t)i * N; }
};

// Q~_yyy of node (x, y) (y mapped) by a direct gather, with the fixed-state pairs where
// its pulls cross a fixed face (used once per segment).
template <bool CAL>
__device__ __forceinline__ R direct_anomaly_y(const KParams& p, const P* __restrict__ src, int x, int y) {
    PullRows r;
    pull_rows(p, x, y, 0, r);
    R f[Q], g[Q];
    gather(p, src, r, f, g);
    Moments<R> m;
    node_moments<kD, R, false, DEV, CAL>(f, g, p, m);
    return anomaly(m.rho, m.uy, m.T);
}

// FIX = false compiles the march for grids without fixed-state faces: the face tests and
// the per-direction substitutions fold away (FP16 store at 4096^2: 46.7 -> 50.0 GLUPS,
// 80 -> 72 registers, seven CTAs per SM instead of six).
template <int W, int NB, bool CAL, bool FIX, class PL>
__device__ __forceinline__ void march2d_segment(const KParams& p, const PL& pl, int x0, int y0, int ye,
                                                unsigned char* smem, Acc5& acc, bool& bad) {
    using MC = March2<W, NB>;
    static_assert(NB == 2 || NB == 3, "two or three row buffers");
    constexpr int NS = MC::NS;
    P* buf = reinterpret_cast<P*>(smem);                   // [NB][Q][NS]
    R* qxs = reinterpret_cast<R*>(smem + MC::buf_bytes);   // [2][NS]
    const int t = threadIdx.x;
    const int x = x0 + t;
    const bool active = x < p.nx;
    const int xl = min(x0 + W, p.nx) - 1 - x0;   // last local column of the strip
    const int nslot = t + 1;
    // the strip's ends: thread 0 the left one (slot 0), thread 1 the right one (slot xl + 2);
    // beyond a fixed-state face an end carries the fixed state's Q~ and is not copied
    const bool has_halo = t < 2;
    const int hux = t == 0 ? x0 - 1 : x0 + xl + 1;
    const int hx = map_axis(hux, p.nx, p.per_x);
    const bool fixed_faces = FIX && p.has_fixed;
    const bool hfixed = has_halo && fixed_faces && beyond_fixed(p, 0, hux, p.nx);
    const int hslot = t == 0 ? 0 : xl + 2;

    auto issue_row = [&](int yq, int sb, bool with_halo) {   // yq already mapped
        P* bb = buf + (size_t)sb * Q * NS;
        if (active) {
            PullRows r;
            pull_rows(p, x, yq, 0, r);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                cp_async<sizeof(P)>(bb + i * NS + nslot, pl.s(i) + (unsigned)(r.row[(i / 3) % 3][1] + r.xs[i % 3]));
        }
        if (with_halo && has_halo && !hfixed) {
            PullRows r;
            pull_rows(p, hx, yq, 0, r);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                cp_async<sizeof(P)>(bb + i * NS + hslot, pl.s(i) + (unsigned)(r.row[(i / 3) % 3][1] + r.xs[i % 3]));
        }
        cp_async_commit();
    };
    // moments of the node in slot `slot` of buffer sb; gm marks the pairs that are the
    // fixed state's (pulled across a fixed face)
    auto row_moments = [&](int sb, int slot, unsigned gm, Moments<R>& m, auto full) {
        const P* bb = buf + (size_t)sb * Q * NS + slot;
        R f[Q], g[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) Cd::dec(bb[i * NS], f[i], g[i]);
        if (gm) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if ((gm >> i) & 1u) fixed_pair(p, i, f[i], g[i]);
        }
        node_moments<kD, R, decltype(full)::value, DEV, CAL>(f, g, p, m);
    };
    using Full = std::true_type;
    using Lite = std::false_type;
    auto QX = [&](int b, int slot) -> R& { return qxs[b * NS + slot]; };
    auto halo_q = [&](int sb, int yq) {
        if (hfixed) return fixed_Q(p, 0);
        Moments<R> hm;
        row_moments(sb, hslot, fixed_mask<FIX>(p, hx, yq), hm, Lite());
        return anomaly(hm.rho, hm.ux, hm.T);
    };

    // prologue: Q~_yyy of the row below the segment, rows y0 and y0+1 in flight, moments of y0
    R qy_prev = R(0), qy_cur = R(0), qy_next = R(0);
    if (active) {
        if (fixed_faces && beyond_fixed(p, 1, y0 - 1, p.ny)) qy_prev = fixed_Q(p, 1);
        else qy_prev = direct_anomaly_y<CAL>(p, pl.base, x, map_axis(y0 - 1, p.ny, p.per_y));
    }
    // rows y0 .. y0+NB-1 in flight (a row past ye is not needed; its group stays empty)
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        if (y0 + j <= ye) issue_row(map_axis(y0 + j, p.ny, p.per_y), j, y0 + j < ye);
        else cp_async_commit();
    }
    Moments<R> m_cur, m_next;
    cp_async_wait_pending<NB - 1>();   // row y0 has landed
    __syncthreads();
    if (active) {
        row_moments(0, nslot, fixed_mask<FIX>(p, x, y0), m_cur, Full());
        QX(0, nslot) = anomaly(m_cur.rho, m_cur.ux, m_cur.T);
        qy_cur = anomaly(m_cur.rho, m_cur.uy, m_cur.T);
    }
    if (has_halo) QX(0, hslot) = halo_q(0, y0);

    for (int y = y0; y < ye; ++y) {
        const int k = y - y0;
        const int bq = k & 1;                          // Q~ row of y (y+1: bq ^ 1)
        const int sz = k % NB, sn = (k + 1) % NB;      // row buffers of rows y and y+1
        const bool last = (y + 1 == ye);
        cp_async_wait_pending<NB - 2>();               // row y+1 has landed (y+2.. may be in flight)
        __syncthreads();
        P pk[Q];   // the pulled pairs of row y, as stored
        if (active) {
            const P* bb = buf + (size_t)sz * Q * NS + nslot;
#pragma unroll
            for (int i = 0; i < Q; ++i) pk[i] = bb[i * NS];
        }
        if (y + NB <= ye) issue_row(map_axis(y + NB, p.ny, p.per_y), sz, y + NB < ye);
        else cp_async_commit();   // keep one group per row for the wait count

        const int yn = map_axis(y + 1, p.ny, p.per_y);
        if (active) {
            if (fixed_faces && beyond_fixed(p, 1, y + 1, p.ny)) {
                qy_next = fixed_Q(p, 1);   // the last row of the grid: nothing after it
            } else {
                row_moments(sn, nslot, fixed_mask<FIX>(p, x, yn), m_next, Full());
                qy_next = anomaly(m_next.rho, m_next.uy, m_next.T);
                if (!last) QX(bq ^ 1, nslot) = anomaly(m_next.rho, m_next.ux, m_next.T);
            }
        }
        if (!last && has_halo) QX(bq ^ 1, hslot) = halo_q(sn, yn);

        if (active) {
            bad |= nonphysical(m_cur);
            const R Dx = dQ(p.deriv, m_cur.ux, QX(bq, nslot - 1), QX(bq, nslot), QX(bq, nslot + 1));
            const R Dy = dQ(p.deriv, m_cur.uy, qy_prev, qy_cur, qy_next);
            R v[5];
            node_totals(m_cur, m_cur.rE, v);
            acc.add(v);
            Relax<kD, R, DEV, CAL> rx;
            rx.init(m_cur, Dx, Dy, R(0), p);
            const unsigned gm = fixed_mask<FIX>(p, x, y);
            const unsigned n = (unsigned)(x + p.nx * y);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                R f, g;
                Cd::dec(pk[i], f, g);
                if ((gm >> i) & 1u) fixed_pair(p, i, f, g);
                pl.d(i)[n] = Cd::enc(rx.f(i, f, p), rx.g(i, g, p));
            }
        }
        m_cur = m_next;
        qy_prev = qy_cur;
        qy_cur = qy_next;
    }
    cp_async_wait_all();
    __syncthreads();   // the shared buffers are reused by the next segment of a persistent CTA
}

// The same march for the 16-bit stores, which instruction issue bounds (615 instructions a
// node): a thread has the nodes x0 + 2t and x0 + 2t + 1, their arithmetic as two-lane FP32
// instructions (elbm_pair.cuh).  Both nodes' pairs lie side by side in a row buffer ([direction]
// [slot], slots 2t and 2t + 1, W and W + 1 the strip's ends), so one 8-byte access takes them out;
// where the stores' rows start on 8-byte boundaries (nx even) one 8-byte copy brings those of
// c_x = 0 in and one 8-byte store writes both.
#if ELBM_ST >= 2 && ELBM_D == 2
template <int W>
struct MarchPair {
    static constexpr int NT = W / 2, NS = W + 2, QW = W + 4;   // Q~_xxx: the strip from column 2 on, its ends beside it
    static constexpr size_t buf_bytes = ((size_t)2 * Q * NS * sizeof(P) + 15) / 16 * 16;
    static constexpr size_t smem_bytes = buf_bytes + (size_t)2 * QW * sizeof(float);
};
template <int W, bool CAL, bool FIX, class PL>
__device__ __forceinline__ void march2d_pair_segment(const KParams& p, const PL& pl, int x0, int y0, int ye,
                                                     unsigned char* smem, float2 acc[4], bool& bad) {
    using MC = MarchPair<W>;
    // Which of two products each sum of products rounds by itself (ALT) is that of the one-node march, bit
    // for bit: it differed between the lattice alone without fixed faces and the others, and
    // between a segment's first row and the rest (first).
    constexpr bool kAlone = !FIX && std::is_same<PL, PlanesParam>::value;
    using First = std::true_type;
    using Later = std::false_type;
    constexpr int NS = MC::NS, QW = MC::QW;
    P* buf = reinterpret_cast<P*>(smem);                            // [2][Q][NS]
    float* qxs = reinterpret_cast<float*>(smem + MC::buf_bytes);    // [2][QW]
    const int t = threadIdx.x, x = x0 + 2 * t;
    const bool act0 = x < p.nx, act1 = x + 1 < p.nx;
    const int xl = min(x0 + W, p.nx) - 1 - x0;   // last local column of the strip
    // rows of both stores on 8-byte boundaries
    const bool even = p.nx % 2 == 0 &&
                      ((reinterpret_cast<unsigned long long>(pl.s(0)) | reinterpret_cast<unsigned long long>(pl.d(0))) & 7) == 0;
    const bool has_halo = t < 2;
    const int hux = t == 0 ? x0 - 1 : x0 + xl + 1, hx = map_axis(hux, p.nx, p.per_x);
    const bool fixed_faces = FIX && p.has_fixed;
    const bool hfixed = has_halo && fixed_faces && beyond_fixed(p, 0, hux, p.nx);
    const int xm = map_axis(x - 1, p.nx, p.per_x), xp = map_axis(x + 1, p.nx, p.per_x);
    const int xq = act1 ? map_axis(x + 2, p.nx, p.per_x) : 0;

    auto issue_row = [&](int yq, int sb, bool with_halo) {   // yq already mapped
        P* bb = buf + (size_t)sb * Q * NS;
        const int row[3] = {p.nx * map_axis(yq + 1, p.ny, p.per_y), p.nx * yq, p.nx * map_axis(yq - 1, p.ny, p.per_y)};
        if (act0) {
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const int a = i % 3;
                const unsigned r = (unsigned)row[i / 3];
                P* d = bb + i * NS + 2 * t;
                const P* s = pl.s(i);
                if (a == 1 && even) {
                    cp_async<8>(d, s + (r + (unsigned)x));
                } else {
                    cp_async<4>(d, s + (r + (unsigned)(a == 0 ? xp : a == 1 ? x : xm)));
                    if (act1) cp_async<4>(d + 1, s + (r + (unsigned)(a == 0 ? xq : a == 1 ? x + 1 : x)));
                }
            }
        }
        if (with_halo && has_halo && !hfixed) {
            PullRows r;
            pull_rows(p, hx, yq, 0, r);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                cp_async<4>(bb + i * NS + W + t, pl.s(i) + (unsigned)(r.row[(i / 3) % 3][1] + r.xs[i % 3]));
        }
        cp_async_commit();
    };
    // one node's stored pairs, with the fixed state's in place of those marked in gm
    auto node_fixed = [&](const P* v, unsigned gm, Moments<float>& m) {
        if (!gm) {
            node_moments_stored<kD, kST, true, CAL>([&](int i) { return v[i * NS]; }, p, m);
            return;
        }
        float f[Q], g[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            Cd::dec(v[i * NS], f[i], g[i]);
            if ((gm >> i) & 1u) fixed_pair(p, i, f[i], g[i]);
        }
        node_moments<kD, float, true, true, CAL>(f, g, p, m);
    };
    auto pair_moments = [&](int sb, int y, MomentsPair& m, auto first) {
        const P* bb = buf + (size_t)sb * Q * NS + 2 * t;
        if (FIX) {
            const unsigned g0 = fixed_mask<FIX>(p, x, y), g1 = fixed_mask<FIX>(p, x + 1, y);
            if (g0 | g1) {
                Moments<float> a, b;
                node_fixed(bb, g0, a);
                node_fixed(bb + 1, g1, b);
                m.rho = make_float2(a.rho, b.rho);
                m.ux = make_float2(a.ux, b.ux);
                m.uy = make_float2(a.uy, b.uy);
                m.T = make_float2(a.T, b.T);
                m.rE = make_float2(a.rE, b.rE);
                m.Pxx = make_float2(a.Pxx, b.Pxx);
                m.Pyy = make_float2(a.Pyy, b.Pyy);
                m.Pxy = make_float2(a.Pxy, b.Pxy);
                return;
            }
        }
        uint2 raw[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) raw[i] = *reinterpret_cast<const uint2*>(bb + i * NS);
        node_moments_pair<kST, CAL, kAlone && (CAL || !decltype(first)::value)>(
            [&](int i, int k) { return *reinterpret_cast<const P*>(k ? &raw[i].y : &raw[i].x); }, p, m);
    };
    auto halo_q = [&](int sb, int y) {
        if (hfixed) return fixed_Q(p, 0);
        const P* bb = buf + (size_t)sb * Q * NS + W + t;
        Moments<float> m;
        const unsigned gm = fixed_mask<FIX>(p, hx, y);
        if (FIX && gm) node_fixed(bb, gm, m);
        else node_moments_stored<kD, kST, false, CAL>([&](int i) { return bb[i * NS]; }, p, m);
        return anomaly(m.rho, m.ux, m.T);
    };
    float* const my_qx = qxs + 2 + 2 * t;
    float* const halo_qx = qxs + (t == 0 ? 1 : xl + 3);
    // Q~ of this thread's nodes: xxx to shared memory row b, yyy returned
    auto put_q = [&](int b, const MomentsPair& m, bool x_too, auto first) {
        const float2 c = anomaly_c(m.T);
        if (x_too) {
            const float2 v = anomaly2<kAlone && !decltype(first)::value>(m.rho, m.ux, c);
            if (act1) *reinterpret_cast<float2*>(my_qx + b * QW) = v;
            else my_qx[b * QW] = v.x;
        }
        return anomaly2<kAlone && decltype(first)::value>(m.rho, m.uy, c);
    };

    float2 qy_prev = both(0.f), qy_cur = both(0.f), qy_next = both(0.f);
    if (act0) {
        if (fixed_faces && beyond_fixed(p, 1, y0 - 1, p.ny)) {
            qy_prev = both(fixed_Q(p, 1));
        } else {
            const int yd = map_axis(y0 - 1, p.ny, p.per_y);
            qy_prev.x = direct_anomaly_y<CAL>(p, pl.base, x, yd);
            if (act1) qy_prev.y = direct_anomaly_y<CAL>(p, pl.base, x + 1, yd);
        }
    }
    issue_row(y0, 0, true);
    issue_row(map_axis(y0 + 1, p.ny, p.per_y), 1, y0 + 1 < ye);
    MomentsPair m_cur, m_next;
    cp_async_wait_pending<1>();
    __syncthreads();
    if (act0) {
        pair_moments(0, y0, m_cur, First());
        qy_cur = put_q(0, m_cur, true, First());
    }
    if (has_halo) halo_qx[0] = halo_q(0, y0);

    for (int y = y0; y < ye; ++y) {
        const int bq = (y - y0) & 1, sn = bq ^ 1;   // buffers of rows y and y+1
        const bool last = y + 1 == ye;
        cp_async_wait_all();
        __syncthreads();
        uint2 pk[Q];   // the pulled pairs of row y, as stored
        if (act0) {
            const P* bb = buf + (size_t)bq * Q * NS + 2 * t;
#pragma unroll
            for (int i = 0; i < Q; ++i) pk[i] = *reinterpret_cast<const uint2*>(bb + i * NS);
        }
        if (y + 2 <= ye) issue_row(map_axis(y + 2, p.ny, p.per_y), bq, y + 2 < ye);
        const int yn = map_axis(y + 1, p.ny, p.per_y);
        if (act0) {
            if (fixed_faces && beyond_fixed(p, 1, y + 1, p.ny)) {
                qy_next = both(fixed_Q(p, 1));   // the last row of the grid: nothing after it
            } else {
                pair_moments(sn, yn, m_next, Later());
                qy_next = put_q(sn, m_next, !last, Later());
            }
        }
        if (!last && has_halo) halo_qx[sn * QW] = halo_q(sn, yn);
        if (act0) {
            auto bad_lane = [](float rho, float T, float ux, float uy) {
                return !(rho > 0.f) || !(T > 0.f) || !isfinite(rho) || !isfinite(T) || !isfinite(ux) || !isfinite(uy);
            };
            bad |= bad_lane(m_cur.rho.x, m_cur.T.x, m_cur.ux.x, m_cur.uy.x) ||
                   (act1 && bad_lane(m_cur.rho.y, m_cur.T.y, m_cur.ux.y, m_cur.uy.y));
            const float* qx = my_qx + bq * QW;
            const float2 q0 = *reinterpret_cast<const float2*>(qx);
            const float2 Dx = dQ2(p.deriv, m_cur.ux, make_float2(qx[-1], q0.x), q0, make_float2(q0.y, qx[2]));
            const float2 Dy = dQ2(p.deriv, m_cur.uy, qy_prev, qy_cur, qy_next);
            acc[0] = add2(acc[0], m_cur.rho);
            acc[1] = fma2(m_cur.rho, m_cur.ux, acc[1]);
            acc[2] = fma2(m_cur.rho, m_cur.uy, acc[2]);
            acc[3] = add2(acc[3], m_cur.rE);
            RelaxPair<CAL> rx;
            rx.init(m_cur, Dx, Dy, p);
            const unsigned n = (unsigned)(x + p.nx * y);
            const unsigned g0 = fixed_mask<FIX>(p, x, y), g1 = fixed_mask<FIX>(p, x + 1, y);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                float2 f, g;
                Cd::dec(*reinterpret_cast<const P*>(&pk[i].x), f.x, g.x);
                Cd::dec(*reinterpret_cast<const P*>(&pk[i].y), f.y, g.y);
                if ((g0 >> i) & 1u) fixed_pair(p, i, f.x, g.x);
                if ((g1 >> i) & 1u) fixed_pair(p, i, f.y, g.y);
                f = rx.f(i, f, p);
                g = rx.g(i, g, p);
                const P o0 = Cd::enc(f.x, g.x), o1 = Cd::enc(f.y, g.y);
                P* d = pl.d(i) + n;
                if (even) {
                    uint2 o;
                    o.x = *reinterpret_cast<const unsigned*>(&o0);
                    o.y = *reinterpret_cast<const unsigned*>(&o1);
                    *reinterpret_cast<uint2*>(d) = o;
                } else {
                    d[0] = o0;
                    if (act1) d[1] = o1;
                }
            }
        }
        m_cur = m_next;
        qy_prev = qy_cur;
        qy_cur = qy_next;
    }
    cp_async_wait_all();
    __syncthreads();   // the shared buffers are reused by the next segment of a persistent CTA
}
// Sixteen warps of 128 registers per SM (uncapped 145 registers, twelve warps: 4096^2 272 us a
// step, twenty warps: 598, it spills; strips of 128 nodes 269, 512 nodes 253, 256 nodes 249, all with
// an arithmetic that is not used any more, see elbm_pair.cuh).
template <int W> constexpr int kPairCtas = 1024 / W;
template <int W, bool CAL, bool FIX>
__global__ void __launch_bounds__(W / 2, kPairCtas<W>)
march2d_pair_kernel(const __grid_constant__ KParams p, const __grid_constant__ DirPlanes pl, const P* src,
                    double* __restrict__ partials, int* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    wait_for_previous();
    const int x0 = blockIdx.x * W, y0 = blockIdx.y * p.tz, ye = min(y0 + p.tz, p.ny);
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = both(0.f);
    bool bad = false;
    march2d_pair_segment<W, CAL, FIX>(p, PlanesParam{&pl, src}, x0, y0, ye, march_smem, acc, bad);
    launch_dependents();
    flag_if(bad, status);
    const bool act1 = x0 + 2 * (int)threadIdx.x + 1 < p.nx;
    auto lanes = [&](float2 a) { return act1 ? a.x + a.y : a.x; };
    float tot[5] = {lanes(acc[0]), lanes(acc[1]), lanes(acc[2]), 0.f, lanes(acc[3])};
    block_sum5_warp(tot, partials + 5 * (blockIdx.x + gridDim.x * blockIdx.y));
}
#endif

// One lattice: CTA (bx, by) marches strip bx over rows [by * p.tz, min((by + 1) * p.tz, ny)).
#ifndef ELBM_MARCH_MINB
#define ELBM_MARCH_MINB 0
#endif
#if ELBM_MARCH_MINB > 0
#define ELBM_MARCH_BOUNDS(W) __launch_bounds__(W, ELBM_MARCH_MINB)
#else
#define ELBM_MARCH_BOUNDS(W) __launch_bounds__(W)
#endif
template <int W, int NB, bool CAL, bool FIX>
__global__ void ELBM_MARCH_BOUNDS(W)
march2d_kernel(const __grid_constant__ KParams p, const __grid_constant__ DirPlanes pl, const P* src,
               double* __restrict__ partials, int* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    wait_for_previous();
    const int x0 = blockIdx.x * W, y0 = blockIdx.y * p.tz, ye = min(y0 + p.tz, p.ny);
    Acc5 acc;
    acc.zero();
    bool bad = false;
    march2d_segment<W, NB, CAL, FIX>(p, PlanesParam{&pl, src}, x0, y0, ye, march_smem, acc, bad);
    launch_dependents();
    flag_if(bad, status);
    R tot[5];
    acc.total(tot);
    block_sum5_warp(tot, partials + 5 * (blockIdx.x + gridDim.x * blockIdx.y));
}

// Compiled with and without fixed-state faces, as march2d_kernel (64 lattices, 8 steps: 7124 us with
// the face tests always in, 6506 without, both with segments of 32 rows).
// Persistent ensemble step on the row march: the work list holds (instance, strip, segment)
// units (instance order[k] owns units [tile_start[k], tile_start[k+1]), tiles_x[k] strips per
// segment row, the rows shared evenly between its segments); CTA b takes the b-th unit of every round
// of gridDim.x, counted from the end in every other round.  No totals are kept.
// Threads and shared memory of a march CTA: two nodes a thread for the 16-bit stores.
#if ELBM_ST >= 2 && ELBM_D == 2
template <int W, int NB> constexpr int march_threads = W / 2;
#define ELBM_ENSEMBLE_BOUNDS(W) __launch_bounds__(W / 2, kPairCtas<W>)
template <int W, int NB> constexpr size_t march_smem_bytes = MarchPair<W>::smem_bytes;
#else
template <int W, int NB> constexpr int march_threads = W;
#define ELBM_ENSEMBLE_BOUNDS(W) __launch_bounds__(W)
template <int W, int NB> constexpr size_t march_smem_bytes = March2<W, NB>::smem_bytes;
#endif
template <int W, int NB, bool CAL, bool FIX>
__global__ void ELBM_ENSEMBLE_BOUNDS(W)
ensemble_march2d_kernel(const EnsembleArgs a, const P* src, P* __restrict__ dst, int* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    wait_for_previous();
    __shared__ int s_start[kMaxEnsemble + 1];
    for (int k = threadIdx.x; k <= a.n; k += blockDim.x) s_start[k] = a.tile_start[k];
    __syncthreads();
    bool bad = false;
#if ELBM_ST >= 2 && ELBM_D == 2
    float2 acc[4] = {};
#else
    Acc5 acc;
    acc.zero();
#endif
    int k = 0;
    for (int u0 = 0, back = 0; u0 < a.ntiles; u0 += gridDim.x, back ^= 1) {
        const int u = u0 + (back ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x);
        if (u >= a.ntiles) continue;
        while (u >= s_start[k + 1]) ++k;   // u increases, so k only moves forward
        const int local = u - s_start[k], tx = a.tiles_x[k], inst = a.order[k];
        const int bx = local % tx, by = local / tx, nseg = (s_start[k + 1] - s_start[k]) / tx;
        const KParams& p = a.params[inst];
        const long long off = a.offset[inst];
        const int seg = (p.ny + nseg - 1) / nseg, y0 = by * seg;
        const PlanesBase pl{src + off, dst + off, (size_t)p.N, src + off};
#if ELBM_ST >= 2 && ELBM_D == 2
        march2d_pair_segment<W, CAL, FIX>(p, pl, bx * W, y0, min(y0 + seg, p.ny), march_smem, acc, bad);
#else
        march2d_segment<W, NB, CAL, FIX>(p, pl, bx * W, y0, min(y0 + seg, p.ny), march_smem, acc, bad);
#endif
    }
    launch_dependents();
    flag_if(bad, status);
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
// Launch with programmatic dependent launch allowed on the kernel before it in the stream.
template <class... Args, class... Act>
cudaError_t launch_dependent(void (*kern)(Args...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Act... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Args>(args)...);
}

constexpr int kThreads = kThreads1D;
constexpr int kTY2 = 8;                  // D2Q9 tile kernel: 32 x 8 tiles
constexpr int kW2 = kMarchW2;            // D2Q9 row march: strips of kW2 nodes
#ifndef ELBM_MARCH_NB
#define ELBM_MARCH_NB 2
#endif
constexpr int kNBM = ELBM_MARCH_NB;      // row buffers of the march (2: one row in flight, 3: two)
// Strip width of the single-lattice D2Q9 march: 256 nodes for the 16-bit stores, whose
// march is issue-bound and pays for the strip's two halo nodes half as often per node, kW2 for FP32 and FP64, which are bandwidth-bound
// (256 measured 39.2 against 44.9 GLUPS in FP32).  The persistent ensemble keeps kW2.
#ifndef ELBM_MARCH_W16
#define ELBM_MARCH_W16 256
#endif
constexpr int kW2L = sizeof(P) == 4 ? ELBM_MARCH_W16 : kW2;
#ifndef ELBM_TY3
#define ELBM_TY3 8
#endif
constexpr int kTY3 = ELBM_TY3;           // D3Q27 re-read and tensor-copy kernels: tiles 32 x kTY3
// Pipelined (cp.async) D3Q27 kernel: tiles 32 x kTYP.  Taller FP32 tiles (more warps per
// SM, relatively fewer halo nodes) measured slower at 256^3: 10 rows 7 %, 12 rows 37 %
// (their plane buffers leave the L1 cache that the 8-byte cp.async copies go through
// 60 KB and 28 KB instead of about 90 KB, and cap the registers at 168); 8 it is.
#ifndef ELBM_TYP_F32
#define ELBM_TYP_F32 8
#endif
constexpr int kTYP = (kST == ST_F32) ? ELBM_TYP_F32 : kTY3;
constexpr int kTotalsBlocks = kTotCtas * kSms;   // totals_kernel grid (grid-stride)
// Pipelined D3Q27 kernel per store: two plane buffers.  FP32 pairs make them 145 KB
// (one CTA per SM, up to 255 registers; a third buffer would leave L1 almost no
// room and measured 35 % slower); FP16/BF16 pairs are half the size (two CTAs per
// SM); FP64 uses the re-read kernel (its plane buffers would not fit).  With one CTA
// per SM the registers also hold plane z while plane z+1's moments are computed, so
// the prefetch of plane z+2 starts one phase earlier (EARLY; 10 % faster at 256^3;
// with two CTAs per SM and 128 registers it measured 1 % slower).
#ifndef ELBM_PIPE_NB_F32
#define ELBM_PIPE_NB_F32 2
#endif
#ifndef ELBM_PIPE_NB_F16
#define ELBM_PIPE_NB_F16 2
#endif
constexpr bool kPipe = (kST != ST_F64);
constexpr int kNB = (kST == ST_F32) ? ELBM_PIPE_NB_F32 : ELBM_PIPE_NB_F16;
constexpr int kMinB = (PipeBytes<kTYP, kNB>::value * 2 + 2048 <= 228 * 1024) ? 2 : 1;
using PipeCfg = Pipe<kTYP, kNB>;
#ifndef ELBM_EARLY
#define ELBM_EARLY 1
#endif
constexpr bool kEarly = ELBM_EARLY && kMinB == 1;
// TMA-staged D3Q27 kernel: FP32 plane buffers (155 KB) leave room for one CTA per SM,
// FP16/BF16 ones (88 KB) for two.
using TmaCfg = Tma<kTY3>;
constexpr int kTmaMinB = (TmaCfg::smem_bytes * 2 + 4096 <= 228 * 1024) ? 2 : 1;

// Can the TMA-staged kernel run this grid?  The tensor map's row pitch nx * pair size
// must be a multiple of 16 bytes (nx a multiple of 2 for FP32 pairs, 4 for FP16/BF16).
int tma_supported(const KParams& p) {
    if (kD != 3 || !kPipe) return 0;
    return p.nx % TmaCfg::XO == 0 && !p.has_fixed;
}

// Tensor map of a population store as rank 3: x (nx pairs), y (ny), w = i * nz + z (the
// planes of all directions); box TmaCfg::BW x RB x 1 (kTmapStage: the TMA-staged
// kernel's copies) or TX x kTYP + 2 x 1 (kTmapPrefetch: the default pipelined kernel's
// L2 prefetch of a tile's source rows).  The encoder is the driver's, reached through
// the runtime (no link against the driver library).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();   // leave no sticky error behind
        return nullptr;
    }
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
}

int encode_tmap(const KParams& p, const void* base, CUtensorMap* out, int kind) {
    if (!tma_supported(p) || (kind != kTmapStage && kind != kTmapPrefetch && kind != kTmapPrefetchAa)) return 0;
    static const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();   // resolved once, thread-safe
    if (!encode) return -1;
    const cuuint64_t dims[3] = {(cuuint64_t)p.nx, (cuuint64_t)p.ny, (cuuint64_t)p.nz * Q};
    const cuuint64_t strides[2] = {(cuuint64_t)p.nx * sizeof(P), (cuuint64_t)p.nx * p.ny * sizeof(P)};
    const cuuint32_t box[3] = {(cuuint32_t)(kind == kTmapStage ? TmaCfg::BW : TX),
                               (cuuint32_t)(kind == kTmapStage ? TmaCfg::RB : kind == kTmapPrefetch ? kTYP + 2 : kTYP), 1u};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    const CUtensorMapDataType dt = sizeof(P) == 8 ? CU_TENSOR_MAP_DATA_TYPE_UINT64 : CU_TENSOR_MAP_DATA_TYPE_UINT32;
#ifndef ELBM_TMAP_PROMO
#define ELBM_TMAP_PROMO CU_TENSOR_MAP_L2_PROMOTION_L2_128B
#endif
    const CUresult r = encode(out, dt, 3, const_cast<void*>(base), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              (CUtensorMapL2promotion)ELBM_TMAP_PROMO, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 1 : -1;
}

inline unsigned blocks_1d(long long n) { return (unsigned)blocks_1d_of(n); }

// Per-direction plane bases of both stores for the kernels.
DirPlanes dir_planes(const KParams& p, const void* src, void* dst) {
    DirPlanes pl;
    for (int i = 0; i < Q; ++i) {
        pl.src[i] = (const P*)src + (size_t)i * (size_t)p.N;
        pl.dst[i] = (P*)dst + (size_t)i * (size_t)p.N;
    }
    return pl;
}

// Grid of the default fused kernel: D2Q9 row march (strips x row segments of p.tz rows),
// D3Q27 pipelined kernel (32 x kTYP column tiles x z segments of p.tz planes).
dim3 fused_grid(const KParams& p) {
    if (kD == 2) return dim3((p.nx + kW2L - 1) / kW2L, (p.ny + p.tz - 1) / p.tz, 1);
    const int ty = kPipe ? kTYP : kTY3;
    return dim3((p.nx + TX - 1) / TX, (p.ny + ty - 1) / ty, (p.nz + p.tz - 1) / p.tz);
}
// Grid of the D3Q27 re-read and tensor-copy kernels (32 x kTY3 tiles).
dim3 grid3_ty3(const KParams& p) {
    return dim3((p.nx + TX - 1) / TX, (p.ny + kTY3 - 1) / kTY3, (p.nz + p.tz - 1) / p.tz);
}
// Grid of the D2Q9 tile kernel (the re-read schedule of D2Q9): 32 x kTY2 tiles.
dim3 tile2d_grid(const KParams& p) { return dim3((p.nx + TX - 1) / TX, (p.ny + kTY2 - 1) / kTY2, 1); }

int max_blocks(const KParams& p) {
    long long a = blocks_1d(p.N);
    dim3 gf = fused_grid(p);
    long long b = (long long)gf.x * gf.y * gf.z;
    long long m = a > b ? a : b;
    const dim3 gt = kD == 2 ? tile2d_grid(p) : grid3_ty3(p);
    const long long c = (long long)gt.x * gt.y * gt.z;
    if (c > m) m = c;
    if (m < kTotalsBlocks) m = kTotalsBlocks;
    if (kD == 2 && row_strips(p) <= kRowMost && m < row_strips(p)) m = row_strips(p);
    return (int)m;
}

// Dynamic shared memory of spread_share, set as the kernel's limit.  The next kernel's CTAs are set
// up while this one's still run: counted against the same limits, they went two and three to
// an SM while others had none, and in FP64 such CTAs share one pipe.  us a step, zero-gradient
// 2D grids and periodic boxes, without this limit and with it:
//   strips, FP64  800x4  6.46  5.38    800x9 9.58  7.66    800x15 13.18 10.33    800x20 16.05 12.99
//   strips, FP32  800x4  2.66  2.60   800x15 2.94  2.74    800x20  3.05  2.81    800x43  3.37  3.31
//   FP64 passes   140^2  35.2  18.0    220^2 40.6  27.5     256^2  45.2  33.0     320^2  55.4  47.0
//                  24^3  35.1  27.8     28^3 45.0  35.7      32^3  44.1  35.4      36^3  65.1  55.4
// From nine CTAs to an SM on the grid takes several waves anyway: no limit.  (The march, whose rows
// reuse the first-level cache that this takes away, is slower with it: FP32 1024^2 28.0 -> 35.0;
// the tiles and the D3Q27 kernel do not change.)  The function's attribute is set to the same value
// every time: another thread's launch, or a graph captured before, may need more than this one.
template <class... Args>
cudaError_t spread_smem(void (*kern)(Args...), long long ctas, int sms, int stat, size_t* share) {
    *share = spread_share(ctas, sms, stat);
    return *share == 0 ? cudaSuccess
                       : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmShared / 2);
}

template <bool PULL>
cudaError_t launch_two_passes(const KParams& p, const void* src, void* dst, void* qfield, double* partials,
                              int* status, cudaStream_t s) {
    const unsigned nb = blocks_1d(p.N);
#if ELBM_ST == 0
    const unsigned nc = (unsigned)((p.N + kThreads64 - 1) / kThreads64);
    constexpr int stat = 5 * kThreads1D * (int)sizeof(double);   // of the totals
    size_t sm = 0, sc = 0;
    cudaError_t e = spread_smem(collide64_kernel<PULL>, nc, p.sms, 0, &sc);
    if (e == cudaSuccess && nc <= 8u * (unsigned)p.sms) e = spread_smem(moments64_kernel<PULL>, nb, p.sms, stat, &sm);
    if (e != cudaSuccess) return e;
    launch_dependent(moments64_kernel<PULL>, nb, kThreads, sm, s, p, (const P*)src, (R*)qfield, (P*)dst, partials, status);
    launch_dependent(collide64_kernel<PULL>, nc, kThreads64, sc, s, p, (const P*)src, (P*)dst, (const R*)qfield);
#else
    launch_dependent(moments_kernel<PULL>, nb, kThreads, 0, s, p, (const P*)src, (R*)qfield);
    launch_dependent(collide_kernel<PULL>, nb, kThreads, 0, s, p, (const P*)src, (P*)dst, (const R*)qfield, partials, status);
#endif
    return cudaGetLastError();
}

cudaError_t launch_init(const KParams& p, const double* rho, const double* u, const double* T, void* pop,
                        void* spare, void* qfield, double* partials, int* status, cudaStream_t s,
                        long long* launches) {
    // The stored state is post-collision: after step n the store holds C(X_n), where
    // X_n is the post-stream state of the method and C the collision, and a step is
    // pull (X_{n+1} = S(C(X_n))) followed by collide.  Initialisation therefore writes
    // X_0 = (f^eq, g^eq) into the spare store and collides it in place of streaming.
    // Moments of C(X_n) equal those of X_n (the collision conserves them), so field
    // extraction and totals read each node's own values.
    const unsigned nb = blocks_1d(p.N);
    init_kernel<<<nb, kThreads, 0, s>>>(p, rho, u, T, (P*)spare, status, 0, p.N);
    *launches += 3;
    return launch_two_passes<false>(p, spare, pop, qfield, partials, status, s);
}

// f^eq, g^eq of nodes n0 .. n0 + cnt - 1 written in place into pop (fields of those nodes
// only).  For the AA single store this is the first half of initialisation: a step from
// layout L1 (node-local reads, swapped writes) then collides the equilibria without
// streaming, leaving C(X_0) in layout L0.
cudaError_t launch_init_nodes(const KParams& p, const double* rho, const double* u, const double* T, void* pop,
                              long long n0, long long cnt, int* status, cudaStream_t s, long long* launches) {
    init_kernel<<<blocks_1d(cnt), kThreads, 0, s>>>(p, rho, u, T, (P*)pop, status, n0, cnt);
    ++*launches;
    return cudaGetLastError();
}

// rho, u, T of nodes n0 .. n0 + cnt - 1 into fields of cnt nodes.
cudaError_t launch_fields_nodes(const KParams& p, const void* pop, double* rho, double* u, double* T,
                                long long n0, long long cnt, int* status, cudaStream_t s, long long* launches) {
    fields_kernel<<<blocks_1d(cnt), kThreads, 0, s>>>(p, (const P*)pop, rho, u, T, status, n0, cnt);
    ++*launches;
    return cudaGetLastError();
}

#ifndef ELBM_PREF
#define ELBM_PREF 1
#endif
constexpr int kPref = ELBM_PREF;   // planes of L2 prefetch ahead of the cp.async copies (with a tensor map)

// One AA step on the single store A: from layout L1 (node-local reads, swapped writes) or
// from L0 (pulled reads, pushed writes).  D3Q27 with FP32 arithmetic, where aa_march_pays or a segment
// length was set: the edges' Q~, then the march in place; else the two passes.
template <int DD>
cudaError_t launch_aa_march(const KParams& p, void* A, void* qfield, double* partials, int* nblocks, int* status,
                            cudaStream_t s, int from_l1, const CUtensorMap* pmap) {
    if constexpr (DD == 3 && kPipe) {
        const dim3 grid = fused_grid(p);
        AaEdges e;
        e.tx = TX, e.ty = kTYP, e.tz = p.tz;
        e.nr = 2 * (int)grid.y, e.nc = 2 * (int)grid.x, e.ns = 2 * (int)grid.z;
        e.br = (unsigned)blocks_1d_of((long long)e.nr * p.nx);
        e.bc = (unsigned)blocks_1d_of((long long)e.nc * p.ny);
        const unsigned bs = (unsigned)blocks_1d_of((long long)e.ns * p.nx * p.ny);
        auto edges = from_l1 ? aa_edges_kernel<true> : aa_edges_kernel<false>;
        cudaError_t c = launch_dependent(edges, dim3((e.br + e.bc) * (unsigned)p.nz + bs), dim3(kThreads), 0, s, p, e, (P*)A, (R*)qfield);
        if (c != cudaSuccess) return c;
        auto kern = p.eos ? (from_l1 ? fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, true, 2>
                                     : fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, true, 1>)
                          : (from_l1 ? fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, false, 2>
                                     : fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, false, 1>);
        c = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PipeCfg::smem_bytes);
        if (c != cudaSuccess) return c;
        CUtensorMap none;
        std::memset(&none, 0, sizeof(none));
        *nblocks = (int)(grid.x * grid.y * grid.z);
        return launch_dependent(kern, grid, dim3(TX, kTYP), PipeCfg::smem_bytes, s, p, dir_planes(p, A, A), (const P*)A,
                                partials, status, pmap ? *pmap : none, pmap ? kPref : 0, (const R*)qfield);
    } else {
        return cudaErrorInvalidValue;
    }
}
cudaError_t launch_step_aa(const KParams& p, void* A, void* qfield, double* partials, int* nblocks, int* status,
                           cudaStream_t s, long long* launches, int from_l1, const CUtensorMap* pmap) {
    *launches += 2;
    const double bytes = (double)p.N * Q * sizeof(P);
    if (kD == 3 && kPipe && march_launches(p, kD, kTYP) &&
        (p.sched == kSchedSegment ? bytes > 64e6 : aa_march_pays(p, kTYP, bytes)))
        return launch_aa_march<kD>(p, A, qfield, partials, nblocks, status, s, from_l1, pmap);
    const unsigned nb = blocks_1d(p.N);
    if (from_l1) {
        launch_dependent(aa_moments_kernel<true>, nb, kThreads, 0, s, p, (P*)A, (R*)qfield);
        launch_dependent(aa_collide_kernel<true>, nb, kThreads, 0, s, p, (P*)A, (const R*)qfield, partials, status);
    } else {
        launch_dependent(aa_moments_kernel<false>, nb, kThreads, 0, s, p, (P*)A, (R*)qfield);
        launch_dependent(aa_collide_kernel<false>, nb, kThreads, 0, s, p, (P*)A, (const R*)qfield, partials, status);
    }
    *nblocks = (int)nb;
    return cudaGetLastError();
}

cudaError_t launch_fields(const KParams& p, const void* pop, double* rho, double* u, double* T, int* status,
                          cudaStream_t s, long long* launches) {
    fields_kernel<<<blocks_1d(p.N), kThreads, 0, s>>>(p, (const P*)pop, rho, u, T, status, 0, p.N);
    ++*launches;
    return cudaGetLastError();
}

cudaError_t launch_twopass(const KParams& p, const void* src, void* dst, void* qfield, double* partials,
                           int* nblocks, int* status, cudaStream_t s, long long* launches) {
    const unsigned nb = blocks_1d(p.N);
    *launches += 2;
    *nblocks = (int)nb;
    return launch_two_passes<true>(p, src, dst, qfield, partials, status, s);
}

// A template so that the branch of the other lattice is never instantiated; CAL as in
// the kernels (the caloric form only for handles with a Cv(T) model).
// The row march of this store for grid p (D2Q9).
template <int DD, bool CAL>
auto march_kernel(const KParams& p) {
    static_assert(DD == 2, "D2Q9");
#if ELBM_ST >= 2 && ELBM_D == 2
    return p.has_fixed ? march2d_pair_kernel<kW2L, CAL, true> : march2d_pair_kernel<kW2L, CAL, false>;
#else
    return p.has_fixed ? march2d_kernel<kW2L, kNBM, CAL, true> : march2d_kernel<kW2L, kNBM, CAL, false>;
#endif
}

template <int DD, bool CAL>
cudaError_t launch_fused_cal(const KParams& p, const void* src, void* dst, double* partials, int* status,
                             cudaStream_t s, bool reread, const CUtensorMap* pmap = nullptr) {
    const dim3 grid = fused_grid(p);
    if constexpr (DD == 2) {
        if (!reread && p.sched == kSchedRow) {
#if ELBM_ST == 0 && ELBM_D == 2
            auto kern = p.has_fixed ? fused2d_split_kernel<CAL, true> : fused2d_split_kernel<CAL, false>;
            constexpr int threads = 128, stat = kSplitSmem;
#else
            auto kern = p.has_fixed ? fused2d_row_kernel<CAL, true> : fused2d_row_kernel<CAL, false>;
            constexpr int threads = 32, stat = kRowSmem;
#endif
            const long long strips = row_strips(p);
            size_t share = 0;
            const cudaError_t e = spread_smem(kern, strips, p.sms, stat, &share);
            if (e != cudaSuccess) return e;
            return launch_dependent(kern, dim3((unsigned)strips), dim3(threads), share, s, p, (const P*)src, (P*)dst,
                                    (p.nx + kRowW - 1) / kRowW, partials, status);
        } else if (reread || p.sched == kSchedTile) {   // the tile kernel: one 32 x kTY2 tile per CTA, no march
            launch_dependent(fused2d_kernel<kTY2, CAL>, tile2d_grid(p), dim3(TX, kTY2), 0, s, p, (const P*)src, (P*)dst, partials,
                                                                               status);
        } else {
            auto kern = march_kernel<DD, CAL>(p);
            constexpr size_t smem = march_smem_bytes<kW2L, kNBM>;
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            DirPlanes pl = dir_planes(p, src, dst);
            e = launch_dependent(kern, dim3(grid), march_threads<kW2L, kNBM>, smem, s, p, pl, (const P*)src, partials, status);
            if (e != cudaSuccess) return e;
        }
    } else {
        bool launched = false;
        if constexpr (kPipe) {
            if (!reread) {
                auto kern = fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, CAL, 0>;
                // the dynamic shared-memory limit is a per-function attribute; setting it
                // again is cheap and keeps this correct for every device of the process
                cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)PipeCfg::smem_bytes);
                if (e != cudaSuccess) return e;
                DirPlanes pl = dir_planes(p, src, dst);
                CUtensorMap none;
                std::memset(&none, 0, sizeof(none));
                e = launch_dependent(kern, dim3(grid), dim3(TX, kTYP), PipeCfg::smem_bytes, s, p, pl, (const P*)src, partials, status,
                                                                       pmap ? *pmap : none, pmap ? kPref : 0,
                                     (const R*)nullptr);
            if (e != cudaSuccess) return e;
                launched = true;
            }
        }
        if (!launched)
            launch_dependent(fused3d_reread_kernel<kTY3, CAL>, grid3_ty3(p), dim3(TX, kTY3), 0, s, p, (const P*)src, (P*)dst, partials,
                                                                              status);
    }
    return cudaGetLastError();
}

template <int DD, bool CAL>
cudaError_t launch_tma_cal(const KParams& p, const void* src, void* dst, const CUtensorMap* map, double* partials,
                           int* status, cudaStream_t s) {
    if constexpr (DD == 3 && kPipe) {
        auto kern = fused3d_tma_kernel<kTY3, kTmaMinB, DD, CAL>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)TmaCfg::smem_bytes);
        if (e != cudaSuccess) return e;
        DirPlanes pl = dir_planes(p, src, dst);
        e = launch_dependent(kern, dim3(grid3_ty3(p)), dim3(TX, kTY3), TmaCfg::smem_bytes, s, p, pl, *map, (const P*)src, partials, status);
            if (e != cudaSuccess) return e;
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

// TMA-staged fused step; map is the tensor map of src (encode_tmap, kTmapStage).
cudaError_t launch_fused_tma(const KParams& p, const void* src, void* dst, const CUtensorMap* map,
                             double* partials, int* nblocks, int* status, cudaStream_t s, long long* launches) {
    if (!tma_supported(p) || !map) return cudaErrorInvalidValue;
    const cudaError_t e = p.eos ? launch_tma_cal<kD, true>(p, src, dst, map, partials, status, s)
                                : launch_tma_cal<kD, false>(p, src, dst, map, partials, status, s);
    ++*launches;
    const dim3 grid = grid3_ty3(p);
    *nblocks = (int)(grid.x * grid.y * grid.z);
    return e;
}

template <int DD>
cudaError_t launch_fused(const KParams& p, const void* src, void* dst, double* partials, int* nblocks,
                         int* status, cudaStream_t s, long long* launches, bool reread,
                         const CUtensorMap* pmap = nullptr) {
    const cudaError_t e = p.eos ? launch_fused_cal<DD, true>(p, src, dst, partials, status, s, reread, pmap)
                                : launch_fused_cal<DD, false>(p, src, dst, partials, status, s, reread, pmap);
    ++*launches;
    const dim3 grid = DD == 2 ? (!reread && p.sched == kSchedRow ? dim3((unsigned)row_strips(p), 1, 1)
                                 : (reread || p.sched == kSchedTile)   ? tile2d_grid(p)
                                                          : fused_grid(p))
                              : ((reread && kPipe) ? grid3_ty3(p) : fused_grid(p));
    *nblocks = (int)(grid.x * grid.y * grid.z);
    return e;
}

cudaError_t launch_fused_default(const KParams& p, const void* src, void* dst, double* partials, int* nblocks,
                                 int* status, cudaStream_t s, long long* launches) {
    return launch_fused<kD>(p, src, dst, partials, nblocks, status, s, launches, false);
}

cudaError_t launch_fused_reread(const KParams& p, const void* src, void* dst, double* partials, int* nblocks,
                                int* status, cudaStream_t s, long long* launches) {
    return launch_fused<kD>(p, src, dst, partials, nblocks, status, s, launches, true);
}

// The default fused step with src's prefetch tensor map at hand (encode_tmap,
// kTmapPrefetch: L2 prefetch of the planes ahead).
cudaError_t launch_fused_pf(const KParams& p, const void* src, void* dst, const CUtensorMap* map, double* partials,
                            int* nblocks, int* status, cudaStream_t s, long long* launches) {
    return launch_fused<kD>(p, src, dst, partials, nblocks, status, s, launches, false, map);
}

template <bool CAL>
cudaError_t launch_ensemble_march(const EnsembleArgs& a, const void* src, void* dst, int* status, int grid,
                                  cudaStream_t s) {
    auto kern = a.fixed ? ensemble_march2d_kernel<kW2, kNBM, CAL, true> : ensemble_march2d_kernel<kW2, kNBM, CAL, false>;
    constexpr size_t smem = march_smem_bytes<kW2, kNBM>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = launch_dependent(kern, dim3(grid), march_threads<kW2, kNBM>, smem, s, a, (const P*)src, (P*)dst, status);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Persistent ensemble step and `grid` CTAs: ty = 4, 8 or 16 runs one 32 x ty tile per work
// unit; ty = kMarchSegs (32, 64 or 128) runs the row march over strips of kW2 nodes and
// segments of about ty rows.
cudaError_t launch_ensemble(const EnsembleArgs& a, const void* src, void* dst, int* status, int ty, int grid,
                            cudaStream_t s, long long* launches) {
    if constexpr (kD == 2) {
        if (ty > 16) {
            ++*launches;
            return a.caloric ? launch_ensemble_march<true>(a, src, dst, status, grid, s)
                             : launch_ensemble_march<false>(a, src, dst, status, grid, s);
        }
        if (a.caloric) {
            if (ty == 4) launch_dependent(ensemble2d_kernel<4, true>, grid, dim3(TX, 4), 0, s, a, (const P*)src, (P*)dst, status);
            else if (ty == 16)
                launch_dependent(ensemble2d_kernel<16, true>, grid, dim3(TX, 16), 0, s, a, (const P*)src, (P*)dst, status);
            else launch_dependent(ensemble2d_kernel<8, true>, grid, dim3(TX, 8), 0, s, a, (const P*)src, (P*)dst, status);
        } else {
            if (ty == 4) launch_dependent(ensemble2d_kernel<4, false>, grid, dim3(TX, 4), 0, s, a, (const P*)src, (P*)dst, status);
            else if (ty == 16)
                launch_dependent(ensemble2d_kernel<16, false>, grid, dim3(TX, 16), 0, s, a, (const P*)src, (P*)dst, status);
            else launch_dependent(ensemble2d_kernel<8, false>, grid, dim3(TX, 8), 0, s, a, (const P*)src, (P*)dst, status);
        }
        ++*launches;
        return cudaGetLastError();
    } else {
        return cudaErrorInvalidValue;
    }
}

// Occupancy (resident CTAs per SM) of the ensemble kernel with tile height ty (or, above
// 16, of the row-march form).
int ensemble_occupancy(int ty) {
    int nb = 0;
    if constexpr (kD == 2) {
        cudaError_t e;
        if (ty > 16) {
            auto kern = ensemble_march2d_kernel<kW2, kNBM, false, false>;
            constexpr size_t smem = march_smem_bytes<kW2, kNBM>;
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, march_threads<kW2, kNBM>, smem) != cudaSuccess)
                return 0;
            return nb;
        }
        // the constant-gamma form (the caloric one differs by a few registers at most)
        if (ty == 4) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, ensemble2d_kernel<4, false>, TX * 4, 0);
        else if (ty == 16)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, ensemble2d_kernel<16, false>, TX * 16, 0);
        else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, ensemble2d_kernel<8, false>, TX * 8, 0);
        if (e != cudaSuccess) return 0;
    }
    return nb;
}

// Columns of 32 x 8 nodes over segments chosen like those of the fused kernels; a grid has at
// most as many CTAs as the one-dimensional launches, or one per column (max_blocks bounds both).
cudaError_t launch_stats(const KParams& p, const void* pop, double* partials, int* nblocks, cudaStream_t s,
                         long long* launches, bool wide) {
    const int tx = (p.nx + 31) / 32, ty = (p.ny + 7) / 8;
    const long long most = blocks_1d_of(p.N) > kTotalsBlocks ? blocks_1d_of(p.N) : kTotalsBlocks;
    int tz = choose_segment((double)tx * ty, p.nz, p.sms, 2, 32);
    while (tz < p.nz && (long long)tx * ty * ((p.nz + tz - 1) / tz) > most) tz = tz < p.nz / 2 ? 2 * tz : p.nz;
    const long long grid = (long long)tx * ty * ((p.nz + tz - 1) / tz);
    auto kern = wide ? stats_kernel<kD, true> : stats_kernel<kD, sizeof(R) == 8>;
    kern<<<(unsigned)grid, dim3(32, 8), 0, s>>>(p, (const P*)pop, partials, tz, (unsigned)tx, (unsigned)ty);
    ++*launches;
    *nblocks = (int)grid;
    return cudaGetLastError();
}

cudaError_t launch_totals(const KParams& p, const void* pop, double* partials, int* nblocks, cudaStream_t s,
                          long long* launches) {
    constexpr int run = kTotThreads * kTotRun;
    totals_kernel<<<kTotalsBlocks, kTotThreads, 0, s>>>(p, (const P*)pop, partials, (int)((p.N + run - 1) / run));
    ++*launches;
    *nblocks = kTotalsBlocks;
    return cudaGetLastError();
}

// Resident CTAs per SM of the default fused kernel for grid p (a template so that the
// kernel of the other lattice is never instantiated).
template <int DD>
int fused_occupancy_impl(const KParams& p) {
    int n = 0;
    if constexpr (DD == 3 && kPipe) {
        auto kern = fused3d_kernel<kTYP, kNB, kMinB, kEarly, DD, false, 0>;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PipeCfg::smem_bytes) !=
                cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, TX * kTYP, PipeCfg::smem_bytes) != cudaSuccess)
            return 0;
    } else if constexpr (DD == 3) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fused3d_reread_kernel<kTY3, false>, TX * kTY3, 0) !=
            cudaSuccess)
            return 0;
    } else {
        auto kern = march_kernel<DD, false>(p);
        constexpr size_t smem = march_smem_bytes<kW2L, kNBM>;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, march_threads<kW2L, kNBM>, smem) != cudaSuccess)
            return 0;
    }
    return n;
}
int fused_occupancy(const KParams& p) { return fused_occupancy_impl<kD>(p); }

const Ops kOps = {kD,          kST,           sizeof(P) / 2,  sizeof(R),            max_blocks,
                  launch_init, launch_fields, launch_twopass, launch_fused_default, launch_fused_reread,
                  launch_totals, launch_ensemble, ensemble_occupancy, launch_stats,
                  kD == 3 ? (kPipe ? kTYP : kTY3) : 1, fused_occupancy, launch_fused_tma, tma_supported, encode_tmap,
                  launch_fused_pf, launch_init_nodes, launch_fields_nodes, launch_step_aa, kW2L};

}  // namespace

#define ELBM_CAT2(a, b) a##b
#define ELBM_CAT(a, b) ELBM_CAT2(a, b)
const Ops* ELBM_CAT(ops_, ELBM_OPS_NAME)() { return &kOps; }

}  // namespace elbm
