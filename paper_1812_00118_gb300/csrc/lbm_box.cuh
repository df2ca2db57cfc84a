// Resident step of small grids: one launch advances a grid that fits on the
// chip by many time steps.
//
// What bounds a small grid is not memory but latency: the march of
// lbm_kernels.cuh walks its planes one after the other and pays a launch per
// step, and a 256 x 256 grid gives it 32 CTAs of 18 dependent planes.  Here
// the grid is cut into boxes of BX x BY x BZ nodes, one thread per node and
// one CTA per box, all boxes resident at once: a step is one round of loads,
// one barrier, one collision and one round of stores.  (us per step, march of
// 16-plane chunks / this: 64^2 FP64 190 / 13.5, 256^2 FP32 22.7 / 4.3, 150 x 600 with
// walls 28.8 / 6.0, 32^3 45 / 6.5.  At 64^2 FP32 the 3.1 are, in clk: the wait for
// the flags 640, loads and sums 1600, collision 830, release 1000.)
//
// Between steps a box waits only for the boxes around it.  A node's new
// populations depend on cells at most two nodes away (the phi stencil reaches
// one node, that node's pull another), so with boxes at least two nodes wide
// the data of step s come from the up to 26 adjacent boxes, and the buffer
// step s writes was last read, in step s - 1, by the same boxes.  flags[box]
// counts the warps that have completed a step: box b starts step s once every
// adjacent flag shows step s - 1 done by all of them, which covers both.  The counts go on
// from launch to launch (a box reads its own at the start), so a captured
// launch can be replayed.  The launch is cooperative whenever boxes wait, so
// they are all resident; the waits are bounded (lbm_set_wait_limit), and one that
// gives up raises *err, on which every box that still waits leaves.  The state is
// lost then, and reads out as NaN (phi_kernel, get_kernel).
#pragma once
#include "lbm_kernels.cuh"

namespace lbm {

// The counts are 32 bits wide and never reset while a context steps on: 8 warps
// pass 2^31 after 2.7e8 steps, 19 minutes of a 256 x 256 grid.  They are unsigned
// and compared by their difference, which a wrap leaves as it is (it never
// exceeds two steps).  A context's counts start just below 2^31, so that every
// run passes the sign bit in its first steps and not only one of 19 minutes.
constexpr unsigned kBoxFirstCount = 0x7ffffff0u;

// the count of a box that has completed `steps` steps since it stood at `first`
__host__ __device__ __forceinline__ unsigned box_count(unsigned first, int steps, int warps) {
    return first + (unsigned)steps * (unsigned)warps;
}
__host__ __device__ __forceinline__ bool box_reached(unsigned count, unsigned want) {
    return count - want < 0x80000000u;
}

// Loads of populations another CTA may have written in this launch: coherent
// at the GPU scope (never the read-only path).
template <typename S> __device__ __forceinline__ S ld_coherent(const S* p);
template <> __device__ __forceinline__ double ld_coherent<double>(const double* p) {
    double v; asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p)); return v;
}
template <> __device__ __forceinline__ float ld_coherent<float>(const float* p) {
    float v; asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p)); return v;
}
template <> __device__ __forceinline__ __half ld_coherent<__half>(const __half* p) {
    unsigned short v; asm volatile("ld.relaxed.gpu.global.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return __ushort_as_half(v);
}
template <> __device__ __forceinline__ __nv_bfloat16 ld_coherent<__nv_bfloat16>(const __nv_bfloat16* p) {
    unsigned short v; asm volatile("ld.relaxed.gpu.global.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return __ushort_as_bfloat16(v);
}

// How a grid is cut: boxes along each internal axis (box i of n spans nodes
// [i N / n, (i + 1) N / n), so all are about equally wide) and the variant.
struct BoxPlan {
    int variant = -1;
    int nx = 0, ny = 0, nz = 0;
    int boxes = 0;
    int ctas = 0;      // CTAs of a launch whose boxes wait for one another
};

__device__ __forceinline__ int box_bound(int i, int N, int n) { return (int)((long long)i * N / n); }

template <int LAT, int ST, int BX, int BY, int BZ>
struct BoxSmem {
    static constexpr int HY = Lattice<LAT>::kHasY ? 1 : 0;
    typename Storage<ST>::R phis[BZ + 2][BY + 2 * HY][BX + 2];
};

// One step of the box `box`; false if a wait gave up.  wait_for > 0: the
// adjacent boxes' flags must have reached first + wait_for.
template <int LAT, int ST, int BX, int BY, int BZ, bool WALLS>
__device__ __forceinline__ bool box_step(const DirPtrs<typename Storage<ST>::S, Lattice<LAT>::Q>& D, const Geom& G,
                                         const PhysT<typename Storage<ST>::R>& p, const BoxPlan& pl, int box,
                                         unsigned first, int wait_for, const unsigned* flags, int* err, int polls,
                                         BoxSmem<LAT, ST, BX, BY, BZ>& sm) {
    using L = Lattice<LAT>;
    using St = Storage<ST>;
    using R = typename St::R;
    constexpr int Q = L::Q;
    constexpr int HY = L::kHasY ? 1 : 0;
    constexpr int NT = BX * BY * BZ;
    const int tid = threadIdx.x;
    const int bx = box % pl.nx, by = (box / pl.nx) % pl.ny, bz = box / (pl.nx * pl.ny);
    const int x0 = box_bound(bx, G.NX, pl.nx), ex = box_bound(bx + 1, G.NX, pl.nx) - x0;
    const int y0 = HY ? box_bound(by, G.NY, pl.ny) : 0, ey = HY ? box_bound(by + 1, G.NY, pl.ny) - y0 : 1;
    const int z0 = box_bound(bz, G.NZ, pl.nz), ez = box_bound(bz + 1, G.NZ, pl.nz) - z0;
    const int lx = tid % BX, ly = (tid / BX) % BY, lz = tid / (BX * BY);
    const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
    const bool active = lx < ex && ly < ey && lz < ez;
    // the box's halo shell: in 3-D two full faces in z and the ring of every
    // plane between them, in 2-D two rows and the columns beside the box
    const int row = ex + 2, face = HY ? row * (ey + 2) : row, ring = HY ? 2 * (row + ey) : 2;
    const int shell = 2 * face + ring * ez;
    auto shell_pos = [&](int k, int* a, int* b, int* c) {
        if (k < 2 * face) {
            *c = k < face ? -1 : ez;
            const int r = k < face ? k : k - face;
            *a = r % row - 1;
            *b = HY ? r / row - 1 : 0;
        } else {
            const int r = k - 2 * face, q = r % ring;
            *c = r / ring;
            if (HY && q < 2 * row) { *a = q % row - 1; *b = q < row ? -1 : ey; }
            else { const int e = HY ? q - 2 * row : q; *a = (e & 1) ? ex : -1; *b = HY ? e >> 1 : 0; }
        }
    };
    auto shell_offsets = [&](int k, int* slot) {
        int a, b, c;
        shell_pos(k, &a, &b, &c);
        *slot = ((c + 1) * (BY + 2 * HY) + b + HY) * (BX + 2) + a + 1;
        PullOffsets o = pull_offsets(G, stencil_coord(x0 + a, G.NX, G.wall[0]),
                                     HY ? stencil_coord(y0 + b, G.NY, G.wall[1]) : 0,
                                     stencil_coord(z0 + c, G.NZ, G.wall[2]));
        checked_offsets(o, G.NP);
        return o;
    };
    PullOffsets own = pull_offsets(G, active ? x : x0, active ? y : y0, active ? z : z0);
    checked_offsets(own, G.NP);
    int slot0 = 0;
    PullOffsets sh0 = own;
    const bool has0 = tid < shell;
    if (has0) sh0 = shell_offsets(tid, &slot0);

    bool ok = true;
    if (wait_for > 0) {
        constexpr int NNB = HY ? 27 : 9;
        if (tid < NNB) {
            int a = bx + tid % 3 - 1, b = HY ? by + (tid / 3) % 3 - 1 : 0, c = bz + (HY ? tid / 9 : tid / 3) - 1;
            // a wall ends the dependence, a periodic axis wraps it
            const bool none = (G.wall[0] && (a < 0 || a >= pl.nx)) || (HY && G.wall[1] && (b < 0 || b >= pl.ny)) ||
                              (G.wall[2] && (c < 0 || c >= pl.nz));
            if (!none) {
                a = a < 0 ? pl.nx - 1 : (a >= pl.nx ? 0 : a);
                b = b < 0 ? pl.ny - 1 : (b >= pl.ny ? 0 : b);
                c = c < 0 ? pl.nz - 1 : (c >= pl.nz ? 0 : c);
                const unsigned* f = flags + (c * pl.ny + b) * pl.nx + a;
                const unsigned want = box_count(first, wait_for, NT / 32);
                ok = false;
                for (int i = 0; i < polls; ++i) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
                    if (box_reached(v, want)) { ok = true; break; }
                    if ((i & 255) == 255 && *(volatile int*)err) break;   // another box gave up
                }
                if (!ok) atomicExch(err, 1);
            }
        }
        ok = __syncthreads_and(ok) != 0;   // also: the phi of the step before is read
        if (!ok) return false;
    }

    // one round of loads: the node's own h and g and its first halo position
    typename St::S hv[Q], gv[Q], sv[Q];
    Unroll<0, Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        hv[i] = ld_coherent(pull_ptr<LAT, i>(D.hin, own));
    });
    if ((tid & ~31) < shell) {   // uniform over the warp
        Unroll<0, Q>::run([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            sv[i] = ld_coherent(pull_ptr<LAT, i>(D.hin, sh0));
        });
    }
    Unroll<0, Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        gv[i] = ld_coherent(pull_ptr<LAT, i>(D.gin, own));
    });
    auto with_shift = [&](R v) {
        if constexpr (St::kShifted) return v + p.h_shift;
        else return v;
    };
    PhiSum<R> phi;
    Unroll<0, Q>::run([&](auto ic) { phi.add(St::raw(hv[decltype(ic)::value])); });
    if (active) sm.phis[lz + 1][ly + HY][lx + 1] = with_shift(phi.value());
    if (has0) {
        PhiSum<R> s;
        Unroll<0, Q>::run([&](auto ic) { s.add(St::raw(sv[decltype(ic)::value])); });
        (&sm.phis[0][0][0])[slot0] = with_shift(s.value());
    }
    R gr[Q];
    Unroll<0, Q>::run([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr double W = L::w[i];
        gr[i] = St::load(gv[i], (R)W * p.g_shift, p.g_inv_scale);
    });
    const Moments<R> m = g_moments<LAT>([&](int i) { return gr[i]; });
    for (int k = tid + NT; k < shell; k += NT) {
        int slot;
        const PullOffsets o = shell_offsets(k, &slot);
        PhiSum<R> s;
        Unroll<0, Q>::run([&](auto ic) { sv[decltype(ic)::value] = ld_coherent(pull_ptr<LAT, decltype(ic)::value>(D.hin, o)); });
        Unroll<0, Q>::run([&](auto ic) { s.add(St::raw(sv[decltype(ic)::value])); });
        (&sm.phis[0][0][0])[slot] = with_shift(s.value());
    }
    __syncthreads();
    if (active) {
        const int rb = (y + G.GY) * G.PX + x + G.GX;
        auto h_of = [&](int i) { return St::raw(hv[i]); };
        // a warp with a node next to a wall takes one path, not both
        if (WALLS && __any_sync(__activemask(), wall_adjacent<LAT>(G, x, y, z)))
            collide_node<LAT, ST, true>(D, G, p, sm.phis, lz, lz + 1, lz + 2, lx + 1, ly + HY, m, h_of, x, y, z, rb);
        else
            collide_node<LAT, ST, false>(D, G, p, sm.phis, lz, lz + 1, lz + 2, lx + 1, ly + HY, m, h_of, x, y, z, rb);
    }
    return true;
}

// The buffers of even and odd steps of a launch.
template <typename S, int Q>
struct BoxPtrs {
    DirPtrs<S, Q> d[2];
};

// n_steps steps from the buffers d[0].hin, d[0].gin.
template <int LAT, int ST, int BX, int BY, int BZ, int MINB, bool WALLS>
__global__ void __launch_bounds__(BX * BY * BZ, MINB)
box_kernel(const __grid_constant__ BoxPtrs<typename Storage<ST>::S, Lattice<LAT>::Q> ptrs, const __grid_constant__ Geom G,
           const __grid_constant__ PhysT<typename Storage<ST>::R> p, const __grid_constant__ BoxPlan pl, int n_steps,
           unsigned* flags, int* err, int polls) {
    __shared__ BoxSmem<LAT, ST, BX, BY, BZ> sm;
    const unsigned first = n_steps > 1 ? *(volatile unsigned*)(flags + blockIdx.x) : 0u;
#pragma unroll 1
    for (int s = 0; s < n_steps; ++s) {
        for (int box = blockIdx.x; box < pl.boxes; box += gridDim.x) {
            if (s == 0 && box != blockIdx.x) __syncthreads();   // phi of the box before (later steps wait instead)
            if (!box_step<LAT, ST, BX, BY, BZ, WALLS>(ptrs.d[s & 1], G, p, pl, box, first, s, flags, err, polls, sm))
                return;
            // a warp's stores are done, each on its own account: no barrier, and
            // the releases of a box's warps overlap
            if (n_steps > 1) {
                __syncwarp();
                if ((threadIdx.x & 31) == 0)
                    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(flags + box) : "memory");
            }
        }
    }
}

// Counts in memory just allocated (those of a new state: NewState).
static __global__ void box_start_kernel(unsigned* flags, int boxes) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < boxes) flags[k] = kBoxFirstCount;
}

}  // namespace lbm
