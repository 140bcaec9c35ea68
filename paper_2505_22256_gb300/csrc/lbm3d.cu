// Three-dimensional form of the time step (arXiv 2505.22256, Sec. 3.5) and its C ABI
// (include/lbm3d.h).
//
// State: the post-collision populations f*_i^k of one lattice, [19][N] pairs (f*_i^A, f*_i^B) in the
// storage / compute type R (float or double), N = nx ny nz, x fastest; two buffers.  One vector
// access moves both components of a direction.  One time step is two
// launches:
//   k3_rho    pull f_i(x) = f*_i(x - e_i), or f*_opp(i)(x) across a blocked link (halfway
//             bounce-back, Sec. 3.5); (rho_A, rho_B) = sum_i f_i (Eq. 3) into one interleaved
//             density array
//   k3_march  the same pull for the node's own populations and momentum (Eq. 4); cohesion (Eq. 8)
//             and adhesion (Eq. 9, local parameter of Eqs. 10-12) on the 92-offset eighth-order
//             stencil -- nodes with a solid node inside the stencil apply the second-layer copy
//             x + sign(e) (Sec. 2.4) and the solid switch; body force; velocity with Guo's
//             half-force shift (Eq. 5); SRT collision with Guo forcing (Eqs. 1, 2, 6, 7) written to
//             the other buffer.  Blocks march along z with the stencil's density planes in shared
//             memory.  Its fields forms write rho and u in FP64 instead of colliding, one of them
//             per-block diagnostic records, too.
// Periodic in x, y and z.
#include <math.h>
#include <stdarg.h>

#include <mutex>
#include <type_traits>
#include <vector>

#include "lbm_internal.h"
#include "../../include/lbm3d.h"

namespace lbm {
lbm_status report_error(lbm_status s, const char* fmt, ...);
}

using namespace lbm;

namespace {

// D3Q19: 0 rest; 1..6 = +x, -x, +y, -y, +z, -z; 7..18 = (1,1,0), (-1,-1,0), (1,-1,0), (-1,1,0),
// (1,0,1), (-1,0,-1), (1,0,-1), (-1,0,1), (0,1,1), (0,-1,-1), (0,1,-1), (0,-1,1)
__host__ __device__ __forceinline__ constexpr int e3x(int i) {
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1 : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__host__ __device__ __forceinline__ constexpr int e3y(int i) {
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1 : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__host__ __device__ __forceinline__ constexpr int e3z(int i) {
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1 : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
__host__ __device__ __forceinline__ constexpr int opp3(int i) { return i == 0 ? 0 : (i % 2 ? i + 1 : i - 1); }
__host__ __device__ __forceinline__ constexpr double w19(int i) { return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0); }
// The collision's weights in the compute type.  1/3, 1/18 and 1/36 rounded to FP32 one by one sum to
// 1 + 2e-8, and every step redistributes each node's mass with them, so an FP32 run gained that much
// mass per step; the FP32 set below sums to 1 exactly (w_0 + 6 w_1 + 12 w_2 = 1 with w_2 = w_1 / 2,
// w_1 = 7456540 2^-27, w_0 = 11184812 2^-25), each weight within 1.2e-7 (relative) of its value.
template <class R>
__host__ __device__ __forceinline__ constexpr double w19c(int i) { return w19(i); }
template <>
__host__ __device__ __forceinline__ constexpr double w19c<float>(int i) {
    return i == 0 ? 11184812.0 / 33554432.0 : (i <= 6 ? 7456540.0 / 134217728.0 : 3728270.0 / 134217728.0);
}
// eighth-order stencil weights by |e|^2 (0: not in the stencil)
__host__ __device__ __forceinline__ constexpr double w92(int q) {
    return q == 1 ? 4.0 / 45.0 : q == 2 ? 1.0 / 21.0 : q == 3 ? 2.0 / 105.0 : q == 4 ? 5.0 / 504.0
         : q == 5 ? 1.0 / 315.0 : q == 6 ? 1.0 / 630.0 : q == 8 ? 1.0 / 5040.0 : 0.0;
}

// node flags: bits 0..17 link i = bit+1 blocked (x - e_i solid); 18 solid; 19 a solid node lies in
// the 92-offset stencil; 20 a solid node within three cells (Chebyshev; contact-angle exclusion)
constexpr uint32_t k3Solid = 1u << 18;
constexpr uint32_t k3Wall = 1u << 19;
constexpr uint32_t k3Near = 1u << 20;

struct Geo3 {
    int nx, ny, nz;
    long long N;
};

__device__ __forceinline__ int wrapc(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
__device__ __forceinline__ long long site(const Geo3& g, int x, int y, int z) {
    return ((long long)wrapc(z, g.nz) * g.ny + wrapc(y, g.ny)) * g.nx + wrapc(x, g.nx);
}

template <class R>
struct P3 {
    R omega[2], cF[2], G, Gw2, lam, delta, s1, s2, s3, t2, t3, g[3];
    R sh[3][2];  // storage shifts w rho0_store[k] of the 16-bit storage modes, by weight class
    int mode;
    int psi;  // second-layer reading: a replaced (solid) site copies psi only and keeps s = 1
    int adh;  // 1: adhesion sum of Eq. 9 with the D3Q19 weights over the first layer
};

// Stored populations: FP64 and FP32 pairs as computed; the 16-bit types hold h = f - w_i rho0_k per
// component (rho0 = lbm3d_params.rho0_store), which ld3 adds back (one rounding, the widening is
// exact) and st3 takes off before rounding to 16 bits.
__host__ __device__ __forceinline__ constexpr int wcls3(int i) { return i == 0 ? 0 : (i <= 6 ? 1 : 2); }
template <class S, class R>
__device__ __forceinline__ V2<R> ld3(const Pair<S>* p, const P3<R>& P, int i) {
    V2<R> v;
    if constexpr (Store<S>::kShift) load_pair<S, R>(p, P.sh[wcls3(i)][0], P.sh[wcls3(i)][1], v.x, v.y);
    else load_pair<S, R>(p, (R)0, (R)0, v.x, v.y);
    return v;
}
template <class S, class R>
__device__ __forceinline__ void st3(Pair<S>* p, V2<R> v, const P3<R>& P, int i) {
    if constexpr (Store<S>::kShift) store_pair<S, R>(p, v.x - P.sh[wcls3(i)][0], v.y - P.sh[wcls3(i)][1]);
    else store_pair<S, R>(p, v.x, v.y);
}

// Adhesion variants of the wall stencil: 0 the 92-offset sum with the solid switch of a replaced
// second-layer site, 1 the same keeping s = 1 there, 2 the D3Q19 first-layer sum (Eq. 9 as printed).
enum { kAdhE8 = 0, kAdhE8Psi = 1, kAdhD3Q19 = 2 };
__host__ __device__ constexpr double w19q(int q) { return q == 1 ? 1.0 / 18.0 : (q == 2 ? 1.0 / 36.0 : 0.0); }

__global__ void k3_flags(Geo3 g, const uint8_t* __restrict__ solid, uint32_t* __restrict__ flags) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long s = ((long long)z * g.ny + y) * g.nx + x;
    uint32_t f = 0;
    if (solid[s]) f |= k3Solid;
    for (int i = 1; i < 19; ++i)
        if (solid[site(g, x - e3x(i), y - e3y(i), z - e3z(i))]) f |= 1u << (i - 1);
    for (int dz = -3; dz <= 3; ++dz)
        for (int dy = -3; dy <= 3; ++dy)
            for (int dx = -3; dx <= 3; ++dx) {
                if (!solid[site(g, x + dx, y + dy, z + dz)]) continue;
                f |= k3Near;
                const int q = dx * dx + dy * dy + dz * dz;
                if (dx >= -2 && dx <= 2 && dy >= -2 && dy <= 2 && dz >= -2 && dz <= 2 && w92(q) != 0.0) f |= k3Wall;
            }
    flags[s] = f;
}

// Wrapped neighbourhood of one node: the x index and the y, z offsets (y nx, z nx ny) for the
// displacements -2..2, as 32-bit values, so every stencil site is one three-operand add.
struct Nb3 {
    int xw[5], yo[5], zo[5];
    __device__ __forceinline__ Nb3(const Geo3& g, int x, int y, int z) {
        const int nxy = g.nx * g.ny;
#pragma unroll
        for (int d = -2; d <= 2; ++d) {
            xw[d + 2] = wrapc(x + d, g.nx);
            yo[d + 2] = wrapc(y + d, g.ny) * g.nx;
            zo[d + 2] = wrapc(z + d, g.nz) * nxy;
        }
    }
    __device__ __forceinline__ int at(int dx, int dy, int dz) const { return zo[dz + 2] + yo[dy + 2] + xw[dx + 2]; }
};

// density pair (rho_A, rho_B) of a node, stored interleaved
template <class R>
struct Rho2;
template <>
struct Rho2<float> {
    using T = float2;
};
template <>
struct Rho2<double> {
    using T = double2;
};

// the node's 38 post-streaming populations (f[i]: component A, f[19 + i]: component B)
template <class S, class R>
__device__ __forceinline__ void pull3(const Geo3& g, const Nb3& nb, const Pair<S>* __restrict__ fs, const P3<R>& P,
                                      uint32_t fl, int s, R (&f)[38]) {
#pragma unroll
    for (int i = 0; i < 19; ++i) {
        int src, q;
        if (i > 0 && ((fl >> (i - 1)) & 1u)) {
            src = s;
            q = opp3(i);
        } else {
            src = i == 0 ? s : nb.at(-e3x(i), -e3y(i), -e3z(i));
            q = i;
        }
        const V2<R> v = ld3<S, R>(fs + (long long)q * g.N + src, P, q);
        f[i] = v.x;
        f[19 + i] = v.y;
    }
}

// k3_rho and k3_march follow each other as programmatic dependent launches: a block may be resident while
// the launch before it still writes what this one reads (the populations fs, the densities rho).  So
// those are plain coherent loads behind pdl_wait(), through pointers that promise nothing about the
// kernel's lifetime: no __ldg and no __restrict__, either of which makes them read-only loads that the
// compiler may move across the wait and that need not see the writes.  The flags never change.
template <class S, class R>
__global__ void __launch_bounds__(128) k3_rho(Geo3 g, P3<R> P, const uint32_t* __restrict__ flags, const Pair<S>* fs,
                                              typename Rho2<R>::T* rho) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
    pdl_wait();
    pdl_launch_next();
    if (x >= g.nx || y >= g.ny) return;
    const int s = (z * g.ny + y) * g.nx + x;
    const uint32_t fl = flags[s];
    typename Rho2<R>::T r;
    r.x = (R)-1;  // solid sites carry -1: the step kernel's wall path tells them apart by the sign
    r.y = (R)-1;
    if (!(fl & k3Solid)) {
        const Nb3 nb(g, x, y, z);
        V2<R> f[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            const bool bl = i > 0 && ((fl >> (i - 1)) & 1u);
            const int q = bl ? opp3(i) : i;
            f[i] = ld3<S, R>(fs + (long long)q * g.N + (bl || i == 0 ? s : nb.at(-e3x(i), -e3y(i), -e3z(i))), P, q);
        }
        // rho_k = sum_i f_i as a balanced tree (rounding grows with the depth, not the count), both
        // components at once
        const V2<R> a = vadd(vadd(vadd(f[0], f[1]), vadd(f[2], f[3])), vadd(vadd(f[4], f[5]), vadd(f[6], f[7])));
        const V2<R> b = vadd(vadd(vadd(f[8], f[9]), vadd(f[10], f[11])), vadd(vadd(f[12], f[13]), vadd(f[14], f[15])));
        r = vadd(vadd(a, b), vadd(f[16], vadd(f[17], f[18])));
    }
    rho[s] = r;
}

// record: mass A, mass B, mom x, y, z, max |u|^2 (|u| after the last combine), rhoA min/max, rhoB
// min/max, n, unstable
constexpr int k3DiagN = 12;

__device__ __forceinline__ double d3_combine(int q, double a, double b) {
    if (q == 5 || q == 7 || q == 9) return fmax(a, b);
    if (q == 6 || q == 8) return fmin(a, b);
    if (q == 11) return fmax(a, b);
    return a + b;
}
__device__ __forceinline__ double d3_neutral(int q) {
    return (q == 6 || q == 8) ? INFINITY : (q == 7 || q == 9) ? -INFINITY : 0.0;
}

// One thread's diagnostics.  The sums are FP64; the extrema compare in the compute type (exact), and
// |u|^2, taken in FP64, only where its value in the compute type could raise the maximum: FP64
// operations run at two per SM and cycle, and the record's were what the diagnostics pass waited for.
template <class R>
struct Diag3 {
    double mA = 0.0, mB = 0.0, px = 0.0, py = 0.0, pz = 0.0, u2 = 0.0;
    R near_u2 = (R)0, aMin = (R)INFINITY, aMax = (R)-INFINITY, bMin = (R)INFINITY, bMax = (R)-INFINITY;
    int n = 0;
    bool bad = false;
    __device__ __forceinline__ void add(R rA, R rB, const R (&u)[3]) {
        const double dr = (double)(rA + rB);
        mA += (double)rA;
        mB += (double)rB;
        px += dr * (double)u[0];
        py += dr * (double)u[1];
        pz += dr * (double)u[2];
        const R v = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        // v is within a few roundings of |u|^2 (a denormal or overflowing v says nothing)
        if (v >= near_u2 * (R)0.9999 || v < (R)1e-30 || !isfinite(v)) {
            const double w = (double)u[0] * u[0] + (double)u[1] * u[1] + (double)u[2] * u[2];
            u2 = fmax(u2, w);
            near_u2 = fmax(near_u2, isfinite(v) ? v : (R)0);
            if (!isfinite(w)) bad = true;
        }
        aMin = fmin(aMin, rA);
        aMax = fmax(aMax, rA);
        bMin = fmin(bMin, rB);
        bMax = fmax(bMax, rB);
        ++n;
        if (!(rA > (R)0) || !(rB > (R)0) || !isfinite(rA) || !isfinite(rB)) bad = true;
    }
    __device__ __forceinline__ void to_record(double (&v)[k3DiagN]) const {
        v[0] = mA; v[1] = mB; v[2] = px; v[3] = py; v[4] = pz; v[5] = u2;
        v[6] = (double)aMin; v[7] = (double)aMax; v[8] = (double)bMin; v[9] = (double)bMax;
        v[10] = (double)n; v[11] = bad ? 1.0 : 0.0;
    }
};

// ------------------------------------------------------------------------------------------------
// Step kernel of the 3-D form.  A block of 32 x 4 columns (x, y) marches over a chunk of z planes.
// The density pairs (rho_A, rho_B) of the planes z-2 .. z+2 over the block's columns and a halo of
// two on each side (36 x 8 sites per plane) sit in a six-plane shared-memory ring; solid sites
// hold -1, so nodes near the wall take the second-layer copy and the solid switch out of the ring
// as well.  Each thread loads its share of the halo of plane z+3 into registers while plane z is
// worked on, and the flags of the next plane.  Per plane: pull of the node's 38
// populations, stencil sums out of the ring, moments, forces, collision, store; one barrier.  Both
// components share each instruction: densities, gradients, forces and populations are (A, B) pairs.
// ------------------------------------------------------------------------------------------------
constexpr int k3TX = 32, k3TY = 4, k3T = k3TX * k3TY;   // block = 32 x 4 columns
constexpr int k3HX = k3TX + 4, k3HY = k3TY + 4;           // halo region of one plane: 36 x 8
constexpr int k3HP = k3HX * k3HY;
constexpr int k3HN = (k3HP + k3T - 1) / k3T;              // halo sites loaded per thread
constexpr int k3Ring = 6;                                 // density planes resident

template <class R>
constexpr size_t k3_ring_bytes() {
    return (size_t)k3Ring * k3HP * sizeof(V2<R>);
}
template <class R>
constexpr size_t k3_march_smem() {
    return k3_ring_bytes<R>();
}

// Stencil sums of a node whose stencil reaches a solid site: second-layer copy of x + sign(e) for a
// solid second-layer site (Sec. 2.4), density 0 and solid switch 1 at a solid site; solid sites
// hold -1 in the ring.  b0..b4: ring rows of the planes z-2..z+2 at the node.  (Inlined: an
// out-of-line call measured 7 % slower on the full case and twice as slow on a small one.)
template <class R, int kAdh>
__device__ __forceinline__ void wall_stencil3(const V2<R>* b0, const V2<R>* b1, const V2<R>* b2, const V2<R>* b3,
                                           const V2<R>* b4, V2<R>& gx, V2<R>& gy, V2<R>& gz, R (&ad)[3]) {
    using V = V2<R>;
    const V* bs[5] = {b0, b1, b2, b3, b4};
#pragma unroll
    for (int dz = 0; dz <= 2; ++dz)
#pragma unroll
        for (int dy = -2; dy <= 2; ++dy)
#pragma unroll
            for (int dx = -2; dx <= 2; ++dx) {
                if (dz == 0 && (dy < 0 || (dy == 0 && dx <= 0))) continue;
                const int q = dx * dx + dy * dy + dz * dz;
                const double wq = w92(q);
                if (wq == 0.0) continue;
                const bool second = dx == 2 || dx == -2 || dy == 2 || dy == -2 || dz == 2 || dz == -2;
                V v[2];
                R vs[2];
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                    const int sg = side == 0 ? 1 : -1;
                    const int ex = sg * dx, ey = sg * dy, ez = sg * dz;
                    V w = bs[2 + ez][ey * k3HX + ex];
                    const bool own = w.x < (R)0;
                    if (second && own) {
                        const int fx = (ex > 0) - (ex < 0), fy = (ey > 0) - (ey < 0), fz = (ez > 0) - (ez < 0);
                        w = bs[2 + fz][fy * k3HX + fx];
                    }
                    const bool sol = w.x < (R)0;
                    v[side] = sol ? vbc<R>(0) : w;
                    vs[side] = (sol || (kAdh == kAdhE8Psi && own)) ? (R)1 : (R)0;
                }
                const V a = vsub(v[0], v[1]);
                gx = vfma(vbc<R>(wq * dx), a, gx);
                gy = vfma(vbc<R>(wq * dy), a, gy);
                gz = vfma(vbc<R>(wq * dz), a, gz);
                const double wa = kAdh == kAdhD3Q19 ? w19q(q) : wq;
                if (wa != 0.0) {
                    const R w = (R)wa, sw = vs[0] - vs[1];
                    ad[0] += w * dx * sw;
                    ad[1] += w * dy * sw;
                    ad[2] += w * dz * sw;
                }
            }
}

#ifndef LBM3_MIN_BLOCKS
#define LBM3_MIN_BLOCKS 3
#endif
// Blocks per SM.  16-bit storage, whose DRAM time is half, waits for its pulls' latency: with the pulled
// pairs held as stored behind the stencil sums (19 registers, not 38) and one density plane in flight it
// fits 128 registers, four blocks (no spill in the step but for 8 bytes with the D3Q19 adhesion; the fields
// forms spill up to 136 bytes) (100 x 100 x 140: 120.0 -> 105.2 us a step, three blocks
// of the same form 113.6; 200 x 200 x 280: 730 -> 637, 677).  FP32 spills at four and is slower (851 -> 897).
#ifndef LBM3_MIN_BLOCKS_16
#define LBM3_MIN_BLOCKS_16 4
#endif
template <class S>
__host__ __device__ constexpr int march_blocks() {
    return sizeof(S) == 8 ? 2 : (sizeof(S) == 2 ? LBM3_MIN_BLOCKS_16 : LBM3_MIN_BLOCKS);
}
// kMode: kStep collides.  The fields forms write rho_A, rho_B and u (FP64, each of o5 may be NULL) in
// place of the collision; kFieldsDiag also adds each node's values to the thread's diagnostic record,
// and each block writes one record (block index blockIdx.x + gridDim.x (blockIdx.y + gridDim.y
// blockIdx.z)) to part.  Apart, since the FP64 sums of the records run at two operations per SM and
// cycle: reading the fields of 200 x 200 x 280 took 1.0 ms with them.
enum { kStep = 0, kFieldsOnly = 1, kFieldsDiag = 2 };
struct Out5 {
    double* p[5];
};
template <class S, class R, int kAdh, int kMode = kStep>
__global__ void __launch_bounds__(k3T, march_blocks<S>())
    k3_march(Geo3 g, P3<R> P, int zc, const uint32_t* __restrict__ flags, const Pair<S>* fs, const V2<R>* rho,
             Pair<S>* fout, Out5 o5, double* part) {
    using V = V2<R>;
    constexpr bool kFields = kMode != kStep, kDiag = kMode == kFieldsDiag;
    extern __shared__ __align__(16) unsigned char smem3[];
    V* ring = reinterpret_cast<V*>(smem3);
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * k3TX + tx;
    const int x0 = blockIdx.x * k3TX, y0 = blockIdx.y * k3TY;
    const int x = x0 + tx, y = y0 + ty;
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, g.nz);
    const bool active = x < g.nx && y < g.ny;
    const int nxy = g.nx * g.ny;

    // this thread's halo sites: in-plane offsets of the wrapped columns
    int hoff[k3HN];
#pragma unroll
    for (int k = 0; k < k3HN; ++k) {
        const int j = t + k * k3T;
        const int hx = j % k3HX, hy = j / k3HX;
        const int gx = ((x0 - 2 + hx) % g.nx + g.nx) % g.nx, gy = ((y0 - 2 + hy) % g.ny + g.ny) % g.ny;
        hoff[k] = j < k3HP ? gy * g.nx + gx : -1;
    }
    auto load_plane = [&](int p, V (&v)[k3HN]) {
        const int zo = wrapc(p, g.nz) * nxy;
#pragma unroll
        for (int k = 0; k < k3HN; ++k)
            if (hoff[k] >= 0) v[k] = rho[zo + hoff[k]];
    };
    auto slot = [&](int p) -> int { return wrapc(p % k3Ring, k3Ring); };  // ring slot of plane p >= -2
    auto store_plane = [&](int p, const V (&v)[k3HN]) {
        V* dst = ring + slot(p) * k3HP;
#pragma unroll
        for (int k = 0; k < k3HN; ++k)
            if (hoff[k] >= 0) dst[t + k * k3T] = v[k];
    };
    const int yx = active ? y * g.nx + x : 0;
    const Nb3 nb(g, active ? x : 0, active ? y : 0, 0);
    // the node's 38 populations at plane z: f_i(x) = f*_i(x - e_i), or f*_opp(i)(x) across a blocked link
    // (16-bit storage: as stored; widened where they are used, behind the stencil sums)
    using Held = typename std::conditional<sizeof(S) == 2, Pair<S>, V>::type;
    auto pull_plane = [&](int z, uint32_t fl, Held (&f)[19]) {
        const int s = z * nxy + yx;
        const int zoff[3] = {wrapc(z - 1, g.nz) * nxy, z * nxy, wrapc(z + 1, g.nz) * nxy};
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            int src, q;
            if (i > 0 && ((fl >> (i - 1)) & 1u)) {
                src = s;
                q = opp3(i);
            } else {
                src = i == 0 ? s : zoff[1 - e3z(i)] + nb.yo[2 - e3y(i)] + nb.xw[2 - e3x(i)];
                q = i;
            }
            if constexpr (sizeof(S) == 2) f[i] = fs[(long long)q * g.N + src];
            else f[i] = ld3<S, R>(fs + (long long)q * g.N + src, P, q);
        }
    };

    Diag3<R> diag;  // kFieldsDiag
    pdl_wait();
    pdl_launch_next();

    // prologue: planes z0-2 .. z0+2 into the ring, plane z0+3 into registers, populations of z0
    uint32_t fl_nx = active ? flags[z0 * nxy + yx] : k3Solid;
    {
        V v[5][k3HN];
#pragma unroll
        for (int d = 0; d < 5; ++d) load_plane(z0 - 2 + d, v[d]);
#pragma unroll
        for (int d = 0; d < 5; ++d) store_plane(z0 - 2 + d, v[d]);
    }
    __syncthreads();

    for (int z = z0; z < z1; ++z) {
        V nxt[k3HN];  // enters the ring when this plane is done; planes up to z1 + 1 are needed
        if (z + 3 <= z1 + 1) load_plane(z + 3, nxt);
        const uint32_t fl = fl_nx;  // the flags are loaded one plane ahead
        if (z + 1 < z1 && active) fl_nx = flags[(z + 1) * nxy + yx];
        const int s = z * nxy + yx;
        if (!(fl & k3Solid)) {
            Held held[19];
            pull_plane(z, fl, held);
            // the node's stencil out of the ring: bs[d] = plane z - 2 + d at the node's column
            const V* bs[5];
#pragma unroll
            for (int d = 0; d < 5; ++d) bs[d] = ring + slot(z - 2 + d) * k3HP + (ty + 2) * k3HX + (tx + 2);
            const V r2 = bs[2][0];
            V gx = vbc<R>(0), gy = vbc<R>(0), gz = vbc<R>(0);  // (A, B) density gradients
            R ad[3] = {(R)0, (R)0, (R)0};
            if (!(fl & k3Wall)) {
                // symmetric pairs (e, -e): w e (rho(x+e) - rho(x-e)), the differences first; two sets
                // of partial sums (odd / even dx) shorten the dependency chains
                V hx[2] = {gx, gx}, hy[2] = {gy, gy}, hz[2] = {gz, gz};
#pragma unroll
                for (int dz = 0; dz <= 2; ++dz)
#pragma unroll
                    for (int dy = -2; dy <= 2; ++dy)
#pragma unroll
                        for (int dx = -2; dx <= 2; ++dx) {
                            if (dz == 0 && (dy < 0 || (dy == 0 && dx <= 0))) continue;  // one of each pair
                            const int q = dx * dx + dy * dy + dz * dz;
                            if (w92(q) == 0.0) continue;
                            const int h = dx & 1;
                            const V a = vsub(bs[2 + dz][dy * k3HX + dx], bs[2 - dz][-dy * k3HX - dx]);
                            if (dx != 0) hx[h] = vfma(vbc<R>(w92(q) * dx), a, hx[h]);
                            if (dy != 0) hy[h] = vfma(vbc<R>(w92(q) * dy), a, hy[h]);
                            if (dz != 0) hz[h] = vfma(vbc<R>(w92(q) * dz), a, hz[h]);
                        }
                gx = vadd(hx[0], hx[1]);
                gy = vadd(hy[0], hy[1]);
                gz = vadd(hz[0], hz[1]);
            } else {
                wall_stencil3<R, kAdh>(bs[0], bs[1], bs[2], bs[3], bs[4], gx, gy, gz, ad);
            }
            const R rA = r2.x, rB = r2.y;
            R GA = (R)0;
            if (fl & k3Wall) {
                if (P.mode == 1) {
                    const R re = (rA - rB) / (rA + rB);
                    R h;
                    if (re > P.delta) h = P.lam;
                    else if (re > (R)0) h = P.s1 + re * (P.s2 + re * P.s3);
                    else if (re > -P.delta) h = P.s1 + re * (P.t2 + re * P.t3);
                    else h = (R)1;
                    GA = P.Gw2 * h;
                } else {
                    GA = P.lam * P.Gw2;
                }
            }
            V f[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                if constexpr (sizeof(S) == 2) f[i] = ld3<S, R>(&held[i], P, i);  // opposite directions share w rho0
                else f[i] = held[i];
            }
            // momentum per component from the differences of opposite populations (i odd, opp = i + 1)
            V mv[3] = {vbc<R>(0), vbc<R>(0), vbc<R>(0)};
#pragma unroll
            for (int i = 1; i < 19; i += 2) {
                const V d = vsub(f[i], f[i + 1]);
                if (e3x(i) != 0) mv[0] = e3x(i) > 0 ? vadd(mv[0], d) : vsub(mv[0], d);
                if (e3y(i) != 0) mv[1] = e3y(i) > 0 ? vadd(mv[1], d) : vsub(mv[1], d);
                if (e3z(i) != 0) mv[2] = e3z(i) > 0 ? vadd(mv[2], d) : vsub(mv[2], d);
            }
            const V gv[3] = {gx, gy, gz};
            const R inv = recip(rA + rB);
            V F[3];
            R u[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                // each component is pushed by the other's gradient (Eq. 8); adhesion (Eq. 9); body force
                const R FA = -P.G * rA * gv[d].y - GA * rA * ad[d] + rA * P.g[d];
                const R FB = -P.G * rB * gv[d].x - P.Gw2 * rB * ad[d] + rB * P.g[d];
                F[d] = V{FA, FB};
                u[d] = ((mv[d].x + mv[d].y) + (R)0.5 * (FA + FB)) * inv;
            }
            if constexpr (kFields) {
                if (o5.p[0]) o5.p[0][s] = (double)rA;
                if (o5.p[1]) o5.p[1][s] = (double)rB;
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (o5.p[2 + d]) o5.p[2 + d][s] = (double)u[d];
                if constexpr (kDiag) diag.add(rA, rB, u);
            } else {
                // SRT collision with Guo forcing, per pair of directions (e, -e), both components at
                // once.  With a = e.u, b = e.F_k, P = om rho a + cF b, C0 = om rho (1 - 1.5u^2) - 3 cF u.F:
                //   f*_+- = (1 - om) f_+- + w (C0 + 4.5 a (P + cF b)) +- 3 w P,  f*_0 = (1 - om) f_0 + w_0 C0
                const V om = V{P.omega[0], P.omega[1]}, cf = V{P.cF[0], P.cF[1]};
                const V om1 = vsub(vbc<R>(1), om);
                const V wr = vmul(om, r2);
                const V u2v[3] = {vbc<R>(u[0]), vbc<R>(u[1]), vbc<R>(u[2])};
                const R tq = (R)1 - (R)1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                const V uF = vfma(u2v[2], F[2], vfma(u2v[1], F[1], vmul(u2v[0], F[0])));
                const V C0 = vfma(wr, vbc<R>(tq), vmul(vmul(vbc<R>(-3), cf), uF));
                V o[19];
                o[0] = vfma(om1, f[0], vmul(vbc<R>(w19c<R>(0)), C0));
                const V sAx = vmul(vbc<R>(w19c<R>(1)), C0), sDg = vmul(vbc<R>(w19c<R>(7)), C0);
#pragma unroll
                for (int i = 1; i < 19; i += 2) {
                    auto dot = [&](const V* vv) -> V {  // e_i . vv for a pair-valued vector
                        V r = vbc<R>(0);
                        bool first = true;
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const int e = d == 0 ? e3x(i) : d == 1 ? e3y(i) : e3z(i);
                            if (e == 0) continue;
                            if (first) r = e > 0 ? vv[d] : vsub(vbc<R>(0), vv[d]);
                            else r = e > 0 ? vadd(r, vv[d]) : vsub(r, vv[d]);
                            first = false;
                        }
                        return r;
                    };
                    const double w = w19c<R>(i);
                    const V a = dot(u2v), b = dot(F);
                    const V cb = vmul(cf, b);
                    const V Pp = vfma(wr, a, cb);
                    const V sym = vfma(vbc<R>(4.5 * w), vmul(a, vadd(Pp, cb)), i <= 6 ? sAx : sDg);
                    const V anti = vmul(vbc<R>(3.0 * w), Pp);
                    o[i] = vfma(om1, f[i], vadd(sym, anti));
                    o[i + 1] = vfma(om1, f[i + 1], vsub(sym, anti));
                }
#pragma unroll
                for (int i = 0; i < 19; ++i) st3<S, R>(fout + (long long)i * g.N + s, o[i], P, i);
            }
        } else if constexpr (kFields) {  // solid node: zero fields
            if (active)
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    if (o5.p[q]) o5.p[q][s] = 0.0;
        }
        if (z + 3 <= z1 + 1) store_plane(z + 3, nxt);
        __syncthreads();
    }
    if constexpr (kDiag) {  // the block's record: warps by shuffles, then the warps in order
        __shared__ double red[k3T / 32][k3DiagN];
        const int lane = t & 31, warp = t >> 5;
        double rec[k3DiagN];
        diag.to_record(rec);
#pragma unroll
        for (int q = 0; q < k3DiagN; ++q) {
            double v = rec[q];
            for (int off = 16; off > 0; off >>= 1) v = d3_combine(q, v, __shfl_xor_sync(0xffffffffu, v, off));
            if (lane == 0) red[warp][q] = v;
        }
        __syncthreads();
        if (t == 0) {
            const long long b = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
            for (int q = 0; q < k3DiagN; ++q) {
                double v = red[0][q];
                for (int w = 1; w < k3T / 32; ++w) v = d3_combine(q, v, red[w][q]);
                part[b * k3DiagN + q] = v;
            }
        }
    }
}

// Combine the per-block records in two levels, each in a fixed order (deterministic): k3DiagMid
// blocks each combine a contiguous range of records (a thread takes whole records, strided by the
// block size; then a shuffle tree and the warps in order), then one warp combines their k3DiagMid
// results (k3_diag_final).  A single warp over all records waited on one dependent load per record.
constexpr int k3DiagMid = 256, k3DiagMidThreads = 256;
__global__ void __launch_bounds__(k3DiagMidThreads) k3_diag_mid(long long nblocks, const double* __restrict__ part,
                                                               double* __restrict__ mid) {
    const long long per = (nblocks + gridDim.x - 1) / gridDim.x;
    const long long b0 = (long long)blockIdx.x * per, b1 = b0 + per < nblocks ? b0 + per : nblocks;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    double v[k3DiagN];
#pragma unroll
    for (int q = 0; q < k3DiagN; ++q) v[q] = d3_neutral(q);
    for (long long b = b0 + t; b < b1; b += k3DiagMidThreads) {
#pragma unroll
        for (int q = 0; q < k3DiagN; ++q) v[q] = d3_combine(q, v[q], part[b * k3DiagN + q]);
    }
    __shared__ double red[k3DiagMidThreads / 32][k3DiagN];
#pragma unroll
    for (int q = 0; q < k3DiagN; ++q) {
        double x = v[q];
        for (int off = 16; off > 0; off >>= 1) x = d3_combine(q, x, __shfl_xor_sync(0xffffffffu, x, off));
        if (lane == 0) red[warp][q] = x;
    }
    __syncthreads();
    if (t < k3DiagN) {
        double x = red[0][t];
        for (int w = 1; w < k3DiagMidThreads / 32; ++w) x = d3_combine(t, x, red[w][t]);
        mid[(long long)blockIdx.x * k3DiagN + t] = x;
    }
}

// Combine records in record order (one warp per value; deterministic); max |u| from max |u|^2.
__global__ void __launch_bounds__(32 * k3DiagN) k3_diag_final(long long nblocks, const double* __restrict__ part,
                                                             double* __restrict__ out) {
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double v = d3_neutral(q);
    for (long long b = lane; b < nblocks; b += 32) v = d3_combine(q, v, part[b * k3DiagN + q]);
    for (int off = 16; off > 0; off >>= 1) v = d3_combine(q, v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) out[q] = q == 5 ? sqrt(v) : v;
}

// post-streaming populations (FP64 [2][19][N]) <-> post-collision buffer
template <class S, class R>
__global__ void k3_get(Geo3 g, P3<R> P, const uint32_t* __restrict__ flags, const Pair<S>* __restrict__ fs,
                       double* __restrict__ f) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long s = ((long long)z * g.ny + y) * g.nx + x;
    const uint32_t fl = flags[s];
    R v[38];
    if (fl & k3Solid) {
        for (int q = 0; q < 38; ++q) v[q] = (R)0;
    } else {
        const Nb3 nb(g, x, y, z);
        pull3<S, R>(g, nb, fs, P, fl, (int)s, v);
    }
    for (int q = 0; q < 38; ++q) f[(long long)q * g.N + s] = (double)v[q];
}

template <class S, class R>
__global__ void k3_set(Geo3 g, P3<R> P, const uint32_t* __restrict__ flags, const double* __restrict__ f,
                       Pair<S>* __restrict__ fs) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long s = ((long long)z * g.ny + y) * g.nx + x;
    const uint32_t fl = flags[s];
    for (int i = 0; i < 19; ++i) {
        R v[2] = {(R)0, (R)0};
        for (int k = 0; k < 2; ++k)
            if (!(fl & k3Solid)) {
                // f*_i(x) streams to x + e_i; if that node is solid it comes back as f_opp(i)(x)
                if (i > 0 && ((fl >> (opp3(i) - 1)) & 1u)) v[k] = (R)f[(long long)(19 * k + opp3(i)) * g.N + s];
                else v[k] = (R)f[(long long)(19 * k + i) * g.N + (i == 0 ? s : site(g, x + e3x(i), y + e3y(i), z + e3z(i)))];
            }
        if (fl & k3Solid) store_pair<S, R>(fs + (long long)i * g.N + s, (R)0, (R)0);
        else st3<S, R>(fs + (long long)i * g.N + s, V2<R>{v[0], v[1]}, P, i);
    }
}

// f = f^eq(rho_k, 0) written straight into the post-collision buffer as the pull expects it: the
// stored f*_i at x is w_i rho(x + e_i), or w_i rho(x) when x + e_i is solid (the link comes back by
// bounce-back), minus the storage shift, and 0 at solid nodes.  The value is (R)(w_i rho) with an FP64
// product.  1/18 and 1/36 in FP64 are a factor of two apart, so the axis populations are exactly twice
// q = (R)(rho / 36): per node and component one FP64 product and conversion for q and one for the rest
// population, instead of 19 (the pass ran at the FP64 pipe's rate, two operations per SM and cycle:
// 1.61 ms on 200 x 200 x 280 in FP32, where its 168 B per node take 0.28 ms of HBM time; now 0.36 ms).
// A q so small that scaling it up could differ from rounding the larger product takes the direct form.
//
// A block of 32 x 8 columns marches along `planes` planes of z; q of the plane ahead, with a halo of one
// node, goes into a ring of four shared-memory planes, one barrier per plane.  At most kR3Z planes, and
// fewer where those do not fill the GPU (us, 16 planes -> this rule, FP32 / FP64:
// 24 x 24 x 34 31.1 -> 6.4 / 51.3 -> 6.4, 40 x 40 x 56 34.7 -> 12.6 / 56.6 -> 13.3, 64^3 33.4 -> 16.8 / 57.3 -> 20.9).
constexpr int kR3X = 32, kR3Y = 8, kR3T = kR3X * kR3Y, kR3Z = 16;
constexpr int kR3HX = kR3X + 2, kR3P = kR3HX * (kR3Y + 2), kR3N = (kR3P + kR3T - 1) / kR3T;

template <class S, class R>
__global__ void __launch_bounds__(kR3T) k3_set_rest(Geo3 g, P3<R> P, int planes,
                                                    const uint32_t* __restrict__ flags,
                                                    const double* __restrict__ rA, const double* __restrict__ rB,
                                                    Pair<S>* __restrict__ fs) {
    using V = V2<R>;
    __shared__ V ring[4][kR3P];
    const int tx = threadIdx.x, ty = threadIdx.y, t = ty * kR3X + tx;
    const int x0 = blockIdx.x * kR3X, y0 = blockIdx.y * kR3Y, x = x0 + tx, y = y0 + ty;
    const int z0 = blockIdx.z * planes, z1 = min(z0 + planes, g.nz);
    const bool active = x < g.nx && y < g.ny;
    const long long nxy = (long long)g.nx * g.ny;
    int hoff[kR3N];  // in-plane offsets of this thread's halo sites
#pragma unroll
    for (int k = 0; k < kR3N; ++k) {
        const int j = t + k * kR3T;
        const int hx = x0 - 1 + j % kR3HX, hy = y0 - 1 + j / kR3HX;
        hoff[k] = j < kR3P ? ((hy + g.ny) % g.ny) * g.nx + (hx + g.nx) % g.nx : -1;
    }
    double nA[kR3N], nB[kR3N];  // densities of the plane about to enter the ring
    auto load = [&](int z) {
        const long long o = (long long)wrapc(z, g.nz) * nxy;
#pragma unroll
        for (int k = 0; k < kR3N; ++k)
            if (hoff[k] >= 0) {
                nA[k] = rA[o + hoff[k]];
                nB[k] = rB[o + hoff[k]];
            }
    };
    auto put = [&](int z) {
#pragma unroll
        for (int k = 0; k < kR3N; ++k)
            if (hoff[k] >= 0) ring[(z + 4) & 3][t + k * kR3T] = V{(R)(w19(7) * nA[k]), (R)(w19(7) * nB[k])};
    };
    auto tiny = [&](R q) {  // 0 too: twice what rounds to 0 need not
        if constexpr (sizeof(R) == 8) return (__double2hiint(q) & 0x7fffffff) < (60 << 20);  // below 2^-963
        else return q < (R)1e-30 && q > (R)-1e-30;
    };
    load(z0 - 1);
    put(z0 - 1);
    load(z0);
    put(z0);
    load(z0 + 1);
    const int c0 = (ty + 1) * kR3HX + tx + 1;
    for (int z = z0; z < z1; ++z) {
        put(z + 1);
        if (z + 1 < z1) load(z + 2);
        __syncthreads();
        if (!active) continue;
        const long long s = (long long)z * nxy + (long long)y * g.nx + x;
        const uint32_t fl = flags[s];
        if (fl & k3Solid) {
#pragma unroll
            for (int i = 0; i < 19; ++i) store_pair<S, R>(fs + (long long)i * g.N + s, (R)0, (R)0);
            continue;
        }
        st3<S, R>(fs + s, V{(R)(w19(0) * rA[s]), (R)(w19(0) * rB[s])}, P, 0);
        const V own = ring[(z + 4) & 3][c0];
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const bool bl = (fl >> (opp3(i) - 1)) & 1u;
            const V q = bl ? own : ring[(z + e3z(i) + 4) & 3][c0 + e3y(i) * kR3HX + e3x(i)];
            const R up = (R)(i <= 6 ? 2 : 1);
            V v{q.x * up, q.y * up};
            if (i <= 6 && (tiny(q.x) || tiny(q.y))) {
                const long long n = bl ? s : site(g, x + e3x(i), y + e3y(i), z + e3z(i));
                v = V{(R)(w19(i) * rA[n]), (R)(w19(i) * rB[n])};
            }
            st3<S, R>(fs + (long long)i * g.N + s, v, P, i);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Contact angle on a sphere (FP64): interface points, algebraic sphere fit, one Gauss-Newton step
// ------------------------------------------------------------------------------------------------
constexpr int kC3Threads = 256;
constexpr int kC3Blocks = 304;  // fixed: the summation order does not depend on the device
constexpr int kC3Vals = 14;
constexpr int kC3Seg = 4 * kC3Threads;  // nodes of a block of k3_ca_cross
constexpr int kC3Group = 4 * kC3Seg;    // nodes a block of a pass works on together

template <class R>
struct Ca3 {
    Geo3 g;
    const uint32_t* flags;
    const typename Rho2<R>::T* rho;  // interleaved (rho_A, rho_B)
    uint8_t* cross;                  // per node: bit a set where the link to the +a neighbour crosses
                                     // rho^e = 0 (written by k3_ca_cross, read by the passes)
    int* count;                      // links that cross, per kC3Seg nodes
};

__device__ __forceinline__ double phi3(double a, double b) { return (a - b) / (a + b); }
__device__ __forceinline__ bool phi3_pos(double a, double b) {
    if (a == b) return false;  // 0 or undefined; solid sites hold equal values, and take no division
    const double sum = a + b;
    return (sum > 0.0 && sum < INFINITY) ? a > b : phi3(a, b) > 0.0;
}
// phi3_pos of densities in the compute type.  For finite FP32 values with a positive FP32 sum the
// FP64 test reduces to a > b (the FP64 sum of two floats is finite and has the sign of their FP32
// sum; the comparison is exact in either type), so FP32 takes it without the FP64 pipe; every other
// case goes through the FP64 form.  The decision is the FP64 one bit for bit.
__device__ __forceinline__ bool phi3_pos_r(float a, float b) {
    if (a == b) return false;
    if (isfinite(a) && isfinite(b) && a + b > 0.0f) return a > b;
    return phi3_pos((double)a, (double)b);
}
__device__ __forceinline__ bool phi3_pos_r(double a, double b) { return phi3_pos(a, b); }

// st: 0 N, 1-3 centroid, 4-6 centre, 7 r, 8 rms, 9 theta, 10 status (1: too few points)
// Crossing links of every node.  The links of a node are tested by the signs of rho^e alone, a thread's
// four nodes and their neighbours in flight together; flags and coordinates (a usable pair of nodes, no
// pair across the periodic seam) are looked at only where a sign changes.  As part of a pass over all
// nodes that looked at the flags first, one node after the other, it took 387 us on 200 x 200 x 280
// (the whole angle 0.95 ms; now 0.24 ms after the density pass).
template <class R>
__global__ void __launch_bounds__(kC3Threads) k3_ca_cross(Ca3<R> c) {
    const unsigned nx = c.g.nx, ny = c.g.ny, n = (unsigned)c.g.N;  // N < 2^31
    const unsigned base = blockIdx.x * kC3Seg + threadIdx.x;
    const unsigned step[3] = {1u, nx, nx * ny};
    typename Rho2<R>::T r[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned s = min(base + j * kC3Threads, n - 1);
        r[j][0] = c.rho[s];
#pragma unroll
        for (int a = 0; a < 3; ++a) r[j][1 + a] = c.rho[min(s + step[a], n - 1)];
    }
    uint32_t change[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const bool p = phi3_pos_r(r[j][0].x, r[j][0].y);
        change[j] = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (p != phi3_pos_r(r[j][1 + a].x, r[j][1 + a].y)) change[j] |= 1u << a;
        if (base + j * kC3Threads >= n) change[j] = 0;
    }
    int links = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const unsigned s = base + j * kC3Threads;
        uint32_t found = 0;
        if (change[j]) {
            const unsigned row = s / nx, at[3] = {s - row * nx, row % ny, row / ny};
            const unsigned lim[3] = {nx, ny, (unsigned)c.g.nz};
            uint32_t fl[4];
            fl[0] = c.flags[s];
#pragma unroll
            for (int a = 0; a < 3; ++a) fl[1 + a] = c.flags[min(s + step[a], n - 1)];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if ((change[j] >> a & 1u) && at[a] + 1 < lim[a] && ((fl[0] | fl[1 + a]) & (k3Solid | k3Near)) == 0)
                    found |= 1u << a;
        }
        c.cross[s] = (uint8_t)found;  // the array is padded to whole groups
        links += __popc(found);
    }
    __shared__ int red[kC3Threads / 32];
    links = __reduce_add_sync(0xffffffffu, links);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = links;
    __syncthreads();
    if (threadIdx.x == 0) {
        int v = 0;
        for (int w = 0; w < kC3Threads / 32; ++w) v += red[w];
        c.count[blockIdx.x] = v;
    }
}

// st: 0 N, 1-3 centroid, 4-6 centre, 7 r, 8 rms, 9 theta, 10 status (1: too few points)
// One kernel per pass over the crossing links (kPass 0: count and centroid, 1: algebraic fit sums, 2:
// Gauss-Newton sums, 3: residual), so that each holds only the sums it needs.  Block b takes the
// groups of nodes b, b + gridDim.x, ... that hold any link (most hold none) and packs a group's links in
// node order, so that whole warps work on them: the FP64 divisions of a link cost a warp as much as
// those of 32.
template <class R, int kPass>
__global__ void __launch_bounds__(kC3Threads) k3_ca_pass(Ca3<R> c, int ngroup, const double* __restrict__ st,
                                                        double* __restrict__ part) {
    constexpr int pass = kPass;
    constexpr int nv = pass == 0 ? 4 : pass == 1 ? 13 : pass == 2 ? 14 : 1;  // sums this pass forms
    __shared__ uint16_t keys[3 * kC3Group];  // 4 x node within the group + axis
    __shared__ int warp_sum[kC3Threads / 32];
    double acc[kC3Vals];
#pragma unroll
    for (int q = 0; q < kC3Vals; ++q) acc[q] = 0.0;
    const double m0 = st[1], m1 = st[2], m2 = st[3], c0 = st[4], c1 = st[5], c2 = st[6], r = st[7];
    const unsigned nx = c.g.nx, ny = c.g.ny;
    auto link = [&](unsigned s, int axis) {
        const unsigned row = s / nx;
        const typename Rho2<R>::T r0 = c.rho[s], r1 = c.rho[s + (axis == 0 ? 1u : (axis == 1 ? nx : nx * ny))];
        const double a = phi3((double)r0.x, (double)r0.y), b = phi3((double)r1.x, (double)r1.y), d = a / (a - b);
        const double p[3] = {(double)(s - row * nx) + (axis == 0 ? d : 0.0), (double)(row % ny) + (axis == 1 ? d : 0.0),
                             (double)(row / ny) + (axis == 2 ? d : 0.0)};
        if constexpr (pass == 0) {
            acc[0] += 1.0;
            acc[1] += p[0];
            acc[2] += p[1];
            acc[3] += p[2];
        } else if constexpr (pass == 1) {
            const double q0 = p[0] - m0, q1 = p[1] - m1, q2 = p[2] - m2, qq = q0 * q0 + q1 * q1 + q2 * q2;
            acc[0] += q0 * q0; acc[1] += q0 * q1; acc[2] += q0 * q2;
            acc[3] += q1 * q1; acc[4] += q1 * q2; acc[5] += q2 * q2;
            acc[6] += q0; acc[7] += q1; acc[8] += q2;
            acc[9] += q0 * qq; acc[10] += q1 * qq; acc[11] += q2 * qq; acc[12] += qq;
        } else if constexpr (pass == 2) {
            const double d0 = p[0] - c0, d1 = p[1] - c1, d2 = p[2] - c2;
            const double dd = sqrt(d0 * d0 + d1 * d1 + d2 * d2), res = dd - r;
            const double j[4] = {-d0 / dd, -d1 / dd, -d2 / dd, -1.0};
            int k = 0;
#pragma unroll
            for (int a2 = 0; a2 < 4; ++a2)
#pragma unroll
                for (int b2 = a2; b2 < 4; ++b2) acc[k++] += j[a2] * j[b2];
#pragma unroll
            for (int a2 = 0; a2 < 4; ++a2) acc[10 + a2] += j[a2] * res;
        } else {
            const double d0 = p[0] - c0, d1 = p[1] - c1, d2 = p[2] - c2;
            const double res = sqrt(d0 * d0 + d1 * d1 + d2 * d2) - r;
            acc[0] += res * res;
        }
    };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nb = (int)gridDim.x;
    for (int first = blockIdx.x; first < ngroup; first += 32 * nb) {  // the counts of 32 groups together
        const long long mine = (long long)first + (long long)lane * nb;
        int4 n4 = make_int4(0, 0, 0, 0);
        if (mine < ngroup) n4 = reinterpret_cast<const int4*>(c.count)[mine];
        uint32_t left = __ballot_sync(0xffffffffu, (n4.x | n4.y | n4.z | n4.w) != 0);
        while (left) {  // the same in every warp
            const unsigned group = (unsigned)first + (unsigned)(__ffs(left) - 1) * nb;
            left &= left - 1;
            const uint4 w = *reinterpret_cast<const uint4*>(c.cross + (size_t)group * kC3Group + 16 * threadIdx.x);
            const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
            const int mylinks = __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
            int at = mylinks;  // inclusive prefix over the block's threads
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, at, off);
                if (lane >= off) at += o;
            }
            if (lane == 31) warp_sum[warp] = at;
            __syncthreads();
            int total = 0;
            for (int k = 0; k < kC3Threads / 32; ++k) {
                if (k < warp) at += warp_sum[k];
                total += warp_sum[k];
            }
            at -= mylinks;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                for (uint32_t v = ws[k]; v; v &= v - 1) {  // bit 8 node + axis
                    const int b = __ffs(v) - 1;
                    keys[at++] = (uint16_t)((16 * threadIdx.x + 4 * k + (b >> 3)) * 4 + (b & 7));
                }
            __syncthreads();
            for (int k = threadIdx.x; k < total; k += kC3Threads) link(group * kC3Group + (keys[k] >> 2), keys[k] & 3);
            __syncthreads();
        }
    }
    __shared__ double red[kC3Threads / 32][kC3Vals];
#pragma unroll
    for (int q = 0; q < nv; ++q) {
        double v = acc[q];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) red[warp][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < kC3Vals) {  // the sums a pass does not form are written as 0
        double v = 0.0;
        if ((int)threadIdx.x < nv)
            for (int w = 0; w < kC3Threads / 32; ++w) v += red[w][threadIdx.x];
        part[blockIdx.x * kC3Vals + threadIdx.x] = v;
    }
}

__device__ void solve4(double A[4][4], double b[4], double x[4]) {
    for (int c = 0; c < 4; ++c) {
        int p = c;
        for (int r = c + 1; r < 4; ++r)
            if (fabs(A[r][c]) > fabs(A[p][c])) p = r;
        for (int k = 0; k < 4; ++k) {
            const double t = A[c][k];
            A[c][k] = A[p][k];
            A[p][k] = t;
        }
        const double t = b[c];
        b[c] = b[p];
        b[p] = t;
        for (int r = c + 1; r < 4; ++r) {
            const double f = A[r][c] / A[c][c];
            for (int k = c; k < 4; ++k) A[r][k] -= f * A[c][k];
            b[r] -= f * b[c];
        }
    }
    for (int r = 3; r >= 0; --r) {
        double s = b[r];
        for (int k = r + 1; k < 4; ++k) s -= A[r][k] * x[k];
        x[r] = s / A[r][r];
    }
}

__global__ void __launch_bounds__(32 * kC3Vals) k3_ca_solve(int pass, int nblocks, const double* __restrict__ part,
                                                           double* __restrict__ st, double sc0, double sc1, double sc2,
                                                           double R) {
    __shared__ double S[kC3Vals];  // one warp per sum
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double v = 0.0;
    for (int b = lane; b < nblocks; b += 32) v += part[b * kC3Vals + q];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) S[q] = v;
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (pass == 0) {
        st[0] = S[0];
        st[10] = S[0] < 8.0 ? 1.0 : 0.0;
        for (int d = 0; d < 3; ++d) st[1 + d] = S[0] > 0.0 ? S[1 + d] / S[0] : 0.0;
    } else if (pass == 1) {
        if (st[10] != 0.0) return;
        // [2q, 1] [c; d] = |q|^2 in the least-squares sense
        double A[4][4] = {{4 * S[0], 4 * S[1], 4 * S[2], 2 * S[6]},
                          {4 * S[1], 4 * S[3], 4 * S[4], 2 * S[7]},
                          {4 * S[2], 4 * S[4], 4 * S[5], 2 * S[8]},
                          {2 * S[6], 2 * S[7], 2 * S[8], st[0]}};
        double b[4] = {2 * S[9], 2 * S[10], 2 * S[11], S[12]};
        double x[4];
        solve4(A, b, x);
        st[7] = sqrt(x[3] + x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
        for (int d = 0; d < 3; ++d) st[4 + d] = st[1 + d] + x[d];
    } else if (pass == 2) {
        if (st[10] != 0.0) return;
        double A[4][4];
        int k = 0;
        for (int a = 0; a < 4; ++a)
            for (int b2 = a; b2 < 4; ++b2) {
                A[a][b2] = S[k];
                A[b2][a] = S[k];
                ++k;
            }
        double b[4] = {-S[10], -S[11], -S[12], -S[13]};
        double x[4];
        solve4(A, b, x);
        for (int d = 0; d < 3; ++d) st[4 + d] += x[d];
        st[7] += x[3];
    } else {
        if (st[10] != 0.0) return;
        st[8] = sqrt(S[0] / st[0]);
        const double d0 = st[4] - sc0, d1 = st[5] - sc1, d2 = st[6] - sc2, r = st[7];
        double cth = (R * R + r * r - (d0 * d0 + d1 * d1 + d2 * d2)) / (2.0 * r * R);
        cth = cth > 1.0 ? 1.0 : (cth < -1.0 ? -1.0 : cth);
        st[9] = acos(cth) * (180.0 / 3.14159265358979323846);
    }
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
struct lbm3d_ctx {
    int storage = LBM_STORE_F32;
    size_t elem = 4;               // bytes per stored population value
    size_t relem = 4;              // bytes per value of the compute type (densities)
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Geo3 g{};
    P3<float> pf{};
    P3<double> pd{};
    long long nfluid = 0;
    uint8_t* solid = nullptr;
    uint32_t* flags = nullptr;
    unsigned char* f[2] = {nullptr, nullptr};
    int cur = 0;
    unsigned char* rho = nullptr;  // [N] density pairs in the compute type
    int num_sms = 0;
    int zc = 0;                    // z planes per block of the march
    double* part = nullptr;        // per-block diagnostic records
    long long nparts = 0;
    double* dout = nullptr;        // [k3DiagN]
    double* ca = nullptr;          // contact angle: status record + block partials
    uint8_t* ca_cross = nullptr;   // contact angle: per-node crossing bits (N bytes, whole groups)
    int* ca_count = nullptr;       // crossings per kC3Seg nodes
    double* scratch = nullptr;     // [38][N] doubles for population transfers and fields (on demand)
    double* dens = nullptr;        // [2][N] doubles for lbm3d_set_densities from host arrays (on demand)
    // overlapped host transfers (lbm3d_set_densities_async, lbm3d_fields_async; on first use): copy
    // streams, double-buffered device staging and the events that order them with the stream
    cudaStream_t xs_in = nullptr, xs_out = nullptr;
    double* xin[2] = {nullptr, nullptr};   // [2][N] densities from the host
    double* xout[2] = {nullptr, nullptr};  // [5][N] fields for the host
    cudaEvent_t xin_ready[2] = {nullptr, nullptr}, xin_free[2] = {nullptr, nullptr};
    cudaEvent_t xout_ready[2] = {nullptr, nullptr}, xout_free[2] = {nullptr, nullptr};
    int xin_k = 0, xout_k = 0;
};

namespace {

bool fin(double v) { return isfinite(v) != 0; }

template <class R>
P3<R> make_p3(const lbm3d_params& p) {
    P3<R> P;
    for (int k = 0; k < 2; ++k) {
        P.omega[k] = (R)(1.0 / p.tau[k]);
        P.cF[k] = (R)(1.0 - 0.5 / p.tau[k]);
    }
    P.G = (R)p.G_AB;
    P.Gw2 = (R)p.G_w2;
    P.lam = (R)p.lambda;
    P.delta = (R)p.delta;
    const double l = p.lambda, dl = p.delta;
    P.s1 = (R)(2.0 * l / (1.0 + l));                          // Eq. 12 coefficients
    P.s2 = (R)(2.0 * (l * l - l) / (dl * (1.0 + l)));
    P.s3 = (R)((l - l * l) / (dl * dl * (1.0 + l)));
    P.t2 = (R)(2.0 * (l - 1.0) / (dl * (1.0 + l)));
    P.t3 = (R)((l - 1.0) / (dl * dl * (1.0 + l)));
    for (int d = 0; d < 3; ++d) P.g[d] = (R)p.g[d];
    for (int c = 0; c < 3; ++c)
        for (int k = 0; k < 2; ++k) P.sh[c][k] = (R)(w19(c == 0 ? 0 : (c == 1 ? 1 : 7)) * p.rho0_store[k]);
    P.mode = p.mode;
    P.psi = p.second_layer == LBM_SECOND_LAYER_PSI;
    P.adh = p.adhesion_stencil == LBM3_ADHESION_D3Q19;
    return P;
}

// Calls fn(S*, R*) (null pointers carrying the types) for the context's storage: the stored type S
// and the compute type R.
template <class Fn>
cudaError_t with_types3(int storage, Fn&& fn) {
    switch (storage) {
        case LBM_STORE_F64: return fn((double*)nullptr, (double*)nullptr);
        case LBM_STORE_F32: return fn((float*)nullptr, (float*)nullptr);
        case LBM_STORE_F16_SHIFTED: return fn((__half*)nullptr, (float*)nullptr);
        default: return fn((__nv_bfloat16*)nullptr, (float*)nullptr);
    }
}
#define TYPES3(s_, r_)                                   \
    using S = std::remove_pointer_t<decltype(s_)>;      \
    using R = std::remove_pointer_t<decltype(r_)>

// node kernels run blocks of 32 x 4 nodes (x, y), so that a block's stencil rows share L1
dim3 grid3(const Geo3& g) { return dim3((unsigned)((g.nx + 31) / 32), (unsigned)((g.ny + 3) / 4), (unsigned)g.nz); }
const dim3 kBlock3(32, 4, 1);

// z planes per block of the march.  A block costs its planes plus about 2 (the first density planes, the
// start), and a launch runs its blocks in rounds of `resident`; about 16 planes, spread evenly over
// nz, once there are many rounds (32 measured the same).  With 16 planes for every lattice a small
// one ran as a few blocks: 40 x 40 x 56, 80 blocks, 39 us a step; with this rule 17.
#ifndef LBM3_ZCHUNK
#define LBM3_ZCHUNK 16
#endif
int zchunk3(const Geo3& g, int resident) {
    const long long tiles = (long long)((g.nx + k3TX - 1) / k3TX) * ((g.ny + k3TY - 1) / k3TY);
    double best = -1.0;
    int zc = LBM3_ZCHUNK;
    for (int n = (g.nz + LBM3_ZCHUNK - 1) / LBM3_ZCHUNK; n <= g.nz; ++n) {
        const int h = (g.nz + n - 1) / n;
        const long long blocks = tiles * ((g.nz + h - 1) / h);
        const double rounds = blocks > 3LL * resident ? (double)blocks / resident + 0.5
                                                      : (double)((blocks + resident - 1) / resident);
        const double cost = rounds * (h + 2);
        if (best < 0 || cost < best) {
            best = cost;
            zc = h;
        }
    }
    return zc;
}

cudaError_t scratch_for(lbm3d_ctx* c) {
    if (c->scratch) return cudaSuccess;
    return cudaMalloc(&c->scratch, (size_t)38 * c->g.N * sizeof(double));
}

// the context's parameters in the compute type R
template <class R>
const P3<R>& p3_of(const lbm3d_ctx* c) {
    return *reinterpret_cast<const P3<R>*>(sizeof(R) == 4 ? (const void*)&c->pf : (const void*)&c->pd);
}
template <class S>
Pair<S>* state3(const lbm3d_ctx* c, int buf) {
    return reinterpret_cast<Pair<S>*>(c->f[buf]);
}

// the march kernel instance of the adhesion variant
template <class S, class R, int kMode = kStep>
auto march_kernel(const P3<R>& P) {
    return P.adh ? k3_march<S, R, kAdhD3Q19, kMode>
                 : (P.psi ? k3_march<S, R, kAdhE8Psi, kMode> : k3_march<S, R, kAdhE8, kMode>);
}

dim3 march_grid(const Geo3& g, int zc) {
    return dim3((unsigned)((g.nx + k3TX - 1) / k3TX), (unsigned)((g.ny + k3TY - 1) / k3TY), (unsigned)((g.nz + zc - 1) / zc));
}

// densities of the current state into c->rho
template <class S, class R>
cudaError_t launch_rho3(lbm3d_ctx* c) {
    const PdlLaunch l(grid3(c->g), kBlock3, 0, c->stream);
    return l.launch(k3_rho<S, R>, c->g, p3_of<R>(c), (const uint32_t*)c->flags, (const Pair<S>*)state3<S>(c, c->cur),
                    reinterpret_cast<typename Rho2<R>::T*>(c->rho));
}

// the march over the whole lattice; the density pass comes first
template <class S, class R, int kMode>
cudaError_t launch_march3(lbm3d_ctx* c, const Out5& o5) {
    const P3<R>& P = p3_of<R>(c);
    const PdlLaunch l(march_grid(c->g, c->zc), kBlock3, k3_march_smem<R>(), c->stream);
    auto* kern = march_kernel<S, R, kMode>(P);
    if (k3_march_smem<R>() > 48 * 1024) {  // above the default limit (FP64)
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k3_march_smem<R>());
        if (e != cudaSuccess) return e;
    }
    return l.launch(kern, c->g, P, c->zc, (const uint32_t*)c->flags, (const Pair<S>*)state3<S>(c, c->cur),
                    (const V2<R>*)c->rho, state3<S>(c, 1 - c->cur), o5, c->part);
}

template <class S, class R>
cudaError_t step_once(lbm3d_ctx* c) {
    cudaError_t e = launch_rho3<S, R>(c);
    if (e == cudaSuccess) e = launch_march3<S, R, kStep>(c, Out5{});
    if (e == cudaSuccess) c->cur ^= 1;
    return e;
}

// densities of the current state into c->rho, then a fields form of the march (outputs may be NULL):
// the same pull, stencil sums, moments and forces as a step; diag: per-block diagnostic records,
// combined into c->dout
cudaError_t run_fields(lbm3d_ctx* c, const Out5& o5, bool diag) {
    return with_types3(c->storage, [&](auto* s_, auto* r_) {
        TYPES3(s_, r_);
        cudaError_t e = launch_rho3<S, R>(c);
        if (e == cudaSuccess) e = diag ? launch_march3<S, R, kFieldsDiag>(c, o5) : launch_march3<S, R, kFieldsOnly>(c, o5);
        if (e != cudaSuccess || !diag) return e;
        const dim3 gm = march_grid(c->g, c->zc);
        const long long nb = (long long)gm.x * gm.y * gm.z;  // <= c->nparts (one record per block)
        double* mid = c->part + c->nparts * k3DiagN;         // k3DiagMid records after the per-block ones
        k3_diag_mid<<<k3DiagMid, k3DiagMidThreads, 0, c->stream>>>(nb, c->part, mid);
        k3_diag_final<<<1, 32 * k3DiagN, 0, c->stream>>>(k3DiagMid, mid, c->dout);
        return cudaGetLastError();
    });
}

cudaError_t density_pass(lbm3d_ctx* c) {
    return with_types3(c->storage, [&](auto* s_, auto* r_) {
        TYPES3(s_, r_);
        return launch_rho3<S, R>(c);
    });
}

// the state from post-streaming populations (FP64 [38][N] on the device) / from densities
cudaError_t set_state3(lbm3d_ctx* c, const double* f, int buf) {
    return with_types3(c->storage, [&](auto* s_, auto* r_) {
        TYPES3(s_, r_);
        k3_set<S, R><<<grid3(c->g), kBlock3, 0, c->stream>>>(c->g, p3_of<R>(c), c->flags, f, state3<S>(c, buf));
        return cudaGetLastError();
    });
}
cudaError_t set_rest3(lbm3d_ctx* c, const double* a, const double* b) {
    return with_types3(c->storage, [&](auto* s_, auto* r_) {
        TYPES3(s_, r_);
        const long long tiles = (long long)((c->g.nx + kR3X - 1) / kR3X) * ((c->g.ny + kR3Y - 1) / kR3Y);
        int planes = kR3Z;  // three blocks on every SM, if there are planes enough (128^3: 77 us, eight planes 80)
        while (planes > 1 && tiles * ((c->g.nz + planes - 1) / planes) < 3LL * c->num_sms) planes /= 2;
        const dim3 gr((unsigned)((c->g.nx + kR3X - 1) / kR3X), (unsigned)((c->g.ny + kR3Y - 1) / kR3Y),
                      (unsigned)((c->g.nz + planes - 1) / planes));
        k3_set_rest<S, R><<<gr, dim3(kR3X, kR3Y), 0, c->stream>>>(c->g, p3_of<R>(c), planes, c->flags, a, b, state3<S>(c, c->cur));
        return cudaGetLastError();
    });
}

template <class R>
cudaError_t ca_passes(lbm3d_ctx* c, const double* sc, double R_) {
    const int ngroup = (int)((c->g.N + kC3Group - 1) / kC3Group);
    Ca3<R> ca{c->g, c->flags, reinterpret_cast<const typename Rho2<R>::T*>(c->rho), c->ca_cross, c->ca_count};
    double* st = c->ca;
    double* part = c->ca + 16;
    cudaError_t e = cudaMemsetAsync(st, 0, 16 * sizeof(double), c->stream);
    if (e != cudaSuccess) return e;
    k3_ca_cross<R><<<ngroup * (kC3Group / kC3Seg), kC3Threads, 0, c->stream>>>(ca);
    for (int pass = 0; pass < 4; ++pass) {
        auto* kern = pass == 0 ? k3_ca_pass<R, 0> : pass == 1 ? k3_ca_pass<R, 1> : pass == 2 ? k3_ca_pass<R, 2> : k3_ca_pass<R, 3>;
        kern<<<kC3Blocks, kC3Threads, 0, c->stream>>>(ca, ngroup, st, part);
        k3_ca_solve<<<1, 32 * kC3Vals, 0, c->stream>>>(pass, kC3Blocks, part, st, sc[0], sc[1], sc[2], R_);
    }
    return cudaGetLastError();
}

void free_xfer3(lbm3d_ctx* c) {
    for (cudaStream_t* st : {&c->xs_in, &c->xs_out})
        if (*st) {
            cudaStreamSynchronize(*st);
            cudaStreamDestroy(*st);
            *st = nullptr;
        }
    for (int k = 0; k < 2; ++k) {
        for (cudaEvent_t* ev : {&c->xin_ready[k], &c->xin_free[k], &c->xout_ready[k], &c->xout_free[k]})
            if (*ev) cudaEventDestroy(*ev), *ev = nullptr;
        if (c->xin[k]) cudaFree(c->xin[k]), c->xin[k] = nullptr;
        if (c->xout[k]) cudaFree(c->xout[k]), c->xout[k] = nullptr;
    }
}

void free3(lbm3d_ctx* c) {
    free_xfer3(c);
    void* ptrs[] = {c->solid, c->flags, c->f[0], c->f[1], c->rho, c->part, c->dout, c->ca, c->ca_cross, c->ca_count, c->scratch, c->dens};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

}  // namespace

#define TRY3(call, what)                                                                                 \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) {                                                                         \
            lbm_status s_ = e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;                    \
            if (e_ == cudaErrorMemoryAllocation) cudaGetLastError();                                     \
            return report_error(s_, "%s: %s", what, cudaGetErrorString(e_));                              \
        }                                                                                                \
    } while (0)

extern "C" lbm_status lbm3d_create(const lbm3d_grid* grid, const uint8_t* solid, const lbm3d_params* p,
                                   const double* rA0, const double* rB0, int32_t storage, void* cuda_stream,
                                   lbm3d_ctx** out) {
    if (!out) return report_error(LBM_EINVAL, "NULL output pointer");
    *out = nullptr;
    if (!grid || !solid || !p || !rA0 || !rB0) return report_error(LBM_EINVAL, "NULL argument");
    if (grid->nx < 5 || grid->ny < 5 || grid->nz < 5) return report_error(LBM_EINVAL, "nx, ny, nz must be >= 5");
    if (grid->ny > 65535 || grid->nz > 65535) return report_error(LBM_EINVAL, "ny, nz must be <= 65535");
    if ((long long)grid->nx * grid->ny * grid->nz > (1LL << 31) - 1) return report_error(LBM_EINVAL, "lattice too large (2^31 nodes)");
    if (storage < LBM_STORE_F64 || storage > LBM_STORE_BF16_SHIFTED) return report_error(LBM_EINVAL, "bad storage %d", storage);
    for (int k = 0; k < 2; ++k)
        if (!fin(p->tau[k]) || p->tau[k] <= 0.5) return report_error(LBM_EINVAL, "tau[%d] must be > 0.5", k);
    if (!fin(p->G_AB) || !fin(p->G_w2) || !fin(p->g[0]) || !fin(p->g[1]) || !fin(p->g[2]) || !fin(p->rho0_store[0]) ||
        !fin(p->rho0_store[1]))
        return report_error(LBM_EINVAL, "non-finite parameter");
    if (!fin(p->lambda) || p->lambda <= 0.0) return report_error(LBM_EINVAL, "lambda must be > 0");
    if (!fin(p->delta) || p->delta <= 0.0 || p->delta > 1.0) return report_error(LBM_EINVAL, "delta must lie in (0, 1]");
    if (p->mode != LBM_ADS_ORIGINAL && p->mode != LBM_ADS_IMPROVED) return report_error(LBM_EINVAL, "bad mode");
    if (p->second_layer != LBM_SECOND_LAYER_PSI_AND_SOLID && p->second_layer != LBM_SECOND_LAYER_PSI)
        return report_error(LBM_EINVAL, "bad second_layer");
    if (p->adhesion_stencil != LBM3_ADHESION_E8 && p->adhesion_stencil != LBM3_ADHESION_D3Q19)
        return report_error(LBM_EINVAL, "bad adhesion_stencil");
    const long long N = (long long)grid->nx * grid->ny * grid->nz;
    long long nf = 0;
    for (long long s = 0; s < N; ++s) {
        if (solid[s]) continue;
        ++nf;
        if (!fin(rA0[s]) || !fin(rB0[s]) || rA0[s] <= 0.0 || rB0[s] <= 0.0)
            return report_error(LBM_EINVAL, "initial densities must be finite and > 0 at fluid node %lld", s);
    }
    if (nf == 0) return report_error(LBM_EINVAL, "the mask has no fluid node");
    int dev = 0;
    cudaDeviceProp prop;
    TRY3(cudaGetDevice(&dev), "cudaGetDevice");
    TRY3(cudaGetDeviceProperties(&prop, dev), "cudaGetDeviceProperties");
    if (!(prop.major == 10 && prop.minor == 3))
        return report_error(LBM_ECUDA, "this library is built for sm_103a (GB300); device %d is sm_%d%d", dev, prop.major, prop.minor);

    lbm3d_ctx* c = new (std::nothrow) lbm3d_ctx();
    if (!c) return report_error(LBM_ENOMEM, "host allocation");
    auto bail = [&](lbm_status s) {
        free3(c);
        delete c;
        return s;
    };
#define STEP3(call, what)                                                                            \
    do {                                                                                             \
        cudaError_t e_ = (call);                                                                     \
        if (e_ != cudaSuccess) {                                                                     \
            lbm_status s_ = e_ == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;                \
            if (e_ == cudaErrorMemoryAllocation) cudaGetLastError();                                 \
            report_error(s_, "%s: %s", what, cudaGetErrorString(e_));                                 \
            return bail(s_);                                                                         \
        }                                                                                            \
    } while (0)
    c->storage = storage;
    c->elem = storage == LBM_STORE_F64 ? 8 : (storage == LBM_STORE_F32 ? 4 : 2);  // bytes per stored value
    c->relem = storage == LBM_STORE_F64 ? 8 : 4;                                  // bytes per computed value
    c->g = Geo3{grid->nx, grid->ny, grid->nz, N};
    c->pf = make_p3<float>(*p);
    c->pd = make_p3<double>(*p);
    c->nfluid = nf;
    if (cuda_stream) {
        c->stream = (cudaStream_t)cuda_stream;
    } else {
        STEP3(cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking), "stream");
        c->own_stream = true;
    }
    const dim3 gr = grid3(c->g);
    c->nparts = (long long)gr.x * gr.y * gr.z;
    c->num_sms = prop.multiProcessorCount;
    c->zc = zchunk3(c->g, (storage == LBM_STORE_F64 ? 2 : storage == LBM_STORE_F32 ? march_blocks<float>() : march_blocks<__half>()) *
                               c->num_sms);
    STEP3(cudaMalloc(&c->solid, N), "mask");
    STEP3(cudaMalloc(&c->flags, N * sizeof(uint32_t)), "flags");
    STEP3(cudaMalloc(&c->f[0], 38 * N * c->elem), "population buffer");
    STEP3(cudaMalloc(&c->f[1], 38 * N * c->elem), "population buffer");
    STEP3(cudaMalloc(&c->rho, 2 * N * c->relem), "densities");
    STEP3(cudaMalloc(&c->part, (c->nparts + k3DiagMid) * k3DiagN * sizeof(double)), "diagnostics");
    STEP3(cudaMalloc(&c->dout, k3DiagN * sizeof(double)), "diagnostics");
    STEP3(cudaMalloc(&c->ca, (16 + kC3Blocks * kC3Vals) * sizeof(double)), "contact-angle scratch");
    const size_t ngroup = ((size_t)N + kC3Group - 1) / kC3Group;
    STEP3(cudaMalloc(&c->ca_cross, ngroup * kC3Group), "contact-angle scratch");
    STEP3(cudaMalloc(&c->ca_count, ngroup * (kC3Group / kC3Seg) * sizeof(int)), "contact-angle scratch");
    STEP3(cudaMemsetAsync(c->f[0], 0, 38 * N * c->elem, c->stream), "memset");
    STEP3(cudaMemsetAsync(c->f[1], 0, 38 * N * c->elem, c->stream), "memset");
    STEP3(cudaMemcpy(c->solid, solid, N, cudaMemcpyHostToDevice), "mask upload");
    k3_flags<<<gr, kBlock3, 0, c->stream>>>(c->g, c->solid, c->flags);
    STEP3(cudaGetLastError(), "flags kernel");
    STEP3(cudaMalloc(&c->dens, (size_t)2 * N * sizeof(double)), "density buffer");
    STEP3(cudaMemcpyAsync(c->dens, rA0, N * sizeof(double), cudaMemcpyHostToDevice, c->stream), "density upload");
    STEP3(cudaMemcpyAsync(c->dens + N, rB0, N * sizeof(double), cudaMemcpyHostToDevice, c->stream), "density upload");
    STEP3(set_rest3(c, c->dens, c->dens + N), "init kernel");
    STEP3(cudaStreamSynchronize(c->stream), "initialisation");
    cudaFree(c->dens);  // lbm3d_set_densities from host arrays allocates it again on demand
    c->dens = nullptr;
#undef STEP3
    *out = c;
    return LBM_OK;
}

extern "C" void lbm3d_destroy(lbm3d_ctx* c) {
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    free3(c);
    delete c;
}

extern "C" lbm_status lbm3d_step(lbm3d_ctx* c, int64_t n) {
    NvtxRange nvtx_("lbm3d_step");
    if (!c) return report_error(LBM_EINVAL, "NULL context");
    if (n < 0) return report_error(LBM_EINVAL, "n must be >= 0");
    TRY3(with_types3(c->storage,
                     [&](auto* s_, auto* r_) {
                         TYPES3(s_, r_);
                         cudaError_t e = cudaSuccess;
                         for (int64_t t = 0; t < n && e == cudaSuccess; ++t) e = step_once<S, R>(c);
                         return e;
                     }),
         "step kernels");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_fields(lbm3d_ctx* c, double* rA, double* rB, double* ux, double* uy, double* uz,
                                   int32_t on_device) {
    NvtxRange nvtx_("lbm3d_fields");
    if (!c) return report_error(LBM_EINVAL, "NULL context");
    Out5 outs{{rA, rB, ux, uy, uz}};
    if (on_device) {
        TRY3(run_fields(c, outs, false), "fields kernels");
        return LBM_OK;
    }
    TRY3(scratch_for(c), "fields scratch");
    const long long N = c->g.N;
    Out5 dev;
    for (int q = 0; q < 5; ++q) dev.p[q] = outs.p[q] ? c->scratch + q * N : nullptr;
    TRY3(run_fields(c, dev, false), "fields kernels");
    for (int q = 0; q < 5; ++q)
        if (outs.p[q])
            TRY3(cudaMemcpyAsync(outs.p[q], dev.p[q], N * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "fields copy");
    TRY3(cudaStreamSynchronize(c->stream), "fields");
    return LBM_OK;
}

namespace {
// copy streams, staging and events of the overlapped transfers
lbm_status xfer3_setup(lbm3d_ctx* c) {
    if (c->xs_in) return LBM_OK;
    const size_t N = (size_t)c->g.N;
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
        e = cudaMalloc(&c->xin[k], 2 * N * sizeof(double));
        if (e == cudaSuccess) e = cudaMalloc(&c->xout[k], 5 * N * sizeof(double));
        for (cudaEvent_t* ev : {&c->xin_ready[k], &c->xin_free[k], &c->xout_ready[k], &c->xout_free[k]})
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->xs_out, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->xs_in, cudaStreamNonBlocking);  // set last: marks done
    if (e != cudaSuccess) {
        const bool oom = e == cudaErrorMemoryAllocation;
        cudaGetLastError();
        free_xfer3(c);
        return report_error(oom ? LBM_ENOMEM : LBM_ECUDA, "overlapped transfers: %s", cudaGetErrorString(e));
    }
    return LBM_OK;
}
}  // namespace

extern "C" lbm_status lbm3d_set_densities_async(lbm3d_ctx* c, const double* rho_A, const double* rho_B) {
    NvtxRange nvtx_("lbm3d_set_densities_async");
    if (!c || !rho_A || !rho_B) return report_error(LBM_EINVAL, "NULL argument");
    const lbm_status s = xfer3_setup(c);
    if (s != LBM_OK) return s;
    const long long N = c->g.N;
    const int k = c->xin_k;
    c->xin_k ^= 1;
    double* a = c->xin[k];
    double* b = c->xin[k] + N;
    // the copy may start once the kernel that read this staging buffer two calls ago has run
    TRY3(cudaStreamWaitEvent(c->xs_in, c->xin_free[k], 0), "transfer order");
    TRY3(cudaMemcpyAsync(a, rho_A, N * sizeof(double), cudaMemcpyHostToDevice, c->xs_in), "upload");
    TRY3(cudaMemcpyAsync(b, rho_B, N * sizeof(double), cudaMemcpyHostToDevice, c->xs_in), "upload");
    TRY3(cudaEventRecord(c->xin_ready[k], c->xs_in), "transfer order");
    TRY3(cudaStreamWaitEvent(c->stream, c->xin_ready[k], 0), "transfer order");
    TRY3(set_rest3(c, a, b), "state kernel");
    TRY3(cudaGetLastError(), "state kernel");
    TRY3(cudaEventRecord(c->xin_free[k], c->stream), "transfer order");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_fields_async(lbm3d_ctx* c, double* rho_A, double* rho_B, double* ux, double* uy,
                                         double* uz) {
    NvtxRange nvtx_("lbm3d_fields_async");
    if (!c) return report_error(LBM_EINVAL, "NULL context");
    const lbm_status s = xfer3_setup(c);
    if (s != LBM_OK) return s;
    const long long N = c->g.N;
    const int k = c->xout_k;
    c->xout_k ^= 1;
    // the fields pass may overwrite this staging buffer once its previous copy to the host is done;
    // the copies then run on their own stream, beside the context's next work
    TRY3(cudaStreamWaitEvent(c->stream, c->xout_free[k], 0), "transfer order");
    double* outs[5] = {rho_A, rho_B, ux, uy, uz};
    Out5 dev;
    for (int q = 0; q < 5; ++q) dev.p[q] = outs[q] ? c->xout[k] + q * N : nullptr;
    TRY3(run_fields(c, dev, false), "fields kernels");
    TRY3(cudaEventRecord(c->xout_ready[k], c->stream), "transfer order");
    TRY3(cudaStreamWaitEvent(c->xs_out, c->xout_ready[k], 0), "transfer order");
    for (int q = 0; q < 5; ++q)
        if (outs[q])
            TRY3(cudaMemcpyAsync(outs[q], c->xout[k] + q * N, N * sizeof(double), cudaMemcpyDeviceToHost, c->xs_out),
                 "fields copy");
    TRY3(cudaEventRecord(c->xout_free[k], c->xs_out), "transfer order");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_synchronize(lbm3d_ctx* c) {
    if (!c) return report_error(LBM_EINVAL, "NULL context");
    for (cudaStream_t st : {c->xs_in, c->xs_out, c->stream})
        if (st) TRY3(cudaStreamSynchronize(st), "synchronize");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_get_populations(lbm3d_ctx* c, double* f) {
    if (!c || !f) return report_error(LBM_EINVAL, "NULL argument");
    TRY3(scratch_for(c), "transfer scratch");
    TRY3(with_types3(c->storage,
                     [&](auto* s_, auto* r_) {
                         TYPES3(s_, r_);
                         k3_get<S, R><<<grid3(c->g), kBlock3, 0, c->stream>>>(c->g, p3_of<R>(c), c->flags,
                                                                            state3<S>(c, c->cur), c->scratch);
                         return cudaGetLastError();
                     }),
         "read-back kernel");
    TRY3(cudaGetLastError(), "read-back kernel");
    TRY3(cudaMemcpyAsync(f, c->scratch, (size_t)38 * c->g.N * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "read-back");
    TRY3(cudaStreamSynchronize(c->stream), "read-back");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_set_densities(lbm3d_ctx* c, const double* rho_A, const double* rho_B, int32_t on_device) {
    if (!c || !rho_A || !rho_B) return report_error(LBM_EINVAL, "NULL argument");
    const long long N = c->g.N;
    const double *a = rho_A, *b = rho_B;
    if (!on_device) {
        if (!c->dens) TRY3(cudaMalloc(&c->dens, (size_t)2 * N * sizeof(double)), "density buffer");
        TRY3(cudaMemcpyAsync(c->dens, rho_A, N * sizeof(double), cudaMemcpyHostToDevice, c->stream), "upload");
        TRY3(cudaMemcpyAsync(c->dens + N, rho_B, N * sizeof(double), cudaMemcpyHostToDevice, c->stream), "upload");
        a = c->dens;
        b = c->dens + N;
    }
    TRY3(set_rest3(c, a, b), "state kernel");
    TRY3(cudaGetLastError(), "state kernel");
    if (!on_device) TRY3(cudaStreamSynchronize(c->stream), "upload");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_set_populations(lbm3d_ctx* c, const double* f) {
    if (!c || !f) return report_error(LBM_EINVAL, "NULL argument");
    TRY3(scratch_for(c), "transfer scratch");
    TRY3(cudaMemcpyAsync(c->scratch, f, (size_t)38 * c->g.N * sizeof(double), cudaMemcpyHostToDevice, c->stream), "upload");
    TRY3(set_state3(c, c->scratch, c->cur), "state kernel");
    TRY3(cudaGetLastError(), "state kernel");
    TRY3(cudaStreamSynchronize(c->stream), "upload");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_diagnostics(lbm3d_ctx* c, lbm3d_diag* out) {
    if (!c || !out) return report_error(LBM_EINVAL, "NULL argument");
    TRY3(run_fields(c, Out5{}, true), "diagnostics kernels");
    double v[k3DiagN];
    TRY3(cudaMemcpyAsync(v, c->dout, sizeof v, cudaMemcpyDeviceToHost, c->stream), "diagnostics read-back");
    TRY3(cudaStreamSynchronize(c->stream), "diagnostics");
    out->mass_A = v[0];
    out->mass_B = v[1];
    out->mom_x = v[2];
    out->mom_y = v[3];
    out->mom_z = v[4];
    out->umax = v[5];
    out->rhoA_min = v[6];
    out->rhoA_max = v[7];
    out->rhoB_min = v[8];
    out->rhoB_max = v[9];
    out->n_fluid = (int64_t)llround(v[10]);
    out->unstable = v[11] != 0.0;
    out->pad_ = 0;
    if (out->unstable) return report_error(LBM_EUNSTABLE, "non-finite or non-positive density");
    return LBM_OK;
}

extern "C" lbm_status lbm3d_contact_angle(lbm3d_ctx* c, const double* sc, double R, double* theta_deg, double* fit_rms,
                                          int64_t* npoints) {
    if (!c || !sc) return report_error(LBM_EINVAL, "NULL argument");
    if (!(R > 0.0) || !fin(sc[0]) || !fin(sc[1]) || !fin(sc[2])) return report_error(LBM_EINVAL, "bad sphere");
    cudaError_t e = density_pass(c);
    TRY3(e, "density kernel");
    e = c->storage == LBM_STORE_F64 ? ca_passes<double>(c, sc, R) : ca_passes<float>(c, sc, R);
    TRY3(e, "contact-angle kernels");
    double h[16];
    TRY3(cudaMemcpyAsync(h, c->ca, sizeof h, cudaMemcpyDeviceToHost, c->stream), "contact-angle read-back");
    TRY3(cudaStreamSynchronize(c->stream), "contact angle");
    if (npoints) *npoints = (int64_t)llround(h[0]);
    if (h[10] != 0.0) return report_error(LBM_ESTATE, "only %.0f interface points", h[0]);
    if (theta_deg) *theta_deg = h[9];
    if (fit_rms) *fit_rms = h[8];
    return LBM_OK;
}
