// Geometry preprocessing on the device: node flags (solid, blocked links for halfway bounce-back,
// wall-list membership) and the wall list with the second-layer reconstruction of Sec. 2.4.
//
// Wall list: the fluid nodes whose 24-node eighth-order stencil reaches a site that is not an
// in-array fluid node (solid, or outside the array along a non-periodic axis), in increasing node
// order y*nx + x.  For each entry:
//   subst  bit n-1 set when second-layer stencil node n (Table 1 numbering) is not a fluid node and
//          therefore takes the information of its first-layer partner x + sign(e_n)
//   seff   bit n-1 set when stencil node n counts as solid in the adhesion sum (Eq. 9): a solid or
//          outside first-layer site, or a replaced second-layer node whose partner is one (when it
//          copies the pseudopotential only: whose own site is one, clamped along an open axis)
//   a      sum_n w(|e_n|^2) seff_n e_n  (FP64)
// With the adhesion sum of Eq. 9 as printed (LBM_ADHESION_D2Q9) only the first layer enters it:
// seff keeps the first-layer bits and a = sum_i w_i s(x + e_i) e_i with the D2Q9 weights, opposite
// velocities taken together (i = 1, 2, 5, 6 with opp(i)).
// Along an open axis a first-layer site beyond the boundary column is the boundary column itself.
#include "lbm_internal.h"

namespace lbm {

namespace {

struct Geo {
    int nx, ny, bc_x, bc_y;
    const uint8_t* solid;  // dense [ny][nx]
};

// Is (X, Y) a fluid node after the periodic wrap?  Outside a non-periodic axis: no.
__device__ __forceinline__ bool fluid_at(const Geo& g, int X, int Y) {
    if (X < 0 || X >= g.nx) {
        if (g.bc_x != kPeriodic) return false;
        X = ((X % g.nx) + g.nx) % g.nx;
    }
    if (Y < 0 || Y >= g.ny) {
        if (g.bc_y != kPeriodic) return false;
        Y = ((Y % g.ny) + g.ny) % g.ny;
    }
    return g.solid[(long long)Y * g.nx + X] == 0;
}

// Solid switch of a first-layer site (dx, dy in {-1, 0, 1}).
__device__ __forceinline__ bool first_layer_solid(const Geo& g, int X, int Y, int dx, int dy) {
    int Xs = X + dx;
    if (g.bc_x == kOpen) Xs = Xs < 0 ? 0 : (Xs > g.nx - 1 ? g.nx - 1 : Xs);
    return !fluid_at(g, Xs, Y + dy);
}

__global__ void k_flags(const DevCase* __restrict__ cases, int c, const uint8_t* __restrict__ solid_all,
                        uint16_t* __restrict__ flags_all, int32_t* __restrict__ row_counts) {
    const DevCase C = cases[c];
    const Geo g{C.nx, C.ny, C.bc_x, C.bc_y, solid_all + C.d_off};
    const long long N = (long long)C.nx * C.ny;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
        const int X = (int)(s % C.nx), Y = (int)(s / C.nx);
        const long long o = C.d_off + s;
        if (g.solid[s]) {
            flags_all[o] = kSolidBit;
            continue;
        }
        uint16_t fl = 0;
        for (int i = 1; i < 9; ++i) {
            const int sx = X - cx(i), sy = Y - cy(i);
            bool blocked;
            if (C.bc_x == kOpen && (sx < 0 || sx >= C.nx)) blocked = false;  // enters through the open boundary
            else blocked = !fluid_at(g, sx, sy);
            if (blocked) fl |= (uint16_t)(1u << (i - 1));
        }
        if (C.bc_x == kOpen && X == C.nx - 1) {
            // outflow: entering populations are those of the node one column upstream
            const bool base_fluid = fluid_at(g, X - 1, Y);
            if (!base_fluid) fl |= kOutletOwnBit;
            for (int i = 1; i < 9; ++i) {
                if (cx(i) >= 0) continue;
                const bool blocked = !base_fluid || !fluid_at(g, X, Y - cy(i));
                fl = blocked ? (uint16_t)(fl | (1u << (i - 1))) : (uint16_t)(fl & ~(1u << (i - 1)));
            }
        }
        bool near = false;
        for (int dy = -3; dy <= 3 && !near; ++dy)
            for (int dx = -3; dx <= 3 && !near; ++dx) near = !fluid_at(g, X + dx, Y + dy);
        if (near) fl |= kNearSolidBit;
        bool touches = false;
        for (int n = 0; n < 24 && !touches; ++n) touches = !fluid_at(g, X + s24x(n), Y + s24y(n));
        if (touches) {
            fl |= kWallBit;
            atomicAdd(row_counts + Y, 1);
        }
        flags_all[o] = fl;
    }
}

// Exclusive scan of n counts by one block; offsets[n] receives the total.
__global__ void k_scan(const int32_t* __restrict__ counts, int32_t* __restrict__ offsets, int n) {
    __shared__ int32_t warp_sums[32];
    __shared__ int32_t carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += blockDim.x) {
        const int i = base + tid;
        const int v = i < n ? counts[i] : 0;
        int incl = v;
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += t;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int nw = blockDim.x >> 5;
            int ws = lane < nw ? warp_sums[lane] : 0;
            for (int off = 1; off < 32; off <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, ws, off);
                if (lane >= off) ws += t;
            }
            if (lane < nw) warp_sums[lane] = ws;  // inclusive warp prefix
        }
        __syncthreads();
        const int before = carry + (warp > 0 ? warp_sums[warp - 1] : 0);
        if (i < n) offsets[i] = before + incl - v;
        __syncthreads();
        if (tid == blockDim.x - 1) carry = before + incl;
        __syncthreads();
    }
    if (tid == 0) offsets[n] = carry;
}

// One block per row: wall nodes of the row in increasing x get consecutive entries.
__global__ void k_wall_fill(const DevCase* __restrict__ cases, int c, const uint8_t* __restrict__ solid_all,
                            const uint16_t* __restrict__ flags_all, uint32_t* __restrict__ wsub_all,
                            const int32_t* __restrict__ row_off, int32_t* __restrict__ wl_node,
                            uint32_t* __restrict__ wl_subst, uint32_t* __restrict__ wl_seff,
                            double* __restrict__ wl_a, long long nwall_total, int psi_only, int d2q9) {
    const DevCase C = cases[c];
    const Geo g{C.nx, C.ny, C.bc_x, C.bc_y, solid_all + C.d_off};
    const int Y = blockIdx.x;
    __shared__ int32_t warp_cnt[32];
    __shared__ int32_t running;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) running = 0;
    __syncthreads();
    for (int base = 0; base < C.nx; base += blockDim.x) {
        const int X = base + tid;
        bool is_wall = false;
        if (X < C.nx) is_wall = (flags_all[C.d_off + (long long)Y * C.nx + X] & kWallBit) != 0;
        const unsigned bal = __ballot_sync(0xffffffffu, is_wall);
        if (lane == 0) warp_cnt[warp] = __popc(bal);
        __syncthreads();
        int before = running;
        for (int w = 0; w < warp; ++w) before += warp_cnt[w];
        before += __popc(bal & ((1u << lane) - 1u));
        if (is_wall) {
            const long long e = C.w_off + row_off[Y] + before;
            uint32_t sm = 0, em = 0;
            for (int n = 0; n < 24; ++n) {
                const int ex = s24x(n), ey = s24y(n);
                bool s;
                if (ex >= -1 && ex <= 1 && ey >= -1 && ey <= 1) {
                    s = first_layer_solid(g, X, Y, ex, ey);
                } else if (fluid_at(g, X + ex, Y + ey)) {
                    s = false;
                } else {
                    sm |= 1u << n;
                    // psi only: the site keeps its own solid switch (clamped along an open axis)
                    s = psi_only ? first_layer_solid(g, X, Y, ex, ey)
                                 : first_layer_solid(g, X, Y, (ex > 0) - (ex < 0), (ey > 0) - (ey < 0));
                }
                if (s && (!d2q9 || n < 8)) em |= 1u << n;
            }
            double ax = 0.0, ay = 0.0;
            if (d2q9) {
                for (int h = 0; h < 4; ++h) {  // i = 1, 2, 5, 6 and opp(i); bit i-1 is first-layer node i
                    const int i = h < 2 ? 1 + h : 3 + h;
                    const double ds = (double)((em >> (i - 1)) & 1u) - (double)((em >> (opp(i) - 1)) & 1u);
                    ax += wq(i) * ds * cx(i);
                    ay += wq(i) * ds * cy(i);
                }
            } else {
                for (int p = 0; p < 12; ++p) {  // pairs (n, n+2): e_(n+2) = -e_n within each group of four
                    const int n = (p / 2) * 4 + (p % 2), m = n + 2;
                    const int ex = s24x(n), ey = s24y(n);
                    const double w = w8(ex * ex + ey * ey);
                    const double ds = (double)((em >> n) & 1u) - (double)((em >> m) & 1u);
                    ax += w * ds * ex;
                    ay += w * ds * ey;
                }
            }
            wl_node[e] = Y * C.nx + X;
            wl_subst[e] = sm;
            wl_seff[e] = em;
            wl_a[e] = ax;
            wl_a[nwall_total + e] = ay;
            wsub_all[C.d_off + (long long)Y * C.nx + X] = sm;
        }
        __syncthreads();
        if (tid == 0) {
            int tot = 0;
            for (int w = 0; w < nw; ++w) tot += warp_cnt[w];
            running += tot;
        }
        __syncthreads();
    }
}

// Flags with 8 ghost columns on each side, as the step kernel's tensor loads read them: column x
// at element x + 8; beyond the array a periodic axis wraps, a wall is solid and an open boundary
// repeats its boundary column.
__global__ void k_flags_ghost(const DevCase* __restrict__ cases, int c, const uint16_t* __restrict__ flags_all,
                              uint16_t* __restrict__ out, int pitch) {
    const DevCase C = cases[c];
    const long long n = (long long)C.ny * pitch;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const int Y = (int)(s / pitch), m = (int)(s % pitch), x = m - 8;
        uint16_t v;
        if (m >= C.nx + 16) v = 0;  // row padding
        else if (x >= 0 && x < C.nx) v = flags_all[C.d_off + (long long)Y * C.nx + x];
        else if (C.bc_x == kPeriodic) v = flags_all[C.d_off + (long long)Y * C.nx + ((x % C.nx) + C.nx) % C.nx];
        else if (C.bc_x == kOpen) v = flags_all[C.d_off + (long long)Y * C.nx + (x < 0 ? 0 : C.nx - 1)];
        else v = kSolidBit;
        out[s] = v;
    }
}

// Per-node copy of the adhesion vectors of one case's wall-list entries, in the compute type.
template <class R>
__global__ void k_wall_scatter(const DevCase* __restrict__ cases, int c, const int32_t* __restrict__ wl_node,
                               const double* __restrict__ wl_a, long long nwall_total, long long dense_total,
                               R* __restrict__ wa) {
    const DevCase C = cases[c];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < C.nwall; i += (long long)gridDim.x * blockDim.x) {
        const long long e = C.w_off + i;
        const long long o = C.d_off + wl_node[e];
        wa[o] = (R)wl_a[e];
        wa[dense_total + o] = (R)wl_a[nwall_total + e];
    }
}

// ------------------------------------------------------------------------------------------------
// f = f^eq(rho_k, 0) in the listed cases (along blockIdx.y), straight from the densities (case c at
// d_off - base).  The stored f*_i at x is what the next pull takes: w_i rho(x + e_i) from a fluid
// neighbour, w_i rho(x) across a blocked link or beyond an open edge (the outlet column's own value
// where the copy rule keeps it), minus w_i rho0 in 16-bit storage; G ghost columns repeat the
// periodic edges.
//
// The value is (R)(w_i rho - w_i rho0) with FP64 products.  4/9, 1/9 and 1/36 in FP64 are powers of
// two apart, so every direction's product, shift and rounding is an exact power of two times that of
// q = (R)(rho / 36 - rho0 / 36): one FP64 product and conversion per node and component instead of
// nine, the same bits.  (GB300 issues two FP64 operations per SM and cycle: at 36 of them per node the
// pass ran at the FP64 pipe's rate, 458 us on seven 1024 x 1024 FP32 cases where its 88 B per node
// take 95 us of HBM time; now 150 us, most of it its stores.)  A q so small that scaling it up
// could differ from rounding the larger product takes the direct form.
//
// A block of T columns (one halo column on each side) marches down `rows` rows; q of the row ahead goes
// into a ring of four shared-memory rows, one barrier per row.  A row takes a block about 1 us whatever the
// lattice, so 16 rows (at most: each block reads two halo rows more) serve only where they fill the GPU;
// a smaller lattice takes fewer, down to one, and one narrower than 30 columns blocks of 32.
// us, 16 rows of 128 columns -> this rule, FP32 / FP64: 40 x 300 24.8 -> 6.3 / 37.5 -> 6.4, 200 of 16 x 16
// 22.7 -> 7.6 / 35.2 -> 8.8, 9 x 5000 20.8 -> 10.4 / 35.0 -> 10.6, three 256 x 256 24.9 -> 12.5 / 41.0 -> 14.5.
// ------------------------------------------------------------------------------------------------
constexpr int kRestRows = 16;

// Near the denormals of R, or rounded to 0 (16 times what rounds to 0 need not).  With a storage shift
// 0 is an ordinary value, rho = rho0, and a nonzero difference is far above the denormals.  FP64 looks at
// the exponent: a comparison would cost its pipe as much as a product.
template <class S, class R>
__device__ __forceinline__ bool rest_tiny(R q) {
    if constexpr (sizeof(R) == 8) return (__double2hiint(q) & 0x7fffffff) < (60 << 20);  // below 2^-963
    else return q < (R)1e-30 && q > (R)-1e-30 && !(Store<S>::kShift && q == (R)0);
}

template <class S, int T>
__global__ void __launch_bounds__(T) k_set_rest(const DevCase* __restrict__ cases, int G, int rows, long long base,
                                                const uint8_t* __restrict__ solid_all,
                                                const uint16_t* __restrict__ flags_all,
                                                const double* __restrict__ rhoA_all,
                                                const double* __restrict__ rhoB_all, Pair<S>* __restrict__ out_all) {
    using R = typename ComputeOf<S>::type;
    using V = V2<R>;
    constexpr int W = T - 2;
    __shared__ V ring[4][T];
    const DevCase& C = cases[blockIdx.y];
    const int nx = C.nx, ny = C.ny, bcx = C.bc_x, t = threadIdx.x;
    const int nstrip = (nx + W - 1) / W;
    const int chunk = blockIdx.x / nstrip, xs = (blockIdx.x % nstrip) * W;
    const int y0 = chunk * rows, y1 = min(y0 + rows, ny);
    if (y0 >= ny) return;  // the grid covers the case with the most tiles
    const long long plane = C.pitch, row = 9 * plane;
    const double* rA = rhoA_all + (C.d_off - base);
    const double* rB = rhoB_all + (C.d_off - base);
    const uint8_t* sol = solid_all + C.d_off;
    const uint16_t* flags = flags_all + C.d_off;
    Pair<S>* out = out_all + C.f_off;
    const double sh[2] = {wq(5) * C.rho0[0], wq(5) * C.rho0[1]};
    const int x = xs - 1 + t;  // window column
    int X = x;                 // its lattice column, -1 outside a closed or open edge (never pulled from)
    if (x < 0 || x >= nx) X = bcx != kPeriodic ? -1 : (x < 0 ? x + nx : x % nx);
    const bool mine = t >= 1 && t <= W && x < nx;

    auto scaled = [&](double r, int k) -> double {
        double v = wq(5) * r;
        if constexpr (Store<S>::kShift) v -= sh[k];
        return v;
    };
    double nA = 0.0, nB = 0.0;  // densities of the row about to enter the ring
    auto load = [&](int r) {
        nA = nB = 0.0;
        if (r < 0 || r >= ny) {
            if (C.bc_y != kPeriodic) return;
            r += r < 0 ? ny : -ny;
        }
        if (X < 0) return;
        const long long s = (long long)r * nx + X;  // three loads in flight together
        const bool is_solid = sol[s] != 0;
        const double a = rA[s], b = rB[s];
        nA = is_solid ? 0.0 : a;
        nB = is_solid ? 0.0 : b;
    };
    auto put = [&](int r) { ring[r & 3][t] = V{(R)scaled(nA, 0), (R)scaled(nB, 1)}; };
    load(y0 - 1);
    put(y0 - 1);
    load(y0);
    put(y0);
    load(y0 + 1);
    uint16_t next_fl = mine ? flags[(long long)y0 * nx + x] : 0;
    for (int y = y0; y < y1; ++y) {
        const uint16_t fl = next_fl;
        put(y + 1);
        if (y + 1 < y1) {
            load(y + 2);
            if (mine) next_fl = flags[(long long)(y + 1) * nx + x];
        }
        __syncthreads();
        if (mine) {
            const bool solid = (fl & kSolidBit) != 0;
            Pair<S>* o = out + y * row + x + G;
            const bool gr = bcx == kPeriodic && x < G, gl = bcx == kPeriodic && x >= nx - G;  // ghost copies
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const bool edge = bcx == kOpen && (x + cx(i) < 0 || x + cx(i) >= nx);
                const bool own = i == 0 || edge || ((fl >> (opp(i) - 1)) & 1u);
                const V q = own ? ring[y & 3][t] : ring[(y + cy(i)) & 3][t + cx(i)];
                const R up = (R)(i == 0 ? 16 : (i <= 4 ? 4 : 1));
                V v{q.x * up, q.y * up};
                if (!solid && (rest_tiny<S, R>(q.x) || rest_tiny<S, R>(q.y))) {
                    int tx = x, ty = y;
                    if (!own) {
                        tx += cx(i);
                        ty += cy(i);
                        tx += tx < 0 ? nx : (tx >= nx ? -nx : 0);
                        ty += ty < 0 ? ny : (ty >= ny ? -ny : 0);
                    }
                    const long long z = (long long)ty * nx + tx;
                    double a = wq(i) * rA[z], b = wq(i) * rB[z];
                    if constexpr (Store<S>::kShift) {
                        a -= wq(i) * C.rho0[0];
                        b -= wq(i) * C.rho0[1];
                    }
                    v = sol[z] ? V{(R)0, (R)0} : V{(R)a, (R)b};
                }
                if (solid) v = V{(R)0, (R)0};
                store_pair<S, R>(o + i * plane, v.x, v.y);
                if (gr) store_pair<S, R>(o + i * plane + nx, v.x, v.y);
                if (gl) store_pair<S, R>(o + i * plane - nx, v.x, v.y);
            }
        }
    }
}

}  // namespace

cudaError_t launch_flags(Ctx& c, int ci, int32_t* row_counts) {
    const long long N = (long long)c.hcases[ci].nx * c.hcases[ci].ny;
    const int g = (int)((N + 255) / 256 < 8192 ? (N + 255) / 256 : 8192);
    k_flags<<<g, 256, 0, c.stream>>>(c.dcases, ci, c.solid, c.flags, row_counts);
    return cudaGetLastError();
}

cudaError_t launch_scan_rows(const int32_t* counts, int32_t* offsets, int n, cudaStream_t s) {
    k_scan<<<1, 1024, 0, s>>>(counts, offsets, n);
    return cudaGetLastError();
}

cudaError_t launch_wall_fill(Ctx& c, int ci, const int32_t* row_offsets) {
    k_wall_fill<<<c.hcases[ci].ny, 256, 0, c.stream>>>(c.dcases, ci, c.solid, c.flags, c.wsub, row_offsets,
                                                        c.wl_node, c.wl_subst, c.wl_seff, c.wl_a, c.nwall,
                                                        c.cases[ci].params.second_layer == LBM_SECOND_LAYER_PSI,
                                                        c.cases[ci].params.adhesion_stencil == LBM_ADHESION_D2Q9);
    return cudaGetLastError();
}

cudaError_t launch_flags_ghost(Ctx& c, int ci) {
    const long long n = (long long)c.hcases[ci].ny * c.gf_pitch[ci];
    const int g = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    k_flags_ghost<<<g, 256, 0, c.stream>>>(c.dcases, ci, c.flags, c.gflags + c.gf_off[ci], c.gf_pitch[ci]);
    return cudaGetLastError();
}

cudaError_t launch_wall_cast(Ctx& c, int ci) {
    const long long n = c.hcases[ci].nwall;
    if (n == 0) return cudaSuccess;
    const int g = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
    if (c.storage == LBM_STORE_F64)
        k_wall_scatter<double><<<g, 256, 0, c.stream>>>(c.dcases, ci, c.wl_node, c.wl_a, c.nwall, c.dense_elems, (double*)c.wa);
    else
        k_wall_scatter<float><<<g, 256, 0, c.stream>>>(c.dcases, ci, c.wl_node, c.wl_a, c.nwall, c.dense_elems, (float*)c.wa);
    return cudaGetLastError();
}

template <class S>
static void set_rest_launch(Ctx& c, dim3 g, int T, int rows, long long base, int c0, const double* rhoA, const double* rhoB) {
    const int G = ghost_cols(c.storage);
    Pair<S>* out = (Pair<S>*)c.f[c.cur];
    if (T == 32) k_set_rest<S, 32><<<g, 32, 0, c.stream>>>(c.dcases + c0, G, rows, base, c.solid, c.flags, rhoA, rhoB, out);
    else k_set_rest<S, 128><<<g, 128, 0, c.stream>>>(c.dcases + c0, G, rows, base, c.solid, c.flags, rhoA, rhoB, out);
}

// cases [c0, c0 + n) with the densities of case c at d_off - base
static cudaError_t set_rest_cases(Ctx& c, int c0, int n, long long base, const double* rhoA, const double* rhoB) {
    int widest = 0;
    for (int i = c0; i < c0 + n; ++i) widest = widest > c.hcases[i].nx ? widest : c.hcases[i].nx;
    const int T = widest <= 30 ? 32 : 128;
    auto tiles_of = [&](const DevCase& h, int rows) {
        return (long long)((h.nx + T - 3) / (T - 2)) * ((h.ny + rows - 1) / rows);
    };
    int rows = kRestRows;  // 1,024 threads on every SM, if there are rows enough
    for (; rows > 1; rows /= 2) {
        long long all = 0;
        for (int i = c0; i < c0 + n; ++i) all += tiles_of(c.hcases[i], rows);
        if (all * T >= 1024LL * c.num_sms) break;
    }
    for (const int end = c0 + n; c0 < end; c0 += 65535) {  // cases along gridDim.y, at most 65535 per launch
        const int m = end - c0 < 65535 ? end - c0 : 65535;
        long long tiles = 1;
        for (int i = c0; i < c0 + m; ++i) {
            const long long k = tiles_of(c.hcases[i], rows);
            tiles = tiles > k ? tiles : k;
        }
        const dim3 g((unsigned)tiles, (unsigned)m);
        switch (c.storage) {
            case LBM_STORE_F64: set_rest_launch<double>(c, g, T, rows, base, c0, rhoA, rhoB); break;
            case LBM_STORE_F32: set_rest_launch<float>(c, g, T, rows, base, c0, rhoA, rhoB); break;
            case LBM_STORE_F16_SHIFTED: set_rest_launch<__half>(c, g, T, rows, base, c0, rhoA, rhoB); break;
            default: set_rest_launch<__nv_bfloat16>(c, g, T, rows, base, c0, rhoA, rhoB); break;
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_set_rest_all(Ctx& c, const double* rhoA_all, const double* rhoB_all) {
    return set_rest_cases(c, 0, (int)c.hcases.size(), 0, rhoA_all, rhoB_all);
}

cudaError_t launch_set_rest(Ctx& c, int ci, const double* rhoA, const double* rhoB) {
    return set_rest_cases(c, ci, 1, c.hcases[ci].d_off, rhoA, rhoB);
}

}  // namespace lbm
