// fvlbm_lanes.cuh -- the face-value stages in double for small handles, four threads per cell
// (included by fvlbm_kernels.cu after fvlbm_fused_fv.cuh).
//
// A double operation occupies a scheduler of this GPU for 64 cycles whatever the instruction-level
// parallelism (measured: one warp of dependent or independent FMAs, 64.1 cycles each), so a small
// mesh is bound by how evenly its warps spread over the 608 schedulers: one thread per cell makes
// 128 warps of a 64 x 64 cavity, in 64-cell items on 64 of the 152 SMs, and the ring cells of small
// items are work done twice.  Here each cell is four threads, one direction pair each (512 warps),
// and a stage is two kernels without any halo:
//   k_lane_relax         f^(1) of every cell, and f^n + dt Gamma^c(1) / 3
//   k_lane_face          boundary values and outgoing face values, to memory
//   k_lane_flux<STAGE>   flux and stage algebra
// Moments are sums over the four lanes by shuffles, in the order of fv_moments, and everything else
// is the same chain of operations as in k_fused_fv, so a cell's values do not depend on which of
// the two kinds of kernels ran (a step with statistics runs the fused ones).  The price is the
// part of the algebra that all four lanes repeat (a third more operations), so larger meshes,
// which fill the schedulers anyway, keep one thread per cell.  Measured, us per step, one against
// four threads per cell: quad cavities of 4k cells 49.1 / 33.8, 10k 55.2 / 44.4, 20k 71.0 / 68.5, 24k
// 73.2 / 81.1, 80k 189 / 212; triangles 20k 64.6 / 65.1; SST airfoils of 4k cells 72.3 / 55.0, 10k
// 73.7 / 64.4, 20k 89.1 / 88.7, 24k 94.3 / 97.7.  One warp a block: it is placed on the emptiest
// scheduler, where blocks of two or four ran up to a third longer.
constexpr int kLaneBlock = 32;

// Layout of the stage values, B and C: pairs at [8 i + 2 p], f_0 at [8 np + i]; of the boundary
// values: pairs at [8 b + 2 p].

// Moments of a cell whose pair p = lane & 3 this thread holds.
__device__ __forceinline__ FvMoments<double> lane_moments(double2 f, double f0, double rho0, int p) {
    FvMoments<double> M;
    auto sum = [](double x) {
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        return x + __shfl_xor_sync(0xffffffffu, x, 2);
    };
    const double d = f.x - f.y;
    M.dr = f0 + sum(f.x + f.y);
    M.jx = sum(p == 1 ? 0.0 : (p == 3 ? -d : d));
    M.jy = sum(p == 0 ? 0.0 : d);
    fv_velocity(M, rho0);
    return M;
}

__global__ void __launch_bounds__(kLaneBlock)
    k_lane_relax(const double *fn, const double *tau, double *__restrict__ rows, double *__restrict__ Brow,
                 Geo<double> G) {
    const int t = blockIdx.x * kLaneBlock + threadIdx.x, i = t >> 2, p = t & 3;
    const size_t np = G.np;
    const InstParam &P = G.ip[G.tile_inst[i / kTile]];
    const double rho0 = P.rho0, dt = cell_dt(G, P, i);
    dep_wait();
    const int a1 = fv_first(p);
    double2 f = make_double2(fn[a1 * np + i], fn[(a1 + 2) * np + i]);
    const double f0 = fn[i];
    const FvMoments<double> M = lane_moments(f, f0, rho0, p);
    double a, g;
    fv_factors(dt, tau[i], 0.25, a, g);
    g *= -1.0 / 3.0;
    const double2 eq = fv_feq<double>(M, p);
    const double2 d = make_double2(f.x - eq.x, f.y - eq.y);
    reinterpret_cast<double2 *>(Brow)[4 * static_cast<size_t>(i) + p] =
        make_double2(::fma(g, d.x, f.x), ::fma(g, d.y, f.y));
    reinterpret_cast<double2 *>(rows)[4 * static_cast<size_t>(i) + p] =
        make_double2(::fma(a, d.x, eq.x), ::fma(a, d.y, eq.y));
    if (p == 0) {
        const double eq0 = fv_feq0(M), d0 = f0 - eq0;
        Brow[8 * np + i] = ::fma(g, d0, f0);
        rows[8 * np + i] = ::fma(a, d0, eq0);
    }
}

// bits: bit 4 m + p set when the first member of pair p leaves the cell through face m.
__global__ void __launch_bounds__(kLaneBlock)
    k_lane_face(const double *rows, double *brow, double *__restrict__ fv, Geo<double> G,
                const double *__restrict__ geo, const int *__restrict__ obits, const double *__restrict__ bnrm) {
    const int t = blockIdx.x * kLaneBlock + threadIdx.x, i = t >> 2, p = t & 3;
    const size_t np = G.np;
    const double rho0 = G.ip[G.tile_inst[i / kTile]].rho0;
    int nb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) nb[k] = G.nbr[k * np + i];
    const int bits = obits[i] >> p;
    double A[16];
#pragma unroll
    for (int k = 0; k < 16; k += 4) fv_load_geo4(geo, i, k, A + k);
    dep_wait();
    const double2 *r2 = reinterpret_cast<const double2 *>(rows);
    const double2 c = r2[4 * static_cast<size_t>(i) + p];
    double2 d[4];
    bool bnd = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        d[k] = c;
        if (nb[k] >= 0) d[k] = r2[4 * static_cast<size_t>(nb[k]) + p];
        bnd |= nb[k] < 0 && nb[k] != kNone;
    }
    if (__any_sync(0xffffffffu, bnd)) {  // boundary values of this stage, kept for the flux
        const FvMoments<double> M = lane_moments(c, rows[8 * np + i], rho0, p);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (nb[k] >= 0 || nb[k] == kNone) continue;
            const int b = -nb[k] - 1;
            d[k] = fv_ghost_pair(G.btype[b], G.bval[b], G.bval[G.nbt + b], G.bval[2 * static_cast<size_t>(G.nbt) + b],
                                 bnrm[b], bnrm[G.nbt + b], M, rho0, p, c);
            reinterpret_cast<double2 *>(brow)[4 * static_cast<size_t>(b) + p] = d[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = make_double2(d[k].x - c.x, d[k].y - c.y);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] < 0) continue;
        const bool first = (bits >> (4 * m)) & 1;
        double v = first ? c.x : c.y;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < 3 || nb[3] != kNone) v = ::fma(A[4 * m + k], first ? d[k].x : d[k].y, v);
        fv[16 * static_cast<size_t>(i) + 4 * m + p] = v;
    }
}

template <int STAGE>
__global__ void __launch_bounds__(kLaneBlock)
    k_lane_flux(const double *rows, const double *brow, const double *fv, double *__restrict__ rows_out, double *fn,
                double *Brow, double *Crow, const double *tau, double *__restrict__ mac, Geo<double> G,
                const double *__restrict__ geo, const int *__restrict__ back, const int *__restrict__ obits) {
    const int t = blockIdx.x * kLaneBlock + threadIdx.x, i = t >> 2, p = t & 3;
    const size_t np = G.np;
    const InstParam &P = G.ip[G.tile_inst[i / kTile]];
    const double rho0 = P.rho0, dt = cell_dt(G, P, i);
    int nb[4], src[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        nb[m] = G.nbr[m * np + i];
        src[m] = nb[m] >= 0 ? back[m * np + i] : 0;
    }
    const int bits = obits[i] >> p;
    double sn[8];
    if (nb[3] != kNone) {
        fv_load_geo4(geo, i, 16, sn);
        fv_load_geo4(geo, i, 20, sn + 4);
    } else {  // (see kFvGeo)
        double q[4];
        sn[0] = geo[fv_geo_at<double>(i, 3)];
        sn[1] = geo[fv_geo_at<double>(i, 7)];
        fv_load_geo4(geo, i, 12, q);
        sn[2] = geo[fv_geo_at<double>(i, 11)];
        sn[3] = q[0]; sn[4] = q[1]; sn[5] = q[2];
        sn[6] = sn[7] = 0.0;
    }
    dep_wait();
    double2 ac = make_double2(0.0, 0.0);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
        double2 v;
        if (nb[m] < 0) {
            v = reinterpret_cast<const double2 *>(brow)[4 * static_cast<size_t>(-nb[m] - 1) + p];
        } else {
            const double o = fv[16 * static_cast<size_t>(i) + 4 * m + p];
            const double n = fv[16 * static_cast<size_t>(nb[m]) + 4 * src[m] + p];
            v = (bits >> (4 * m)) & 1 ? make_double2(o, n) : make_double2(n, o);
        }
        const double en = fv_en<double>(p, sn[2 * m], sn[2 * m + 1]);
        ac.x = ::fma(en, v.x, ac.x);
        ac.y = ::fma(-en, v.y, ac.y);
    }
    const size_t at = 4 * static_cast<size_t>(i) + p;
    const int a1 = fv_first(p);
    double2 *B2 = reinterpret_cast<double2 *>(Brow), *C2 = reinterpret_cast<double2 *>(Crow);
    if (STAGE == 3) {
        const double dt3 = -(dt * (1.0 / 3.0));
        const double2 r = reinterpret_cast<const double2 *>(rows)[at], c = C2[at];
        const double2 f = make_double2(::fma(dt3, ac.x, r.x + c.x), ::fma(dt3, ac.y, r.y + c.y));
        const double f0 = rows[8 * np + i];
        fn[a1 * np + i] = f.x;
        fn[(a1 + 2) * np + i] = f.y;
        const FvMoments<double> M = lane_moments(f, f0, rho0, p);
        if (p == 0) fn[i] = f0;
        if (p < 3) mac[p * np + i] = p == 0 ? M.r : (p == 1 ? M.u : M.v);
    } else {
        double a, g;
        fv_factors(dt, tau[i], STAGE == 1 ? 0.25 : 1.0 / 3.0, a, g);
        const double hdt = -0.5 * dt, dt6 = dt * (1.0 / 6.0);
        g *= -1.0 / 3.0;
        const double2 b = B2[at];
        const double B0 = Brow[8 * np + i];
        double2 x;
        double X0;
        if (STAGE == 1) {  // from f^n
            x = make_double2(fn[a1 * np + i], fn[(a1 + 2) * np + i]);
            X0 = fn[i];
        } else {
            x = b;
            X0 = B0;
        }
        x.x = ::fma(hdt, ac.x, x.x);
        x.y = ::fma(hdt, ac.y, x.y);
        const FvMoments<double> M = lane_moments(x, X0, rho0, p);
        const double2 eq = fv_feq<double>(M, p);
        const double2 d = make_double2(x.x - eq.x, x.y - eq.y);
        reinterpret_cast<double2 *>(rows_out)[at] = make_double2(::fma(a, d.x, eq.x), ::fma(a, d.y, eq.y));
        if (STAGE == 1) {
            B2[at] = make_double2(::fma(g, d.x, ::fma(hdt, ac.x, b.x)), ::fma(g, d.y, ::fma(hdt, ac.y, b.y)));
            C2[at] = make_double2(dt6 * ac.x, dt6 * ac.y);
        } else {
            const double2 c = C2[at];
            C2[at] = make_double2(::fma(dt6, ac.x, c.x), ::fma(dt6, ac.y, c.y));
        }
        if (p == 0) {
            const double eq0 = fv_feq0(M), d0 = X0 - eq0;
            if (STAGE == 1) Brow[8 * np + i] = ::fma(g, d0, B0);
            rows_out[8 * np + i] = ::fma(a, d0, eq0);
        }
    }
}
