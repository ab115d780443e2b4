// fvlbm_tangent.cuh -- the IMEX step of tangent handles (included by fvlbm_kernels.cu): the face-value
// form of the stages with every number a Dual, in two kernels a stage.
//
// A Dual product is three FP64 operations and GB300 has few of those, so what counts is how many
// products a step takes.  The generic two-pass kernels formed nine gradients per cell, both sides
// of every face value and products with constants whose derivative is zero; here, as in the
// face-value stages (fvlbm_fused_fv.cuh), a cell forms the outgoing member of each direction pair
// at each of its faces once, from the coefficients A_mk = W_k . r_m, and the flux kernel reads its
// own and its neighbours'.  Where e . n is exactly 0 (axis-aligned faces) a direction carries no flux
// but its derivative with respect to the geometry does; the generic kernels take the cell's own
// value there on both sides of the face, so such pairs ("ties") also publish their other member,
// for the cell itself.  Boundary values are formed once, by the owner's thread, when it
// writes the stage value.  Per stage:
//   k_tan_face         four threads per cell, one direction pair each: face values to HBM (256 bytes
//                      a cell, which costs little beside the arithmetic)
//   k_tan_flux<STAGE>  one thread per cell: flux, stage algebra, boundary values of the new stage
// and k_tan_relax before them (f^(1) and its boundary values).  Measured on two 20k-cell SST
// airfoils: the stages took 694 us a step in the generic kernels, 248 here.
constexpr int kTanBlock = 32;

// e_first(p) . (x, y)
__device__ __forceinline__ Dual tan_en(int p, const Dual &x, const Dual &y) {
    return p == 0 ? x : (p == 1 ? y : (p == 2 ? x + y : y - x));
}

struct TanMoments {
    Dual dr, r, u, v, jx, jy, uu;
};
// f: pairs (first, second) x 4; f0: rest direction
__device__ __forceinline__ TanMoments tan_moments(const Dual *f, const Dual &f0, double rho0) {
    TanMoments M;
    const Dual d2 = f[4] - f[5], d3 = f[6] - f[7];
    M.dr = f0 + (((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])));
    M.jx = (f[0] - f[1]) + (d2 - d3);
    M.jy = (f[2] - f[3]) + (d2 + d3);
    M.r = shift(rho0, M.dr);
    const Dual ir = recip(M.r);
    M.u = M.jx * ir;
    M.v = M.jy * ir;
    M.uu = scale(1.5, mad(M.u, M.u, M.v * M.v));
    return M;
}
__device__ __forceinline__ void tan_feq(const TanMoments &M, int p, Dual &a, Dual &b) {
    const double w = fv_w<double>(p);
    const Dual eu = tan_en(p, M.u, M.v);
    const Dual s = scale(w, mad(M.r, mad(scale(4.5, eu), eu, -M.uu), M.dr));
    const Dual t = scale(3.0 * w, tan_en(p, M.jx, M.jy));
    a = s + t;
    b = s - t;
}
__device__ __forceinline__ Dual tan_feq0(const TanMoments &M) { return scale(4.0 / 9.0, M.dr - M.r * M.uu); }

// Boundary values of face b of a cell with stage value f, f0 and moments M (fv_ghost).
__device__ __forceinline__ void tan_boundary(const Geo<Dual> &G, const Dual *bnrm, int b, const Dual *f,
                                             const TanMoments &M, double rho0, Dual *out) {
    const int type = G.btype[b];
    const Dual rb = G.bval[b], ub = G.bval[G.nbt + b], vb = G.bval[2 * static_cast<size_t>(G.nbt) + b];
    if (type == FVLBM_BC_FARFIELD) {
        TanMoments B;
        B.dr = shift(-rho0, rb);
        B.r = rb;
        B.u = ub;
        B.v = vb;
        B.jx = rb * ub;
        B.jy = rb * vb;
        B.uu = scale(1.5, mad(ub, ub, vb * vb));
        const double nx = bnrm[b].v, ny = bnrm[G.nbt + b].v;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const double en = fv_en<double>(p, nx, ny);
            Dual e1, e2;
            tan_feq(B, p, e1, e2);
            out[2 * p] = en < 0.0 ? e1 : f[2 * p];
            out[2 * p + 1] = en > 0.0 ? e2 : f[2 * p + 1];
        }
        return;
    }
    const bool outlet = type == FVLBM_BC_OUTLET;
    const Dual q = shift(-rho0, rb) - M.dr;
    const Dual du = ub - M.u, dv = vb - M.v, su = ub + M.u, sv = vb + M.v;
    const Dual duu = scale(1.5, mad(du, su, dv * sv));
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        Dual s, a;
        if (outlet) {
            const Dual eu = tan_en(p, M.u, M.v);
            s = q * shift(1.0, mad(scale(4.5, eu), eu, -M.uu));
            a = scale(3.0, q * eu);
        } else {
            const Dual de = tan_en(p, du, dv);
            s = M.r * mad(scale(4.5, de), tan_en(p, su, sv), -duu);
            a = scale(3.0, M.r * de);
        }
        out[2 * p] = mad(fv_w<double>(p), s + a, f[2 * p]);
        out[2 * p + 1] = mad(fv_w<double>(p), s - a, f[2 * p + 1]);
    }
}

// Stage value of cell i: pairs into its row, f_0 after the rows; the boundary values of its
// boundary faces into their rows (M: moments of f, the same for a value and its relaxed one).
__device__ __forceinline__ void tan_store(const Geo<Dual> &G, const Dual *bnrm, int i, const Dual *f, const Dual &f0,
                                          const TanMoments &M, double rho0, Dual *rows, Dual *brow) {
    const size_t np = G.np;
#pragma unroll
    for (int a = 0; a < 8; ++a) rows[8 * static_cast<size_t>(i) + a] = f[a];
    rows[8 * np + i] = f0;
    for (int m = 0; m < 4; ++m) {
        const int nb = G.nbr[m * np + i];
        if (nb >= 0 || nb == kNone) continue;
        Dual b[8];
        tan_boundary(G, bnrm, -nb - 1, f, M, rho0, b);
#pragma unroll
        for (int a = 0; a < 8; ++a) brow[8 * static_cast<size_t>(-nb - 1) + a] = b[a];
    }
}

__global__ void __launch_bounds__(kTanBlock)
    k_tan_relax(const Dual *fn, const Dual *tau, Dual *__restrict__ rows, Dual *__restrict__ brow, Geo<Dual> G,
                const Dual *__restrict__ bnrm) {
    const int i = blockIdx.x * kTanBlock + threadIdx.x;
    const size_t np = G.np;
    const InstParam &P = G.ip[G.tile_inst[i / kTile]];
    const double dt = cell_dt(G, P, i).v, rho0 = P.rho0;
    Dual f[8], f0 = fn[i];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        f[2 * p] = fn[fv_first(p) * np + i];
        f[2 * p + 1] = fn[fv_second(p) * np + i];
    }
    const TanMoments M = tan_moments(f, f0, rho0);
    const Dual t = tau[i], a = t * recip(shift(0.25 * dt, t));
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        Dual e1, e2;
        tan_feq(M, p, e1, e2);
        f[2 * p] = mad(a, f[2 * p] - e1, e1);
        f[2 * p + 1] = mad(a, f[2 * p + 1] - e2, e2);
    }
    const Dual e0 = tan_feq0(M);
    f0 = mad(a, f0 - e0, e0);
    tan_store(G, bnrm, i, f, f0, M, rho0, rows, brow);
}

// Outgoing face values: thread (cell, pair).  obits: bit 4 m + p set when the first member of pair p
// leaves the cell through face m; bit 16 + 4 m + p: a tie, whose other member goes to fv2.
__global__ void __launch_bounds__(kTanBlock * 2)
    k_tan_face(const Dual *rows, const Dual *brow, Geo<Dual> G, const Dual *__restrict__ A,
               const int *__restrict__ obits, Dual *__restrict__ fv, Dual *__restrict__ fv2) {
    const int t = blockIdx.x * (kTanBlock * 2) + threadIdx.x;
    const int i = t >> 2, p = t & 3;
    const size_t np = G.np;
    const Dual c0 = rows[8 * static_cast<size_t>(i) + 2 * p], c1 = rows[8 * static_cast<size_t>(i) + 2 * p + 1];
    int nb[4];
    Dual d[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        nb[k] = G.nbr[k * np + i];
        if (nb[k] == kNone) continue;
        const Dual *r = nb[k] >= 0 ? rows + 8 * static_cast<size_t>(nb[k]) : brow + 8 * static_cast<size_t>(-nb[k] - 1);
        d[k][0] = r[2 * p] - c0;
        d[k][1] = r[2 * p + 1] - c1;
    }
    const int bits = obits[i];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] < 0) continue;
        const bool first = (bits >> (4 * m + p)) & 1;
        auto value = [&](bool one) {
            Dual v = one ? c0 : c1;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (nb[k] == kNone) continue;
                v = mad(A[(4 * m + k) * np + i], one ? d[k][0] : d[k][1], v);
            }
            return v;
        };
        fv[16 * static_cast<size_t>(i) + 4 * m + p] = value(first);
        if ((bits >> (16 + 4 * m + p)) & 1) fv2[16 * static_cast<size_t>(i) + 4 * m + p] = value(!first);
    }
}

// Flux of cell i from the face values, then the stage algebra (fvlbm_fused_fv.cuh, double).
template <int STAGE, bool STATS>
__global__ void __launch_bounds__(STATS ? kTile : kTanBlock)
    k_tan_flux(const Dual *rows_in, Dual *__restrict__ rows_out, Dual *brow, const Dual *fv, const Dual *fv2, Dual *fn,
               Dual *Bacc, Dual *Cacc, const Dual *tau, Dual *mac, double *__restrict__ partial, Geo<Dual> G,
               const int *__restrict__ back, const int *__restrict__ obits, const Dual *__restrict__ bnrm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t np = G.np;
    const InstParam &P = G.ip[G.tile_inst[i / kTile]];
    const double dt = cell_dt(G, P, i).v, rho0 = P.rho0;
    Dual ac[8];
    const int bits = obits[i];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int nb = G.nbr[m * np + i];
        if (nb == kNone) continue;
        const Dual snx = G.sn[(2 * m) * np + i], sny = G.sn[(2 * m + 1) * np + i];
        const Dual *q = nb < 0 ? brow + 8 * static_cast<size_t>(-nb - 1)
                               : fv + 16 * static_cast<size_t>(nb) + 4 * back[m * np + i];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            Dual v1, v2;
            if (nb < 0) {
                v1 = q[2 * p];
                v2 = q[2 * p + 1];
            } else {
                const size_t at = 16 * static_cast<size_t>(i) + 4 * m + p;
                const Dual o = fv[at], n = (bits >> (16 + 4 * m + p)) & 1 ? fv2[at] : q[p];
                const bool first = (bits >> (4 * m + p)) & 1;
                v1 = first ? o : n;
                v2 = first ? n : o;
            }
            const Dual en = tan_en(p, snx, sny);
            ac[2 * p] = mad(en, v1, ac[2 * p]);
            ac[2 * p + 1] = mad(-en, v2, ac[2 * p + 1]);
        }
    }
    double st[4] = {0.0, 0.0, 0.0, 0.0};
    if (STAGE != 3) {
        const Dual t = tau[i];
        const Dual a = t * recip(shift((STAGE == 1 ? 0.25 : 1.0 / 3.0) * dt, t));
        const Dual *src = STAGE == 1 ? fn : Bacc;
        Dual X[8], X0 = src[i];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            X[2 * p] = mad(-0.5 * dt, ac[2 * p], src[fv_first(p) * np + i]);
            X[2 * p + 1] = mad(-0.5 * dt, ac[2 * p + 1], src[fv_second(p) * np + i]);
        }
        const TanMoments M = tan_moments(X, X0, rho0);
        // B = X + dt/3 (Gamma^c(1) + Gamma^c(2)), with dt Gamma^c(J) = 4 (f^(J) - what it was relaxed from)
        auto acc_b = [&](int al, const Dual &x, const Dual &f2, const Dual &f1) {
            const Dual f0 = fn[al * np + i];
            Bacc[al * np + i] = mad(4.0 / 3.0, (f1 - f0) + (f2 - x), x);
        };
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            Dual e[2];
            tan_feq(M, p, e[0], e[1]);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int al = s == 0 ? fv_first(p) : fv_second(p);
                const Dual f = mad(a, X[2 * p + s] - e[s], e[s]);
                if (STAGE == 1) {
                    acc_b(al, X[2 * p + s], f, rows_in[8 * static_cast<size_t>(i) + 2 * p + s]);
                    Cacc[al * np + i] = scale(dt / 6.0, ac[2 * p + s]);
                } else {
                    Cacc[al * np + i] = mad(dt / 6.0, ac[2 * p + s], Cacc[al * np + i]);
                }
                X[2 * p + s] = f;
            }
        }
        const Dual e0 = tan_feq0(M), f0 = mad(a, X0 - e0, e0);
        if (STAGE == 1) acc_b(0, X0, f0, rows_in[8 * np + i]);
        tan_store(G, bnrm, i, X, f0, M, rho0, rows_out, brow);
    } else {
        Dual f[8], f0 = rows_in[8 * np + i];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int al = s == 0 ? fv_first(p) : fv_second(p);
                f[2 * p + s] = mad(-dt / 3.0, ac[2 * p + s],
                                   rows_in[8 * static_cast<size_t>(i) + 2 * p + s] + Cacc[al * np + i]);
                fn[al * np + i] = f[2 * p + s];
            }
        fn[i] = f0;
        const TanMoments M = tan_moments(f, f0, rho0);
        if (STATS) {
            const double un = M.u.v, vn = M.v.v, r = M.r.v;
            const double du = un - mac[np + i].v, dv = vn - mac[2 * np + i].v;
            st[0] = du * du + dv * dv;
            st[1] = un * un + vn * vn;
            st[2] = r * G.area[i].v;
            st[3] = isfinite(un) && isfinite(vn) && isfinite(r) ? 0.0 : 1.0;
        }
        mac[i] = M.r;
        mac[np + i] = M.u;
        mac[2 * np + i] = M.v;
    }
    if (STATS) block_sum<4>(st, partial + 4 * blockIdx.x);
}
