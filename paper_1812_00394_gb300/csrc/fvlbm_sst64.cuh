// fvlbm_sst64.cuh -- the k-omega SST step (Step 1, Sec. 2) beside the face-value stages in double
// (included by fvlbm_kernels.cu after the generic SST kernels, whose equations these are).
//
// On this GPU a double operation takes 64 times a float one, and the generic kernels spend most of
// theirs on divisions, square roots, compares and tanh.  Here:
//   - the geometry is read as stored (weights, offsets, normals, and |n dl / A| / |d| as one number)
//     instead of derived from node positions (two divisions and four square roots a cell);
//   - the Barth-Jespersen factor takes the largest and the smallest increment over the faces
//     first: the quotients of one sign share their numerator, so one division is left per field,
//     and none where the increments stay within the bounds;
//   - the blending functions share 1 / (omega d); the two point-implicit quotients share one
//     division; the cross-diffusion limit of arg1 divides only where it is the smaller;
//   - minima, maxima and signs are taken on the bit patterns by the integer units;
//   - tanh is 1 above 20 and its argument below 4e-9, to double precision;
//   - a cell's diffusion coefficients nu + sigma nu_t are formed once, by the gradient kernel, and
//     read by its neighbours in place of (f1, nu_t).
// Measured on 473k SST cells (with the generic kernels before): gradient 154 us (354),
// update 164 us (397).
// Both are bound by the FP64 pipe, one thread per cell, in blocks of 64 so that a mesh of 50k cells
// still spreads evenly over 608 schedulers.
constexpr int kSst64Block = 64;

// x as an integer in the order of the doubles (NaN apart)
__device__ __forceinline__ long long ord64(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double min64(double a, double b) { return ord64(b) < ord64(a) ? b : a; }
__device__ __forceinline__ double max64(double a, double b) { return ord64(b) > ord64(a) ? b : a; }

// tanh of x >= 0
__device__ __forceinline__ double tanh64(double x) {
    const long long b = __double_as_longlong(x);
    if (b >= __double_as_longlong(20.0) && b <= __double_as_longlong(__longlong_as_double(0x7ff0000000000000ll)))
        return 1.0;
    if (b < __double_as_longlong(4e-9)) return x;
    return tanh(x);
}

// min(1, (hi - c) / up where up > 0, (lo - c) / dn where dn < 0) for lo <= c <= hi
__device__ __forceinline__ double sst_limit64(double c, double lo, double hi, double up, double dn) {
    const double a = hi - c, b = c - lo, nd = -dn;
    const bool fa = ord64(up) > ord64(a), fb = ord64(nd) > ord64(b);
    double r = 1.0;
    if (fa || fb) {
        const bool first = fa && (!fb || a * nd < b * up);
        r = (first ? a : b) / (first ? up : nd);
    }
    return r;
}

// u, v, k, omega of the face datum of slot m (neighbour or boundary value)
__device__ __forceinline__ void sst_datum64(const Geo<double> &G, int nb, const double *mac, const double *kk,
                                            const double *ww, double nu, const double *own, double di, double *q) {
    const size_t np = G.np;
    if (nb >= 0) {
        q[0] = mac[np + nb];
        q[1] = mac[2 * np + nb];
        q[2] = kk[nb];
        q[3] = ww[nb];
    } else {
        sst_bvals(G, -nb - 1, nu, own[0], own[1], own[2], own[3], di, q[0], q[1], q[2], q[3]);
    }
}

// Cells [i0, i0 + 64 blocks): gradients, the limited k and omega gradients, f1.  grads: S_ij S_ij,
// div u, grad k . grad omega / omega; rec8 = (u, v, k, omega, limited grad k, grad omega), rec2 =
// (nu + sigma_k nu_t, nu + sigma_omega nu_t).
__global__ void __launch_bounds__(kSst64Block)
    k_sst_grad64(const double *mac, const double *kk, const double *ww, const double *nut,
                 double *__restrict__ grads, double *__restrict__ f1out, double *__restrict__ rec8,
                 double *__restrict__ rec2, Geo<double> G, int i0) {
    dep_launch();
    const int i = i0 + static_cast<int>(blockIdx.x) * kSst64Block + threadIdx.x;
    const size_t np = G.np;
    const double nu = G.ip[G.tile_inst[i / kTile]].nu;
    const double di = G.wdist[i];
    int nb[4];
    double W[8], R[8];
#pragma unroll
    for (int m = 0; m < 4; ++m) nb[m] = G.nbr[m * np + i];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        W[c] = G.lsq[c * np + i];
        R[c] = G.rown[c * np + i];
    }
    dep_wait();
    const double own[4] = {mac[np + i], mac[2 * np + i], kk[i], ww[i]};
    const double nti = nut[i];
    double g[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    double lo[2] = {own[2], own[3]}, hi[2] = {own[2], own[3]};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
        double q[4];
        sst_datum64(G, nb[m], mac, kk, ww, nu, own, di, q);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double d = q[c] - own[c];
            g[2 * c] = fma(W[2 * m], d, g[2 * c]);
            g[2 * c + 1] = fma(W[2 * m + 1], d, g[2 * c + 1]);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            lo[c] = min64(lo[c], q[2 + c]);
            hi[c] = max64(hi[c], q[2 + c]);
        }
    }
    double up[2] = {0, 0}, dn[2] = {0, 0};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const double d = fma(g[4 + 2 * c], R[2 * m], g[5 + 2 * c] * R[2 * m + 1]);
            up[c] = max64(up[c], d);
            dn[c] = min64(dn[c], d);
        }
    }
    const double pk = sst_limit64(own[2], lo[0], hi[0], up[0], dn[0]);
    const double pw = sst_limit64(own[3], lo[1], hi[1], up[1], dn[1]);
    const double s12 = 0.5 * (g[1] + g[2]);
    const double SS = fma(g[0], g[0], fma(g[3], g[3], 2.0 * s12 * s12));
    const double r = 1.0 / (own[3] * di);                // 1 / (omega d)
    const double id = own[3] * r, iw = di * r;
    const double kw = iw * fma(g[4], g[6], g[5] * g[7]);  // grad k . grad omega / omega
    const double cd = max64(2.0 * kSw2 * kw, 1e-20);
    const double arg = max64((1.0 / kBstar) * sqrt(own[2]) * r, 500.0 * nu * r * id);
    const double num = 4.0 * kSw2 * own[2] * id * id;
    double a1 = arg;
    if (num < arg * cd) a1 = num / cd;                   // min(arg, 4 sigma_w2 k / (CD d^2))
    const double a2 = a1 * a1;
    const double f1 = tanh64(a2 * a2);
    grads[i] = SS;
    grads[np + i] = g[0] + g[3];
    grads[2 * np + i] = kw;
    f1out[i] = f1;
    double2 *o = reinterpret_cast<double2 *>(rec8 + 8 * static_cast<size_t>(i));
    o[0] = make_double2(own[0], own[1]);
    o[1] = make_double2(own[2], own[3]);
    o[2] = make_double2(pk * g[4], pk * g[5]);
    o[3] = make_double2(pw * g[6], pw * g[7]);
    *reinterpret_cast<double2 *>(rec2 + 2 * static_cast<size_t>(i)) =
        make_double2(fma(fma(f1, kSk1 - kSk2, kSk2), nti, nu), fma(fma(f1, kSw1 - kSw2, kSw2), nti, nu));
}

// The update of the same cells: convection, diffusion, sources, point-implicit destruction; f2, nu_t
// and tau.  ddl: |n dl / A| / |d| of every face slot.
__global__ void __launch_bounds__(kSst64Block)
    k_sst_update64(const double *nut, const double *grads, const double *f1a, const double *rec8, const double *rec2,
                   double *__restrict__ k_out, double *__restrict__ w_out, double *__restrict__ nut_out,
                   double *__restrict__ tau, Geo<double> G, const double *__restrict__ ddl, int i0) {
    dep_launch();
    // backwards: the records that k_sst_grad64 wrote last are still in L2
    const int i = i0 + static_cast<int>(gridDim.x - 1 - blockIdx.x) * kSst64Block + threadIdx.x;
    const size_t np = G.np;
    const InstParam P = G.ip[G.tile_inst[i / kTile]];
    const double nu = P.nu, di = G.wdist[i], dt = cell_dt(G, P, i);
    int nb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) nb[m] = G.nbr[m * np + i];
    dep_wait();
    const double2 *o = reinterpret_cast<const double2 *>(rec8 + 8 * static_cast<size_t>(i));
    const double2 uv = o[0], kwi = o[1], lk = o[2], lw = o[3];
    const double2 gi = *reinterpret_cast<const double2 *>(rec2 + 2 * static_cast<size_t>(i));
    const double own[4] = {uv.x, uv.y, kwi.x, kwi.y};
    const double ki = kwi.x, wi = kwi.y;
    double ck = 0, cw = 0, dk = 0, dw = 0;  // all four doubled: mean face values without the halves
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
        const double snx = G.sn[(2 * m) * np + i], sny = G.sn[(2 * m + 1) * np + i];
        const double rox = G.rown[(2 * m) * np + i], roy = G.rown[(2 * m + 1) * np + i];
        const double dl = ddl[m * np + i];
        double su, sv, kj, wj, sk, sw, rnx = 0.0, rny = 0.0;
        double2 jk = make_double2(0.0, 0.0), jw = jk;
        if (nb[m] >= 0) {
            const double2 *q = reinterpret_cast<const double2 *>(rec8 + 8 * static_cast<size_t>(nb[m]));
            const double2 a = q[0], b = q[1];
            jk = q[2];
            jw = q[3];
            const double2 gj = *reinterpret_cast<const double2 *>(rec2 + 2 * static_cast<size_t>(nb[m]));
            su = uv.x + a.x;
            sv = uv.y + a.y;
            kj = b.x;
            wj = b.y;
            sk = gi.x + gj.x;
            sw = gi.y + gj.y;
            rnx = G.rnbr[(2 * m) * np + i];
            rny = G.rnbr[(2 * m + 1) * np + i];
        } else {
            double ub, vb;
            sst_bvals(G, -nb[m] - 1, nu, own[0], own[1], ki, wi, di, ub, vb, kj, wj);
            su = 2.0 * ub;
            sv = 2.0 * vb;
            sk = 2.0 * gi.x;
            sw = 2.0 * gi.y;
        }
        const double un = fma(su, snx, sv * sny);  // 2 (u_f . n) dl / A
        const bool out = __double2hiint(un) >= 0;  // upwind side
        const double rx = out ? rox : rnx, ry = out ? roy : rny;
        const double kup = fma(out ? lk.x : jk.x, rx, fma(out ? lk.y : jk.y, ry, out ? ki : kj));
        const double wup = fma(out ? lw.x : jw.x, rx, fma(out ? lw.y : jw.y, ry, out ? wi : wj));
        ck = fma(un, kup, ck);
        cw = fma(un, wup, cw);
        dk = fma(sk * dl, kj - ki, dk);
        dw = fma(sw * dl, wj - wi, dw);
    }
    const double SS = grads[i], dv = grads[np + i], kw = grads[2 * np + i], f1 = f1a[i], nti = nut[i];
    constexpr double cw1 = kB1 / kBstar - kSw1 * kKappa * kKappa / 0.3;
    constexpr double cw2 = kB2 / kBstar - kSw2 * kKappa * kKappa / 0.3;
    const double gam = fma(f1, cw1 - cw2, cw2), beta = fma(f1, kB1 - kB2, kB2);
    const double sh = fma(-(2.0 / 3.0) * dv, dv, 2.0 * SS);  // 2 S_ij S_ij - 2/3 (div u)^2
    const double kd = (2.0 / 3.0) * ki * dv;
    const double pk = fma(nti, sh, -kd);
    double pw = sh;
    if (ord64(nti) > 0) pw -= kd / nti;
    const double rk = fma(0.5, dk - ck, pk);
    const double rw = fma(0.5, dw - cw, fma(gam, pw, 2.0 * kSw2 * (1.0 - f1) * kw));
    const double ek = fma(dt * kBstar, wi, 1.0), ew = fma(dt * beta, wi, 1.0);
    const double ie = 1.0 / (ek * ew);
    double kn = fma(dt, rk, ki) * (ew * ie), wn = fma(dt, rw, wi) * (ek * ie);
    kn = kn > 0.0 ? kn : 0.0;
    wn = wn > P.omega_min ? wn : P.omega_min;
    const double r = 1.0 / (wn * di);
    const double arg2 = max64((2.0 / kBstar) * sqrt(kn) * r, 500.0 * nu * r * (wn * r));
    const double f2 = tanh64(arg2 * arg2);
    const double nt = kA1 * kn / max64(kA1 * wn, sqrt(2.0 * SS) * f2);
    k_out[i] = kn;
    w_out[i] = wn;
    nut_out[i] = nt;
    tau[i] = 3.0 * (nu + nt);
}
