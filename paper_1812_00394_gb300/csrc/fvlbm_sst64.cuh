// fvlbm_sst64.cuh -- the k-omega SST step (Step 1, Sec. 2) beside the face-value stages, in double and
// for tangents (included by fvlbm_kernels.cu after the generic SST kernels, whose equations these
// are).
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
//   - in Duals, products with constants carry no derivative, and a quotient takes one division;
//   - a cell's diffusion coefficients nu + sigma nu_t are formed once, by the gradient kernel, and
//     read by its neighbours in place of (f1, nu_t).
// Measured on 473k SST cells (with the generic kernels before): gradient 154 us (354),
// update 164 us (397).
// Both are bound by the FP64 pipe, one thread per cell, one warp a block so that a mesh of 50k cells
// still spreads evenly over 608 schedulers.
constexpr int kSst64Block = 32;

// ---- arithmetic of doubles and Duals, the derivatives that are zero left out
__device__ __forceinline__ Dual mad(const Dual &a, const Dual &b, const Dual &c) {
    return Dual(::fma(a.v, b.v, c.v), ::fma(a.v, b.d, ::fma(a.d, b.v, c.d)));
}
__device__ __forceinline__ Dual mad(double a, const Dual &b, const Dual &c) {
    return Dual(::fma(a, b.v, c.v), ::fma(a, b.d, c.d));
}
__device__ __forceinline__ double mad(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ Dual scale(double a, const Dual &b) { return Dual(a * b.v, a * b.d); }
__device__ __forceinline__ double scale(double a, double b) { return a * b; }
__device__ __forceinline__ Dual shift(double a, const Dual &b) { return Dual(a + b.v, b.d); }
__device__ __forceinline__ double shift(double a, double b) { return a + b; }
__device__ __forceinline__ Dual recip(const Dual &b) {
    const double r = 1.0 / b.v;
    return Dual(r, -(r * r) * b.d);
}
__device__ __forceinline__ double recip(double b) { return 1.0 / b; }

// x as an integer in the order of the doubles (NaN apart)
__device__ __forceinline__ long long ord64(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ long long ord64(const Dual &x) { return ord64(x.v); }
template <class S>
__device__ __forceinline__ S min64(const S &a, const S &b) {
    return ord64(b) < ord64(a) ? b : a;
}
template <class S>
__device__ __forceinline__ S max64(const S &a, const S &b) {
    return ord64(b) > ord64(a) ? b : a;
}
// tanh of x >= 0
__device__ __forceinline__ double tanh64(double x) {
    const long long b = __double_as_longlong(x);
    if (b >= __double_as_longlong(20.0) && b <= __double_as_longlong(__longlong_as_double(0x7ff0000000000000ll)))
        return 1.0;
    if (b < __double_as_longlong(4e-9)) return x;
    return tanh(x);
}

__device__ __forceinline__ Dual tanh64(const Dual &x) {
    const double t = tanh64(x.v);
    return Dual(t, x.d * ::fma(-t, t, 1.0));
}

// a / b with one division
__device__ __forceinline__ double quot(double a, double b) { return a / b; }
__device__ __forceinline__ Dual quot(const Dual &a, const Dual &b) {
    const double r = 1.0 / b.v, q = a.v * r;
    return Dual(q, ::fma(-q, b.d, a.d) * r);
}

// min(1, (hi - c) / up where up > 0, (lo - c) / dn where dn < 0) for lo <= c <= hi
template <class S>
__device__ __forceinline__ S sst_limit64(const S &c, const S &lo, const S &hi, const S &up, const S &dn) {
    const S a = hi - c, b = c - lo, nd = -dn;
    const bool fa = ord64(up) > ord64(a), fb = ord64(nd) > ord64(b);
    S r = S(1.0);
    if (fa || fb) {
        const bool first = fa && (!fb || value_of(a) * value_of(nd) < value_of(b) * value_of(up));
        r = quot(first ? a : b, first ? up : nd);
    }
    return r;
}

__device__ __forceinline__ void sst_put2(double *p, double a, double b) {
    *reinterpret_cast<double2 *>(p) = make_double2(a, b);
}
__device__ __forceinline__ void sst_get2(const double *p, double &a, double &b) {
    const double2 x = *reinterpret_cast<const double2 *>(p);
    a = x.x;
    b = x.y;
}
__device__ __forceinline__ void sst_put2(Dual *p, const Dual &a, const Dual &b) {
    p[0] = a;
    p[1] = b;
}
__device__ __forceinline__ void sst_get2(const Dual *p, Dual &a, Dual &b) {
    a = p[0];
    b = p[1];
}

// u, v, k, omega of the face datum of slot m (neighbour or boundary value)
template <class S>
__device__ __forceinline__ void sst_datum64(const Geo<S> &G, int nb, const S *mac, const S *kk, const S *ww, const S &nu,
                                            const S *own, const S &di, S *q) {
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
template <class S>
__global__ void __launch_bounds__(kSst64Block)
    k_sst_grad64(const S *mac, const S *kk, const S *ww, const S *nut, S *__restrict__ grads, S *__restrict__ f1out,
                 S *__restrict__ rec8, S *__restrict__ rec2, Geo<S> G, int i0) {
    const int i = i0 + static_cast<int>(blockIdx.x) * kSst64Block + threadIdx.x;
    const size_t np = G.np;
    const double nu = G.ip[G.tile_inst[i / kTile]].nu;
    const S di = G.wdist[i];
    int nb[4];
    S W[8], R[8];
#pragma unroll
    for (int m = 0; m < 4; ++m) nb[m] = G.nbr[m * np + i];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        W[c] = G.lsq[c * np + i];
        R[c] = G.rown[c * np + i];
    }
    dep_wait();
    const S own[4] = {mac[np + i], mac[2 * np + i], kk[i], ww[i]};
    const S nti = nut[i];
    S g[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) g[c] = S(0.0);
    S lo[2] = {own[2], own[3]}, hi[2] = {own[2], own[3]};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
        S q[4];
        sst_datum64<S>(G, nb[m], mac, kk, ww, S(nu), own, di, q);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const S d = q[c] - own[c];
            g[2 * c] = mad(W[2 * m], d, g[2 * c]);
            g[2 * c + 1] = mad(W[2 * m + 1], d, g[2 * c + 1]);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            lo[c] = min64(lo[c], q[2 + c]);
            hi[c] = max64(hi[c], q[2 + c]);
        }
    }
    S up[2] = {S(0.0), S(0.0)}, dn[2] = {S(0.0), S(0.0)};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const S d = mad(g[4 + 2 * c], R[2 * m], g[5 + 2 * c] * R[2 * m + 1]);
            up[c] = max64(up[c], d);
            dn[c] = min64(dn[c], d);
        }
    }
    const S pk = sst_limit64(own[2], lo[0], hi[0], up[0], dn[0]);
    const S pw = sst_limit64(own[3], lo[1], hi[1], up[1], dn[1]);
    const S s12 = scale(0.5, g[1] + g[2]);
    const S SS = mad(g[0], g[0], mad(g[3], g[3], scale(2.0, s12) * s12));
    const S r = recip(own[3] * di);                     // 1 / (omega d)
    const S id = own[3] * r, iw = di * r;
    const S kw = iw * mad(g[4], g[6], g[5] * g[7]);     // grad k . grad omega / omega
    const S cd = max64(scale(2.0 * kSw2, kw), S(1e-20));
    const S arg = max64(scale(1.0 / kBstar, sqrt(own[2])) * r, scale(500.0 * nu, r) * id);
    const S num = scale(4.0 * kSw2, own[2]) * (id * id);
    S a1 = arg;
    if (value_of(num) < value_of(arg) * value_of(cd)) a1 = quot(num, cd);  // min(arg, 4 sigma_w2 k / (CD d^2))
    const S a2 = a1 * a1;
    const S f1 = tanh64(a2 * a2);
    grads[i] = SS;
    grads[np + i] = g[0] + g[3];
    grads[2 * np + i] = kw;
    f1out[i] = f1;
    S *o = rec8 + 8 * static_cast<size_t>(i);
    sst_put2(o, own[0], own[1]);
    sst_put2(o + 2, own[2], own[3]);
    sst_put2(o + 4, pk * g[4], pk * g[5]);
    sst_put2(o + 6, pw * g[6], pw * g[7]);
    sst_put2(rec2 + 2 * static_cast<size_t>(i), shift(nu, shift(kSk2, scale(kSk1 - kSk2, f1)) * nti),
             shift(nu, shift(kSw2, scale(kSw1 - kSw2, f1)) * nti));
}

// The update of the same cells: convection, diffusion, sources, point-implicit destruction; f2, nu_t
// and tau.  ddl: |n dl / A| / |d| of every face slot.
template <class S>
__global__ void __launch_bounds__(kSst64Block)
    k_sst_update64(const S *nut, const S *grads, const S *f1a, const S *rec8, const S *rec2, S *__restrict__ k_out,
                   S *__restrict__ w_out, S *__restrict__ nut_out, S *__restrict__ tau, Geo<S> G,
                   const S *__restrict__ ddl, int i0) {
    // backwards: the records that k_sst_grad64 wrote last are still in L2
    const int i = i0 + static_cast<int>(gridDim.x - 1 - blockIdx.x) * kSst64Block + threadIdx.x;
    const size_t np = G.np;
    const InstParam P = G.ip[G.tile_inst[i / kTile]];
    const double nu = P.nu, dt = value_of(cell_dt(G, P, i));
    const S di = G.wdist[i];
    int nb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) nb[m] = G.nbr[m * np + i];
    dep_wait();
    S ui, vi, ki, wi, lkx, lky, lwx, lwy, gki, gwi;
    const S *o = rec8 + 8 * static_cast<size_t>(i);
    sst_get2(o, ui, vi);
    sst_get2(o + 2, ki, wi);
    sst_get2(o + 4, lkx, lky);
    sst_get2(o + 6, lwx, lwy);
    sst_get2(rec2 + 2 * static_cast<size_t>(i), gki, gwi);
    S ck = S(0.0), cw = ck, dk = ck, dw = ck;  // all four doubled: mean face values without the halves
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] == kNone) continue;
        const S snx = G.sn[(2 * m) * np + i], sny = G.sn[(2 * m + 1) * np + i];
        const S rox = G.rown[(2 * m) * np + i], roy = G.rown[(2 * m + 1) * np + i];
        const S dl = ddl[m * np + i];
        S su, sv, kj, wj, sk, sw, rnx = S(0.0), rny = rnx, jkx = rnx, jky = rnx, jwx = rnx, jwy = rnx;
        if (nb[m] >= 0) {
            const S *q = rec8 + 8 * static_cast<size_t>(nb[m]);
            S uj, vj, gkj, gwj;
            sst_get2(q, uj, vj);
            sst_get2(q + 2, kj, wj);
            sst_get2(q + 4, jkx, jky);
            sst_get2(q + 6, jwx, jwy);
            sst_get2(rec2 + 2 * static_cast<size_t>(nb[m]), gkj, gwj);
            su = ui + uj;
            sv = vi + vj;
            sk = gki + gkj;
            sw = gwi + gwj;
            rnx = G.rnbr[(2 * m) * np + i];
            rny = G.rnbr[(2 * m + 1) * np + i];
        } else {
            S ub, vb;
            sst_bvals<S>(G, -nb[m] - 1, S(nu), ui, vi, ki, wi, di, ub, vb, kj, wj);
            su = scale(2.0, ub);
            sv = scale(2.0, vb);
            sk = scale(2.0, gki);
            sw = scale(2.0, gwi);
        }
        const S un = mad(su, snx, sv * sny);  // 2 (u_f . n) dl / A
        const bool out = nonneg(un);        // upwind side
        const S rx = out ? rox : rnx, ry = out ? roy : rny;
        const S kup = mad(out ? lkx : jkx, rx, mad(out ? lky : jky, ry, out ? ki : kj));
        const S wup = mad(out ? lwx : jwx, rx, mad(out ? lwy : jwy, ry, out ? wi : wj));
        ck = mad(un, kup, ck);
        cw = mad(un, wup, cw);
        dk = mad(sk * dl, kj - ki, dk);
        dw = mad(sw * dl, wj - wi, dw);
    }
    const S SS = grads[i], dv = grads[np + i], kw = grads[2 * np + i], f1 = f1a[i], nti = nut[i];
    constexpr double cw1 = kB1 / kBstar - kSw1 * kKappa * kKappa / 0.3;
    constexpr double cw2 = kB2 / kBstar - kSw2 * kKappa * kKappa / 0.3;
    const S gam = shift(cw2, scale(cw1 - cw2, f1)), beta = shift(kB2, scale(kB1 - kB2, f1));
    const S sh = mad(scale(-(2.0 / 3.0), dv), dv, scale(2.0, SS));  // 2 S_ij S_ij - 2/3 (div u)^2
    const S kd = scale(2.0 / 3.0, ki) * dv;
    const S pk = mad(nti, sh, -kd);
    S pw = sh;
    if (ord64(nti) > 0) pw = pw - quot(kd, nti);
    const S rk = mad(0.5, dk - ck, pk);
    const S rw = mad(0.5, dw - cw, mad(gam, pw, scale(2.0 * kSw2, shift(1.0, -f1)) * kw));
    const S ek = shift(1.0, scale(dt * kBstar, wi)), ew = shift(1.0, scale(dt, beta) * wi);
    const S ie = recip(ek * ew);
    S kn = mad(dt, rk, ki) * (ew * ie), wn = mad(dt, rw, wi) * (ek * ie);
    kn = value_of(kn) > 0.0 ? kn : S(0.0);
    wn = value_of(wn) > P.omega_min ? wn : S(P.omega_min);
    const S r = recip(wn * di);
    const S arg2 = max64(scale(2.0 / kBstar, sqrt(kn)) * r, scale(500.0 * nu, r) * (wn * r));
    const S f2 = tanh64(arg2 * arg2);
    const S nt = quot(scale(kA1, kn), max64(scale(kA1, wn), sqrt(scale(2.0, SS)) * f2));
    k_out[i] = kn;
    w_out[i] = wn;
    nut_out[i] = nt;
    tau[i] = scale(3.0, shift(nu, nt));
}
