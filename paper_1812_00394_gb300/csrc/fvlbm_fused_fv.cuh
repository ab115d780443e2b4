// fvlbm_fused_fv.cuh -- the face-value form of the fused IMEX stage kernel (included by
// fvlbm_kernels.cu after the common device helpers).
//
// What one stage computes is unchanged: least-squares gradients of f^(J) (Step 2), the upwind
// linear face values f_{alpha,bc} = f_up + grad f_up . (x_f - x_up) and the convection term of
// Eq. (advection), then the local stage algebra (Eqs. (sumimeximplicitnew), (fnewstage),
// (imextwo)).  What changes is who forms the face values, and how.
//
// For a face with normal n the nine directions split into the rest direction (no flux) and
// four opposite pairs (alpha, alpha-bar), e_alphabar = -e_alpha, so that e_alphabar . n =
// -e_alpha . n: of every pair exactly one direction leaves the cell through the face (its
// upwind side is the cell itself) and the other enters it (its upwind side is the neighbour).
// Each cell therefore has, per face, four "outgoing" face values -- one per pair -- and the
// neighbour's incoming values at that face are exactly the neighbour's outgoing values at the
// same face.  Every item cell forms its four outgoing values per face once and publishes them
// in shared memory; the flux of a cell then reads, per face, its own four values and its
// neighbour's four (one 16-byte load each).  Which member of a pair leaves through a face is
// decided once on the host (FP64 geometry, e_alpha . n >= 0 on one side of the face and the
// complement on the other side), so the two sides always agree.
//
// Of a ring-1 cell only the faces it shares with the item matter (a little over one of its
// three or four): each such "cut" face is a record of its own -- five row indices, the
// coefficients, four outgoing bits -- and the ring cell's remaining faces are never formed.
//
// The accumulators B and C are kept in tiles of IT cells, [tile][alpha][IT] (they live from stage
// 1 to stage 3 only), so that an item's rows are one copy and the rows a thread writes are
// at fixed offsets.
//
// Two forms of the face value.  Float: the least-squares gradient, then f_c + grad f . r_m for
// each face.  Double: a face value is linear in the differences to the cell's face data,
// grad f . r_m = sum_k (W_k . r_m) (f_k - f_c), so the host stores A_mk = W_k . r_m and the kernel
// forms only the outgoing member of each pair: 60 operations a triangle instead of about 125,
// which counts where the FP64 rate is 1/64 of the FP32 rate.  (Float keeps the gradient form:
// on y+ ~ 1 meshes the strain rate amplifies the last bits of the velocities, and the eddy
// viscosity moved by 5e-5 with the other order of operations, as much as it is off FP64.)
//
// Boundary faces are ghost rows: before the face values, one thread per boundary face of the
// item and ring-1 cells forms the boundary values (boundary_values) from the owner's staged row
// and stores them as one more staged row, which the face values and the flux then read like a
// neighbour's.  The boundary arithmetic appears once, and no main phase branches on it.
//
// Work items: a block of IT consecutive cells, or -- where its halo would not fit the
// shared-memory budget -- a half, quarter or eighth of one (an instance's cells are padded to a
// multiple of 256, so no item straddles two instances).  One CTA of NT threads per item; see
// FvShape for the block sizes.
//
// Layouts for the stages of this form.  f^n stays structure-of-arrays (shared with the rest of
// the library).  The stage values f^(2), f^(3) that stages 1 and 2 write and stages 2 and 3
// read are cell-major: alpha = 1..8 in pair order (1,3)(2,4)(5,7)(6,8) in one 32-byte row per
// cell (its two halves swapped where bit 2 of the cell index is set), then f_0 of every cell,
// so that an item's own rows are one contiguous bulk copy and a halo cell's eight moving
// directions are one 32-byte sector.  The geometry is read in 16-byte chunks of 32 cells (see
// kFvGeo).
//
// Staging, all issued before any wait: the item's own rows (its stage values, its accumulator
// rows and tau) by bulk copies on one mbarrier, shared out over the warps; the halo rows and
// the instance parameters by cp.async; the item cell's own adjacency and coefficients, the cut
// records and the halo cells' tau straight into registers.  A CTA's first loads (its halo ids
// and its header) do not depend on each other, so the gathers wait on two memory round trips.
// Stage 1 takes its own f^n rows from the accumulator copy (the algebra reads them there too)
// and relaxes every staged cell to f^(1) on chip (Eq. (fnewstage), J = 1), so no f^(1) array
// passes through HBM and f^n is never recovered from a rounded f^(1).
//
// FP32 arithmetic runs on packed pairs (fma.rn.f32x2): the two members of a pair share every
// geometric factor, so the face-value and flux updates are one packed FMA per pair.

// Shape of the items: IT cells at most, NT threads, and the shared-memory capacities: ecap rows
// (item, ring-1, ring-2 and ghost rows), hs halo slots in the fixed-stride table (twice that
// with the overflow table), ccap cut faces.  Items that exceed one are split.
template <int IT>
struct FvShape;
template <>
struct FvShape<256> {
    static constexpr int nt = 256, ecap = 448, hs = 192, ccap = 192;
};
template <>
struct FvShape<64> {
    static constexpr int nt = 128, ecap = 224, hs = 128, ccap = 160;
};

// (an instance is a whole number of blocks: no item straddles two)
static_assert(kBlock % 256 == 0 && kBlock % 64 == 0, "FvShape sizes");

// Staged rows and value rows are named by the address of their first 16 bytes (float; doubles:
// twice that), so that a gather takes one mask: a row address is the byte offset of half 0 of the
// row within sf (half 1 is at that offset with bit 4 flipped), see fv_row_addr.
// Adjacency word (4 per cell): bits 4-13 the row address of the face datum (neighbour, ghost, or
// the cell itself where it has no such face); for a neighbour also bits 14-24 the value row that
// holds its outgoing values at this face and bits 25-28 the outgoing bits (bit 25 + p set when the
// first member of pair p leaves this cell here).  Bit 31: no neighbour (boundary face or no
// face); bit 30: no face.
constexpr unsigned kFvBnd = 0x80000000u, kFvNone = 0xC0000000u;
constexpr unsigned kFvRowMask = 0x3FF0u, kFvValMask = 0x7FF0u;
constexpr int kFvValShift = 10, kFvOutBit = 25;
__host__ __device__ constexpr unsigned fv_row_addr(int j) {  // halves swapped where bit 2 of j is set
    return 32u * static_cast<unsigned>(j) + ((j & 4) ? 16u : 0u);
}

// Geometry values of a cell.  Double: A_mk at 4 m + k, then (n dl / A)_m, x and y, at 16 + 2 m; a
// triangle has no slot 3 and keeps the six normal components in the free places 3, 7, 11-14, so
// that only 16 values are read.  Float: node positions relative to the centroid (8 values; face
// m joins nodes m and m + 1), then the least-squares weights W_m; explicit Euler: the face offsets
// r_m in place of the node positions (see k_fused_fv).  Stored in 16-byte chunks,
// chunk c of 32 consecutive cells together, so that a warp's load of one chunk is contiguous
// (a row per cell took 16 to 24 cache-line accesses a load, up to two fifths of all accesses to
// L1 and shared memory).
template <class T>
constexpr int kFvGeo = sizeof(T) == 4 ? 16 : 24;
template <class T>
__host__ __device__ constexpr size_t fv_geo_at(size_t i, int v) {  // value v of cell i
    constexpr int per = 16 / sizeof(T);
    return (((i >> 5) * (kFvGeo<T> / per) + v / per) * 32 + (i & 31)) * per + v % per;
}
// Coefficients of a cut face.  Double: A_mk of its face, k = 0..3.  Float: the ring cell's W_k (8
// values), then the offset r_m of the face (2 values, 2 unused).
template <class T>
constexpr int kFvCut = sizeof(T) == 4 ? 12 : 4;

// The item tables are laid out so that a CTA can issue its first loads -- the item's halo ids
// and its header -- together, from its item index alone: the halo ids sit at a fixed stride per
// item, and the header carries what the later steps need.  Staging then waits on two memory
// round trips (ids, then the rows they name) instead of three.
struct FvItems {
    const int4 *__restrict__ hdr;       // [2 nitem]: {base cell, cells | cuts << 16, instance,
                                        // overflow offset (-1: none)}, {halo cells, ghosts, first
                                        // ghost, first cut}
    const int *__restrict__ halo;       // [nitem][hs] global ids, ring 1 then ring 2, -1 after
    const int *__restrict__ ovf;        // halo slots hs.. of the items that have them
    const uint4 *__restrict__ adj;      // [np] adjacency words of every cell (within its item)
    const uint2 *__restrict__ cut;      // cut faces: row addresses / 16 of the ring cell and its face
                                        // data, 10 bits each: i, k0, k1; k2, k3, then the outgoing bits
    const int4 *__restrict__ ghost;     // ghosts: owner row, boundary face, owner cell, face slot
    int *__restrict__ err;              // set to 1 if the bulk-copy wait gave up
    long long wait_first;               // polls of that wait (fvlbm_set_wait_limit)
    int *__restrict__ cur;              // explicit Euler: takes next, the number of the buffer that
    int next;                           // f^{n+1} goes to (see k_pack_cells)
};

// Pair p: first members alpha = 1, 2, 5, 6 and their opposites 3, 4, 7, 8.
__host__ __device__ constexpr int fv_first(int p) { return p == 0 ? 1 : (p == 1 ? 2 : (p == 2 ? 5 : 6)); }
__host__ __device__ constexpr int fv_second(int p) { return p == 0 ? 3 : (p == 1 ? 4 : (p == 2 ? 7 : 8)); }
// Position of alpha (1..8) in a pair-ordered row of 8: (1,3)(2,4)(5,7)(6,8).
__host__ __device__ constexpr int fv_pos(int a) {
    return a == 1 ? 0 : (a == 3 ? 1 : (a == 2 ? 2 : (a == 4 ? 3 : (a == 5 ? 4 : (a == 7 ? 5 : (a == 6 ? 6 : 7))))));
}

// e_first(p) . (x, y)
template <class T>
__device__ __forceinline__ T fv_en(int p, T x, T y) {
    return p == 0 ? x : (p == 1 ? y : (p == 2 ? x + y : y - x));
}

// A pair of values (first member, opposite member) with packed FP32 arithmetic where available.
template <class T>
struct FvPair;
template <>
struct FvPair<float> {
    using V = float2;
    static __device__ __forceinline__ V make(float a, float b) { return make_float2(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ V bcast(float a) { return make_float2(a, a); }
};
template <>
struct FvPair<double> {
    using V = double2;
    static __device__ __forceinline__ V make(double a, double b) { return make_double2(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) {
        return make_double2(::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y));
    }
    static __device__ __forceinline__ V bcast(double a) { return make_double2(a, a); }
};

// Shared-memory layout (bytes):
//   sf  [ecap][8]      staged f (moving directions, pair order, halves swapped on bit 2 of the
//                      row): item rows, halo rows, ghost rows
//   sf0 [ecap]         staged f_0
//   sv  [4 IT + ccap][4]  value rows: the outgoing face values of face slot m of item cell c in
//                      row 4 c + (m ^ ((c >> 1) & 3)) (swizzled: the 32 rows that a warp
//                      writes at once spread over the banks), then one row per cut face
//   sacc [19][IT]      the item's rows for the stage algebra, structure of arrays: stage 1
//                      f^n and (formed on chip) f^n + dt Gamma^c(1) / 3; stage 2 B and C;
//                      stage 3 C (alpha = 1..8 of C: C_0 = 0, e_0 carries no flux); row 18 tau
//   the item's instance parameters (copied during staging, read by the stage algebra)
//   one mbarrier for the bulk copies
// In float three CTAs of 256 (24 warps, 80 registers, 55 KB each) share an SM; four at 64
// registers, which would fit the shared memory, spill 12 words and ran slower (sweep step 576
// against 509 us), as did two (588).
template <class T, int IT>
struct FvSmem {
    using S = FvShape<IT>;
    static constexpr size_t sf = 0;
    static constexpr size_t sf0 = sf + size_t(S::ecap) * 8 * sizeof(T);
    static constexpr size_t sv = sf0 + size_t(S::ecap) * sizeof(T);
    static constexpr size_t sacc = sv + size_t(4 * IT + S::ccap) * 4 * sizeof(T);
    static constexpr size_t ip = sacc + size_t(2 * kQ + 1) * IT * sizeof(T);
    static constexpr size_t bar = ip + sizeof(InstParam);
    static constexpr size_t bytes = bar + 16;
    static_assert(S::ecap % 8 == 0 && S::ecap <= 512 && 4 * IT + S::ccap <= 2048 && S::hs <= S::nt,
                  "whole groups of swapped rows, 10-bit row and 11-bit value addresses, one halo slot per thread");
};

// Rows of 8 (staged in shared memory, and the cell-major stage values in global memory) keep
// their two 4-value halves swapped when bit 2 of the row index is set: consecutive rows then
// spread over all banks, and since items start at multiples of 64 cells the item rows keep
// the same bit in both places (one bulk copy moves them unchanged).
__host__ __device__ __forceinline__ int fv_half(int j, int h) { return h ^ ((j >> 2) & 1); }

// Load the 8 moving directions of staged row j as 4 pairs.
template <class T>
__device__ __forceinline__ void fv_load_row(const T *sf, int j, typename FvPair<T>::V *o) {
    using PV = FvPair<T>;
    const T *lo_p = sf + j * 8 + 4 * fv_half(j, 0);
    const T *hi_p = sf + j * 8 + 4 * fv_half(j, 1);
    if constexpr (sizeof(T) == 4) {
        const float4 lo = *reinterpret_cast<const float4 *>(lo_p);
        const float4 hi = *reinterpret_cast<const float4 *>(hi_p);
        o[0] = PV::make(lo.x, lo.y);
        o[1] = PV::make(lo.z, lo.w);
        o[2] = PV::make(hi.x, hi.y);
        o[3] = PV::make(hi.z, hi.w);
    } else {
        o[0] = *reinterpret_cast<const double2 *>(lo_p);
        o[1] = *reinterpret_cast<const double2 *>(lo_p + 2);
        o[2] = *reinterpret_cast<const double2 *>(hi_p);
        o[3] = *reinterpret_cast<const double2 *>(hi_p + 2);
    }
}
// element offset of alpha (1..8) in row j
__device__ __forceinline__ int fv_alpha_off(int j, int a) {
    const int pos = fv_pos(a);
    return j * 8 + 4 * fv_half(j, pos >> 2) + (pos & 3);
}

// Half h of staged row j: pairs 2 h and 2 h + 1 (16 bytes in float).
template <class T>
__device__ __forceinline__ void fv_load_half(const T *sf, int j, int h, typename FvPair<T>::V *o) {
    using PV = FvPair<T>;
    const T *p = sf + j * 8 + 4 * fv_half(j, h);
    if constexpr (sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        o[0] = PV::make(x.x, x.y);
        o[1] = PV::make(x.z, x.w);
    } else {
        o[0] = *reinterpret_cast<const double2 *>(p);
        o[1] = *reinterpret_cast<const double2 *>(p + 2);
    }
}

// The same of the row at address a (fv_row_addr).
template <class T>
__device__ __forceinline__ void fv_load_half_at(const T *sf, unsigned a, int h, typename FvPair<T>::V *o) {
    using PV = FvPair<T>;
    const unsigned char *p = reinterpret_cast<const unsigned char *>(sf) + (sizeof(T) / 4) * (a ^ (16u * h));
    if constexpr (sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        o[0] = PV::make(x.x, x.y);
        o[1] = PV::make(x.z, x.w);
    } else {
        o[0] = reinterpret_cast<const double2 *>(p)[0];
        o[1] = reinterpret_cast<const double2 *>(p)[1];
    }
}

template <class T>
__device__ __forceinline__ void fv_store_row(T *sf, int j, const typename FvPair<T>::V *f) {
    T *lo = sf + j * 8 + 4 * fv_half(j, 0), *hi = sf + j * 8 + 4 * fv_half(j, 1);
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(lo) = make_float4(f[0].x, f[0].y, f[1].x, f[1].y);
        *reinterpret_cast<float4 *>(hi) = make_float4(f[2].x, f[2].y, f[3].x, f[3].y);
    } else {
        *reinterpret_cast<double2 *>(lo) = f[0];
        *reinterpret_cast<double2 *>(lo + 2) = f[1];
        *reinterpret_cast<double2 *>(hi) = f[2];
        *reinterpret_cast<double2 *>(hi + 2) = f[3];
    }
}

// Four consecutive values at a 16-byte (float) or 32-byte (double) aligned address.
template <class T>
__device__ __forceinline__ void fv_load4(const T *p, T *v) {
    if constexpr (sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4 *>(p);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
        const double2 a = *reinterpret_cast<const double2 *>(p);
        const double2 b = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
}
// Geometry values v .. v + 3 of cell i (v a multiple of 4)
template <class T>
__device__ __forceinline__ void fv_load_geo4(const T *__restrict__ geo, int i, int v, T *o) {
    if constexpr (sizeof(T) == 4) {
        fv_load4(geo + fv_geo_at<T>(i, v), o);
    } else {
        const double2 a = *reinterpret_cast<const double2 *>(geo + fv_geo_at<T>(i, v));
        const double2 b = *reinterpret_cast<const double2 *>(geo + fv_geo_at<T>(i, v + 2));
        o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
    }
}
template <class T>
__device__ __forceinline__ void fv_store4(T *p, T a, T b, T c, T d) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
    } else {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(c, d);
    }
}

// Store of a stage value f^(2) or f^(3) of cell i as a cell-major row: alpha = 1..8 in pair order
// at f[8 i] (the two halves swapped where bit 2 of i is set), f_0 at f[8 np + i].
template <class T>
__device__ __forceinline__ void fv_store_stage(T *__restrict__ f, size_t np, int i, T f0,
                                               const typename FvPair<T>::V *o) {
    T *row = f + 8 * static_cast<size_t>(i);
    fv_store4(row + 4 * fv_half(i, 0), o[0].x, o[0].y, o[1].x, o[1].y);
    fv_store4(row + 4 * fv_half(i, 1), o[2].x, o[2].y, o[3].x, o[3].y);
    f[8 * np + i] = f0;
}

// ---- float: the direction-by-direction algebra that the two-pass kernels share
// Stage 1: f^(1) = [f^n + (dt/tau)/4 f^eq(f^n)] / (1 + (dt/tau)/4) (Eq. (fnewstage), J = 1)
// of a cell given as f[9] (alpha order), written to staged row e.
__device__ __forceinline__ void fv_relax_to_row(float *f, float *sf, float *sf0, int e, float rho0, float dt,
                                                float tau_e, float *eq_out = nullptr) {
    relax9(f, rho0, dt, tau_e, eq_out);
    sf0[e] = f[0];
    fv_store4(sf + e * 8 + 4 * fv_half(e, 0), f[1], f[3], f[2], f[4]);
    fv_store4(sf + e * 8 + 4 * fv_half(e, 1), f[5], f[7], f[6], f[8]);
}

// End node of face m of a cell (m compile-time): node m + 1, wrapping to node 0 after the last
// face; selects between static indices keep q in registers.
#define FV_END_X(m) ((m) == 3 ? q[0] : ((m) == 2 && tri ? q[0] : q[2 * (m) + 2]))
#define FV_END_Y(m) ((m) == 3 ? q[1] : ((m) == 2 && tri ? q[1] : q[2 * (m) + 3]))

// Gradient (Step 2) and outgoing face values of item cell c, two pairs at a time (packed FMAs).
// g: node positions q relative to the centroid (OFF: the face offsets r_m), then least-squares
// weights W_m (x, y per face slot); w: adjacency.
// Absent faces have weight 0 and the cell itself as datum, and values at faces without a neighbour
// are formed but not read, so the only branch is the warp's on the fourth slot (quads).
template <bool OFF>
__device__ __forceinline__ void fv_cell(int c, const float *g, const unsigned *w, bool quads,
                                        const float *__restrict__ sf, float *__restrict__ sv) {
    using PV = FvPair<float>;
    using V = PV::V;
    const float *q = g, *lw = g + 8;
    const bool tri = w[3] >= kFvNone;
    const V mone = PV::bcast(-1.f);
    const unsigned own = fv_row_addr(c);
    float o[4][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        V fc[2], gx[2], gy[2];
        fv_load_half_at(sf, own, h, fc);
        gx[0] = gx[1] = gy[0] = gy[1] = PV::bcast(0.f);
        auto datum = [&](int k) {
            V fk[2];
            fv_load_half_at(sf, w[k] & kFvRowMask, h, fk);
            const V wx = PV::bcast(lw[2 * k]), wy = PV::bcast(lw[2 * k + 1]);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const V df = PV::fma(fc[s], mone, fk[s]);  // f_k - f_c, one rounding
                gx[s] = PV::fma(wx, df, gx[s]);
                gy[s] = PV::fma(wy, df, gy[s]);
            }
        };
        auto face = [&](int m) {
            const V rx = PV::bcast(OFF ? q[2 * m] : 0.5f * (q[2 * m] + FV_END_X(m)));
            const V ry = PV::bcast(OFF ? q[2 * m + 1] : 0.5f * (q[2 * m + 1] + FV_END_Y(m)));
            float out[2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const V val = PV::fma(gy[s], ry, PV::fma(gx[s], rx, fc[s]));
                out[s] = (w[m] & (1u << (kFvOutBit + 2 * h + s))) ? val.x : val.y;
            }
            if (h == 0) {
                o[m][0] = out[0];
                o[m][1] = out[1];
            } else {
                fv_store4(sv + 4 * (4 * c + (m ^ ((c >> 1) & 3))), o[m][0], o[m][1], out[0], out[1]);
            }
        };
        datum(0);
        datum(1);
        datum(2);
        if (quads) datum(3);
        face(0);
        face(1);
        face(2);
        if (quads) face(3);
    }
}

// n dl / A of every face of a cell from its node positions.
__device__ __forceinline__ void fv_normals(const float *q, bool tri, float *sn) {
    float a2x = 0.f;  // twice the area (shoelace on centroid-relative nodes)
#pragma unroll
    for (int m = 0; m < 4; ++m)
        if (m < 3 || !tri) a2x += q[2 * m] * FV_END_Y(m) - FV_END_X(m) * q[2 * m + 1];
    const float inv_a = a2x > 0.f ? sdiv(2.f, a2x) : 0.f;  // padding cells have no faces
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const float x1 = FV_END_X(m), y1 = FV_END_Y(m);
        sn[2 * m] = (y1 - q[2 * m + 1]) * inv_a;
        sn[2 * m + 1] = -(x1 - q[2 * m]) * inv_a;
    }
}
#undef FV_END_X
#undef FV_END_Y

// ---- double: the cell algebra on pairs.  With S = f + f-bar and D = f - f-bar of a pair the moments
// are plain sums, and f^eq of a pair is w (s + a), w (s - a) with the parts even and odd in u:
// about half the operations of the direction-by-direction form, which counts in double, where
// every operation takes 64 times a float one on this GPU.  Products that are added are written as
// fused operations, so that every kernel that uses these functions rounds alike.
template <class T>
struct FvMoments {
    T dr, r, u, v, jx, jy, uu;  // uu = 1.5 (u^2 + v^2)
};
template <class T>
__device__ __forceinline__ void fv_velocity(FvMoments<T> &M, T rho0) {
    M.r = rho0 + M.dr;
    const T ir = sdiv(T(1), M.r);
    M.u = M.jx * ir;
    M.v = M.jy * ir;
    M.uu = T(1.5) * fma(M.u, M.u, M.v * M.v);
}
template <class T>
__device__ __forceinline__ FvMoments<T> fv_moments(const typename FvPair<T>::V *f, T f0, T rho0) {
    FvMoments<T> M;
    const T d2 = f[2].x - f[2].y, d3 = f[3].x - f[3].y;
    M.dr = f0 + (((f[0].x + f[0].y) + (f[1].x + f[1].y)) + ((f[2].x + f[2].y) + (f[3].x + f[3].y)));
    M.jx = (f[0].x - f[0].y) + (d2 - d3);
    M.jy = (f[1].x - f[1].y) + (d2 + d3);
    fv_velocity(M, rho0);
    return M;
}
template <class T>
__device__ __forceinline__ T fv_w(int p) {
    return p < 2 ? T(1.0 / 9.0) : T(1.0 / 36.0);
}
// f^eq - w rho0 of pair p, and of the rest direction
template <class T>
__device__ __forceinline__ typename FvPair<T>::V fv_feq(const FvMoments<T> &M, int p) {
    const T eu = fv_en<T>(p, M.u, M.v);
    const T s = fv_w<T>(p) * fma(M.r, fma(T(4.5) * eu, eu, -M.uu), M.dr);
    const T ej = fv_en<T>(p, M.jx, M.jy), w3 = p < 2 ? T(1.0 / 3.0) : T(1.0 / 12.0);
    return FvPair<T>::make(fma(w3, ej, s), fma(-w3, ej, s));
}
template <class T>
__device__ __forceinline__ T fv_feq0(const FvMoments<T> &M) {
    return T(4.0 / 9.0) * fma(-M.r, M.uu, M.dr);
}

// Relaxation factors of an implicit collision with coefficient m: f = f^eq + a (X - f^eq) with
// a = 1 / (1 + m dt / tau), and g = (dt / tau) a, so that dt Gamma^c = -g (X - f^eq); one
// division.  In this form rounding of a leaves the conserved moments alone.
template <class T>
__device__ __forceinline__ void fv_factors(T dt, T tau, T m, T &a, T &g) {
    const T r = sdiv(T(1), fma(m, dt, tau));
    a = tau * r;
    g = dt * r;
}

// Pair p of the boundary values f_{alpha,bc} (boundary_values, which states the readings) of a cell
// with that pair f and moments M, as differences to the cell's own values: wall and inlet
// f + f^eq(rho, u_b) - f^eq(rho, u), outlet f + f^eq(rho_b, u) - f^eq(rho, u), far field
// f^eq(rho_b, u_b) where e . n < 0.
__device__ __forceinline__ double2 fv_ghost_pair(int type, double rb, double ub, double vb, double nx, double ny,
                                                 const FvMoments<double> &M, double rho0, int p, double2 f) {
    if (type == FVLBM_BC_FARFIELD) {
        FvMoments<double> B;
        B.dr = rb - rho0;
        B.r = rb;
        B.u = ub;
        B.v = vb;
        B.jx = rb * ub;
        B.jy = rb * vb;
        B.uu = 1.5 * ::fma(ub, ub, vb * vb);
        const double en = fv_en<double>(p, nx, ny);
        const double2 eq = fv_feq<double>(B, p);
        return make_double2(en < 0.0 ? eq.x : f.x, en > 0.0 ? eq.y : f.y);
    }
    double s, a;
    if (type == FVLBM_BC_OUTLET) {
        const double q = (rb - rho0) - M.dr;  // rho_b - rho
        const double eu = fv_en<double>(p, M.u, M.v);
        s = ::fma(q, ::fma(4.5 * eu, eu, -M.uu), q);
        a = 3.0 * q * eu;
    } else {
        const double du = ub - M.u, dv = vb - M.v, su = ub + M.u, sv = vb + M.v;
        const double de = fv_en<double>(p, du, dv);
        s = M.r * ::fma(4.5 * de, fv_en<double>(p, su, sv), -(1.5 * ::fma(du, su, dv * sv)));
        a = 3.0 * M.r * de;
    }
    const double w = fv_w<double>(p);
    return make_double2(::fma(w, s + a, f.x), ::fma(w, s - a, f.y));
}

// Boundary values of a cell with staged row fc, f0 at ghost gh.  The face's type and values are read
// kept in L2, like the item tables: a few hundred kB read once per launch by the items along the
// boundaries.  OFF: as in fv_cell.
template <class T, bool OFF>
__device__ __forceinline__ void fv_ghost(const Geo<T> &G, const T *__restrict__ bnrm, const T *__restrict__ geo,
                                         const int4 &gh, T rho0, const typename FvPair<T>::V *fc, T f0,
                                         typename FvPair<T>::V *out) {
    using PV = FvPair<T>;
    const unsigned long long keep = l2_keep_policy();
    const int bf = gh.y;
    const int type = ld_keep(G.btype + bf, keep);
    if constexpr (sizeof(T) == 4) {  // boundary_values itself, the far field's normal as the flux has it
        T bval[3], fcs[kQ], fb[kQ], dr, r, u, v, nx = T(0), ny = T(0);
#pragma unroll
        for (int c = 0; c < 3; ++c) bval[c] = ld_keep(G.bval + static_cast<size_t>(c) * G.nbt + bf, keep);
        if (type == FVLBM_BC_FARFIELD && OFF) {
            nx = G.sn[static_cast<size_t>(2 * gh.w) * G.np + gh.z];
            ny = G.sn[static_cast<size_t>(2 * gh.w + 1) * G.np + gh.z];
        } else if (type == FVLBM_BC_FARFIELD) {
            const bool tri = G.nbr[3 * static_cast<size_t>(G.np) + gh.z] == kNone;
            const int m = gh.w, e = m == 3 || (m == 2 && tri) ? 0 : m + 1;
            nx = geo[fv_geo_at<T>(gh.z, 2 * e + 1)] - geo[fv_geo_at<T>(gh.z, 2 * m + 1)];
            ny = -(geo[fv_geo_at<T>(gh.z, 2 * e)] - geo[fv_geo_at<T>(gh.z, 2 * m)]);
        }
        fcs[0] = f0;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            fcs[fv_first(p)] = fc[p].x;
            fcs[fv_second(p)] = fc[p].y;
        }
        moments(fcs, rho0, dr, r, u, v);
        boundary_values(type, bval, 0, 1, nx, ny, fcs, dr, r, u, v, rho0, fb);
#pragma unroll
        for (int p = 0; p < 4; ++p) out[p] = PV::make(fb[fv_first(p)], fb[fv_second(p)]);
        return;
    }
    if constexpr (sizeof(T) == 8) {
        const T rb = ld_keep(G.bval + bf, keep), ub = ld_keep(G.bval + G.nbt + bf, keep),
                vb = ld_keep(G.bval + 2 * static_cast<size_t>(G.nbt) + bf, keep);
        const T nx = ld_keep(bnrm + bf, keep), ny = ld_keep(bnrm + G.nbt + bf, keep);
        const FvMoments<T> M = fv_moments<T>(fc, f0, rho0);
#pragma unroll
        for (int p = 0; p < 4; ++p) out[p] = fv_ghost_pair(type, rb, ub, vb, nx, ny, M, rho0, p, fc[p]);
    }
}

// Outgoing face values of item cell c at its interior faces: f_c + sum_k A_mk (f_k - f_c), A at
// a[4 m + k]; of each pair the outgoing member is taken first (selects cost nothing beside the
// arithmetic).  A value is the same chain of fused multiply-adds as in fv_cut.
__device__ __forceinline__ void fv_cell(int c, const double *a, const unsigned *w, bool quads,
                                        const double *__restrict__ sf, double *__restrict__ sv) {
    using PV = FvPair<double>;
    const unsigned own = fv_row_addr(c);
    const bool four = w[3] < kFvNone;  // (per cell: an operation saved counts here)
    double o[4][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        PV::V fc[2], d[4][2];
        fv_load_half_at(sf, own, h, fc);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k == 3 && !four) continue;
            fv_load_half_at(sf, w[k] & kFvRowMask, h, d[k]);
#pragma unroll
            for (int q = 0; q < 2; ++q) d[k][q] = PV::make(d[k][q].x - fc[q].x, d[k][q].y - fc[q].y);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (w[m] & kFvBnd) continue;  // no neighbour
            double out[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const bool first = w[m] & (1u << (kFvOutBit + 2 * h + q));
                double v = first ? fc[q].x : fc[q].y;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k < 3 || four) v = ::fma(a[4 * m + k], first ? d[k][q].x : d[k][q].y, v);
                out[q] = v;
            }
            if (h == 0) {
                o[m][0] = out[0];
                o[m][1] = out[1];
            } else {
                fv_store4(sv + 4 * (4 * c + (m ^ ((c >> 1) & 3))), o[m][0], o[m][1], out[0], out[1]);
            }
        }
    }
}

// Half h (two direction pairs) of the outgoing face values of a cut face: the ring cell's values
// at the face it shares with the item (absent face data: its own row with coefficient 0).
template <class T>
__device__ __forceinline__ void fv_cut(T *__restrict__ dst, int h, uint2 r, const T *a, const T *__restrict__ sf) {
    using PV = FvPair<T>;
    using V = typename PV::V;
    const unsigned row[5] = {(r.x << 4) & kFvRowMask, (r.x >> 6) & kFvRowMask, (r.x >> 16) & kFvRowMask,
                             (r.y << 4) & kFvRowMask, (r.y >> 6) & kFvRowMask};
    const bool b0 = r.y & (1u << (20 + 2 * h)), b1 = r.y & (2u << (20 + 2 * h));
    auto member = [&](unsigned a) {
        V f[2];
        fv_load_half_at(sf, a, h, f);
        return PV::make(b0 ? f[0].x : f[0].y, b1 ? f[1].x : f[1].y);
    };
    const V c = member(row[0]);
    const V mone = PV::bcast(T(-1));
    V v;
    if constexpr (sizeof(T) == 4) {
        V gx = PV::bcast(T(0)), gy = PV::bcast(T(0));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const V df = PV::fma(c, mone, member(row[1 + k]));
            gx = PV::fma(PV::bcast(a[2 * k]), df, gx);
            gy = PV::fma(PV::bcast(a[2 * k + 1]), df, gy);
        }
        v = PV::fma(gy, PV::bcast(a[9]), PV::fma(gx, PV::bcast(a[8]), c));
    } else {
        v = c;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const V f = member(row[1 + k]);
            v = PV::fma(PV::bcast(a[k]), PV::make(f.x - c.x, f.y - c.y), v);
        }
    }
    *reinterpret_cast<V *>(dst + 2 * h) = v;
}

// Convection term of item cell t (Eq. (advection)): per face its own outgoing values and the
// neighbour's (its incoming ones), both from the value rows, or the ghost row of a boundary face.
// ac = sum_m (e_alpha . n_m dl_m / A) f_{alpha,bc,m} (= -Gamma^a), in pairs.
template <class T>
__device__ __forceinline__ void fv_flux(int t, const T *sn, const unsigned *w, const T *__restrict__ sf,
                                        const T *__restrict__ sv, typename FvPair<T>::V *ac) {
    using PV = FvPair<T>;
    using V = typename PV::V;
#pragma unroll
    for (int p = 0; p < 4; ++p) ac[p] = PV::bcast(T(0));
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (w[m] >= kFvNone) continue;
        V val[4];
        if (w[m] & kFvBnd) {
            fv_load_half_at(sf, w[m] & kFvRowMask, 0, val);
            fv_load_half_at(sf, w[m] & kFvRowMask, 1, val + 2);
        } else {
            T vo[4], vn[4];
            fv_load4(sv + 4 * (4 * t + (m ^ ((t >> 1) & 3))), vo);
            fv_load4(reinterpret_cast<const T *>(reinterpret_cast<const unsigned char *>(sv) +
                                                 (sizeof(T) / 4) * ((w[m] >> kFvValShift) & kFvValMask)),
                     vn);
#pragma unroll
            for (int p = 0; p < 4; ++p)
                val[p] = (w[m] & (1u << (kFvOutBit + p))) ? PV::make(vo[p], vn[p]) : PV::make(vn[p], vo[p]);
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const T en = fv_en<T>(p, sn[2 * m], sn[2 * m + 1]);
            ac[p] = PV::fma(PV::make(en, -en), val[p], ac[p]);
        }
    }
}

// Accumulator alpha of cell i.
template <int IT>
__host__ __device__ constexpr size_t fv_acc_at(size_t i, int alpha) {
    return (i / IT * kQ + alpha) * IT + i % IT;
}

// One IMEX stage (see fvlbm_kernels.cu's stage_algebra for what STAGE computes) in the
// face-value form, one CTA per work item.  fin: stage 1 f^n (structure of arrays), stages 2, 3
// f^(2), f^(3) (cell-major rows); fs_out: stages 1, 2 write f^(2), f^(3) cell-major; fn: stage 3
// writes f^{n+1}; geo: the geometry rows, cutc: the cut faces' coefficients.  STAGE 4 is the explicit
// Euler step: fin f^n, fs_out f^{n+1} (structure of arrays, another buffer: neighbours read f^n).
//
// Geometry of the float Euler step: offsets and normals formed in FP64 on the host and rounded once, as
// the two-pass kernels read them.  Formed in float from the nodes, the area of a slim rotated cell
// cancels: on quads of aspect 1000 the largest error of f against FP64 was 6.2e-7 after 8 steps, 1.0e-7
// now, which is what the two-pass kernels have (f comes out the same).  The normals are loaded
// before the barrier, not with the other geometry: eight registers more would leave four 64-cell CTAs to
// an SM instead of five.  40k-cell cavity: 5.0 us a step either way.
//
// What bounds it.  Float: the chain inside a CTA (ids, rows, face values, barrier, flux, algebra)
// at 24 warps an SM, neither memory nor issue alone.  A 2.57M-cell batch takes 145 + 119 + 109 us
// for the stages (2.9, 4.3 and 3.3 TB/s of state words; 47 % of the issue slots in stage 1), 217 +
// 174 + 156 before cut faces, ghost rows and byte addresses took the warp instructions of 640k cells
// from 27.5 / 23.5 / 19.9 M to 21.6 / 16.2 / 13.4 M.  Double: the FP64 pipe, 84 to 87 % busy (one warp
// instruction holds a scheduler for 64 cycles, compares and conversions too), so operations are
// what is saved: 640k cells, 475 + 292 + 223 us.
template <class T, int STAGE, bool STATS, int IT>
__global__ void __launch_bounds__(FvShape<IT>::nt, sizeof(T) == 4 ? (IT == 256 ? 3 : 1) : (IT == 256 ? 2 : 1))
    k_fused_fv(const T *fin, T *__restrict__ fs_out, T *__restrict__ fn, T *Bacc, T *Cacc, const T *tau, T *mac, double *__restrict__ partial, Geo<T> G, FvItems W,
               const T *__restrict__ geo, const T *__restrict__ cutc, const T *__restrict__ bnrm) {
    using PV = FvPair<T>;
    using V = typename PV::V;
    using S = FvShape<IT>;
    using L = FvSmem<T, IT>;
    constexpr int NT = S::nt, HS = S::hs;
    constexpr bool SOA = STAGE == 1 || STAGE == 4;  // reads f^n
    constexpr bool OFF = STAGE == 4 && sizeof(T) == 4;  // r_m and normals as formed in FP64 on the host
    extern __shared__ __align__(128) unsigned char smem_raw[];
    T *sf = reinterpret_cast<T *>(smem_raw + L::sf);
    T *sf0 = reinterpret_cast<T *>(smem_raw + L::sf0);
    T *sv = reinterpret_cast<T *>(smem_raw + L::sv);
    T *sacc = reinterpret_cast<T *>(smem_raw + L::sacc);
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(smem_raw + L::bar);

    const int t = threadIdx.x;
    // Stage 2 walks the items backwards: what stage 1 wrote last (100 MB or so of a large batch) it
    // finds in L2, and stage 3 what stage 2 wrote last (sweep step 502 -> 494 us).
    const int it = static_cast<int>(STAGE == 2 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
    // halo slot t of the fixed-stride table and the header, loaded together (kept in L2)
    const unsigned long long keep = l2_keep_policy();
    const int gid0 = t < HS ? ld_keep(W.halo + static_cast<size_t>(it) * HS + t, keep) : -1;
    const int4 hd = ld_keep(W.hdr + 2 * it, keep), hx = ld_keep(W.hdr + 2 * it + 1, keep);
    const int base = hd.x, cnt = hd.y & 0xFFFF, ncut = hd.y >> 16;
    // slot HS + t, in the overflow table (items with a large halo only)
    const int gid1 = hd.w >= 0 && t < HS ? ld_keep(W.ovf + hd.w + t, keep) : -1;
    const size_t np = G.np;
    const InstParam *__restrict__ Pp = G.ip + hd.z;  // read where used
    const T rho0 = ipv<T>(Pp->rho0, Pp->rho0_f);
    const bool mine = t < cnt;
    const int i = base + t;
    const T *fa0 = fin + 8 * np;  // stages 2, 3: f_0 of every cell after the cell-major rows

    // 1. staging, issued before any wait: first what is fixed at create, beside the last blocks of
    // the kernel before; then the copies.
    // The bulk copies are shared out over the lanes 0 of the warps, so that no warp issues
    // more than a few of them: each such lane arrives on the mbarrier (count: the warps) with the
    // bytes of its own copies, then issues them.
    constexpr int kWarps = NT / 32;
    if (t == 0) mbar_init(bar, kWarps);
    __syncthreads();
    static_assert(sizeof(InstParam) % 16 == 0 && L::ip % 16 == 0, "16-byte copies of the parameters");
    if (t < static_cast<int>(sizeof(InstParam) / 16))  // (device arrays of InstParam: 16-byte aligned rows)
        cp_async<16>(smem_raw + L::ip + 16 * t, reinterpret_cast<const unsigned char *>(Pp) + 16 * t);
    // the item cell's adjacency and coefficients, the thread's first cut face and ghost
    unsigned w[4] = {kFvNone, kFvNone, kFvNone, kFvNone};
    T A[16];
    if (mine) {
        const uint4 w4 = W.adj[i];
        w[0] = w4.x; w[1] = w4.y; w[2] = w4.z; w[3] = w4.w;
#pragma unroll
        for (int k = 0; k < 16; k += 4) fv_load_geo4(geo, i, k, A + k);
    }
    // cut units: (cut face, half), over the threads that hold no cell where there are any
    constexpr int CB = NT > IT ? IT : 0, CS = NT - CB;
    const int cu = t - CB;
    const bool cut0 = cu >= 0 && cu < 2 * ncut;
    uint2 cr = make_uint2(0, 0);
    T ca[kFvCut<T>];
    auto load_cut = [&](int c) {
        cr = W.cut[hx.w + c];
#pragma unroll
        for (int k = 0; k < kFvCut<T>; k += 4) fv_load4(cutc + kFvCut<T> * static_cast<size_t>(hx.w + c) + k, ca + k);
    };
    if (cut0) load_cut(cu >> 1);
    dep_wait();  // f, the accumulators and tau of the kernels before
    if (STAGE == 4 && blockIdx.x == 0 && t == 0) *W.cur = W.next;
    if ((t & 31) == 0) {
        const unsigned row = static_cast<unsigned>(cnt * sizeof(T));
        // copies: (stages 2, 3) the item's f rows and f_0, then the accumulator rows (stage 1:
        // f^n; stage 2: B, then C of alpha = 1..8; stage 3: C of alpha = 1..8), then tau; the rows of
        // a whole tile are one copy
        const bool whole = !SOA && cnt == IT;
        constexpr int nf = SOA ? 0 : 2;
        const int n1 = STAGE == 3 ? 0 : (whole ? 1 : kQ), n2 = SOA ? 0 : (whole ? 1 : kQ - 1);
        const int ncopy = nf + n1 + n2 + (STAGE == 3 ? 0 : 1);
        const int w = t >> 5;
        const size_t tile = fv_acc_at<IT>(base, 0);
        unsigned bytes = 0;
        for (int c = w; c < ncopy; c += kWarps)
            bytes += nf > 0 && c == 0 ? 8 * row
                                      : (whole && c >= nf && c < nf + n1 + n2 ? (c < nf + n1 ? kQ : kQ - 1) * row : row);
        mbar_expect_tx(bar, bytes);
        for (int c = w; c < ncopy; c += kWarps) {
            if (nf > 0 && c == 0) {
                bulk_g2s(sf, fin + 8 * static_cast<size_t>(base), 8 * row, bar);
            } else if (nf > 0 && c == 1) {
                bulk_g2s(sf0, fa0 + base, row, bar);
            } else if (c < nf + n1) {
                const int a = c - nf;
                if (SOA)
                    bulk_g2s(sacc + a * IT, fin + a * np + base, row, bar);
                else
                    bulk_g2s(sacc + a * IT, Bacc + tile + a * IT, whole ? kQ * row : row, bar);
            } else if (c < nf + n1 + n2) {
                const int a = c - nf - n1;  // C_{a + 1}
                bulk_g2s(sacc + ((STAGE == 3 ? 0 : kQ) + a) * IT, Cacc + tile + (a + 1) * IT,
                         whole ? (kQ - 1) * row : row, bar);
            } else {
                bulk_g2s(sacc + 2 * kQ * IT, tau + base, row, bar);
            }
        }
    }
    constexpr int per = 16 / sizeof(T);  // elements per 16-byte chunk
    T htau[2], hdt[2];
    const T dtg = ipv<T>(Pp->dt, Pp->dt_f);
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // halo cells (item rows come in bulk): slots t, HS + t
        const int gid = k == 0 ? gid0 : gid1;
        if (gid < 0) continue;
        const int e = cnt + t + k * HS;
        if (SOA) {  // f^n is structure of arrays: one element per direction
#pragma unroll
            for (int a = 1; a < kQ; ++a) cp_async<sizeof(T)>(sf + fv_alpha_off(e, a), fin + a * np + gid);
            cp_async<sizeof(T)>(sf0 + e, fin + gid);
            if (STAGE == 1) {
                htau[k] = tau[gid];
                hdt[k] = G.dtc != nullptr ? G.dtc[gid] : dtg;
            }
        } else {  // one cell-major row: half h sits at half fv_half(gid, h) there, fv_half(e, h) here
            const T *src = fin + 8 * static_cast<size_t>(gid);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 4 / per; ++q)
                    cp_async<16>(sf + e * 8 + 4 * fv_half(e, h) + q * per, src + 4 * fv_half(gid, h) + q * per);
            cp_async<sizeof(T)>(sf0 + e, fa0 + gid);
        }
    }
    cp_async_wait_all();
    // stage 1: each thread relaxes the halo cells it staged (its own copies have landed)
    if (STAGE == 1) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if ((k == 0 ? gid0 : gid1) < 0) continue;
            const int e = cnt + t + k * HS;
            V f[4];
            fv_load_row(sf, e, f);
            const T f0 = sf0[e];
            if constexpr (sizeof(T) == 4) {
                T fa[kQ];
                fa[0] = f0;
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    fa[fv_first(p)] = f[p].x;
                    fa[fv_second(p)] = f[p].y;
                }
                fv_relax_to_row(fa, sf, sf0, e, rho0, hdt[k], htau[k]);
                continue;
            }
            T a, g;
            const FvMoments<T> M = fv_moments<T>(f, f0, rho0);
            fv_factors(hdt[k], htau[k], T(0.25), a, g);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const V eq = fv_feq<T>(M, p);
                f[p] = PV::fma(PV::bcast(a), PV::make(f[p].x - eq.x, f[p].y - eq.y), eq);
            }
            const T eq0 = fv_feq0(M);
            sf0[e] = fma(a, f0 - eq0, eq0);
            fv_store_row(sf, e, f);
        }
    }
    {
        long long polls = 0;
        // (a limit of 0 gives up at once, without polling: the diagnostic of the error path)
        bool done = W.wait_first > 0 && mbar_try_wait(bar, 0);
        while (!done && ++polls < W.wait_first) done = mbar_try_wait(bar, 0);
        // the block leaves together if any thread gave up: flag it, wait once more (with the
        // full bound) for its own copies in flight, then return
        if (__syncthreads_or(!done)) {
            if (t == 0) atomicExch(W.err, 1);
            for (long long k = 0; k < kWaitLimit && !mbar_try_wait(bar, 0); ++k) {
            }
            return;
        }
    }
    // stage 1: the item cells' f^(1) from their f^n rows (in the accumulator copy); the rows after
    // them take f^n + dt Gamma^c(1) / 3, which the stage algebra adds to B
    const T dt_i = mine && G.dtc != nullptr ? G.dtc[i] : dtg;
    if (STAGE == 1) {
        if (sizeof(T) == 4) {
            if constexpr (sizeof(T) == 4) {
                if (mine) {  // the free rows take f^eq(f^n), which the stage-1 algebra reads
                    T f[kQ], eq[kQ];
#pragma unroll
                    for (int a = 0; a < kQ; ++a) f[a] = sacc[a * IT + t];
                    fv_relax_to_row(f, sf, sf0, t, rho0, dt_i, sacc[2 * kQ * IT + t], eq);
#pragma unroll
                    for (int a = 0; a < kQ; ++a) sacc[(kQ + a) * IT + t] = eq[a];
                }
            }
        } else if (mine) {
            V f[4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                f[p] = PV::make(sacc[fv_first(p) * IT + t], sacc[fv_second(p) * IT + t]);
            const T f0 = sacc[t];
            T a, g;
            const FvMoments<T> M = fv_moments<T>(f, f0, rho0);
            fv_factors(dt_i, sacc[2 * kQ * IT + t], T(0.25), a, g);
            g *= T(-1.0 / 3.0);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const V eq = fv_feq<T>(M, p);
                const V d = PV::make(f[p].x - eq.x, f[p].y - eq.y);
                const V b = PV::fma(PV::bcast(g), d, f[p]);
                sacc[(kQ + fv_first(p)) * IT + t] = b.x;
                sacc[(kQ + fv_second(p)) * IT + t] = b.y;
                f[p] = PV::fma(PV::bcast(a), d, eq);
            }
            const T eq0 = fv_feq0(M), d0 = f0 - eq0;
            sacc[kQ * IT + t] = fma(g, d0, f0);
            sf0[t] = fma(a, d0, eq0);
            fv_store_row(sf, t, f);
        }
        __syncthreads();
    }
    if (STAGE == 4) {  // the item's staged rows from its f^n rows
        if (mine) {
            V f[4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                f[p] = PV::make(sacc[fv_first(p) * IT + t], sacc[fv_second(p) * IT + t]);
            sf0[t] = sacc[t];
            fv_store_row(sf, t, f);
        }
        __syncthreads();
    }
    // ghost rows of the boundary faces (few items have any; the count is the block's)
    if (hx.y > 0) {
        for (int q = t; q < hx.y; q += NT) {
            const int4 gh = W.ghost[hx.z + q];
            V f[4], b[4];
            fv_load_row(sf, gh.x, f);
            fv_ghost<T, OFF>(G, bnrm, geo, gh, rho0, f, sf0[gh.x], b);
            fv_store_row(sf, cnt + hx.x + q, b);
        }
        __syncthreads();
    }

    // 2. outgoing face values: item cells (thread t takes cell t) and cut faces
    const bool quads = __any_sync(0xffffffffu, w[3] < kFvNone);  // (a triangle has no fourth face)
    if (mine) {
        if constexpr (sizeof(T) == 4)
            fv_cell<OFF>(t, A, w, quads, sf, sv);
        else
            fv_cell(t, A, w, quads, sf, sv);
    }
    if (cut0) fv_cut<T>(sv + 4 * (4 * IT + (cu >> 1)), cu & 1, cr, ca, sf);
    if (cu >= 0)
        for (int u = cu + CS; u < 2 * ncut; u += CS) {
            load_cut(u >> 1);
            fv_cut<T>(sv + 4 * (4 * IT + (u >> 1)), u & 1, cr, ca, sf);
        }
    // the normals: float forms them from the node positions; explicit Euler loads them and double
    // a quad's before the barrier (a triangle's came with its coefficients)
    T sn[8];
    if (mine) {
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int k = 0; k < 8; ++k) sn[k] = OFF ? G.sn[k * np + i] : A[k];
        } else if (w[3] < kFvNone) {
            fv_load_geo4(geo, i, 16, sn);
            fv_load_geo4(geo, i, 20, sn + 4);
        } else {
            sn[0] = A[3]; sn[1] = A[7]; sn[2] = A[11]; sn[3] = A[12];
            sn[4] = A[13]; sn[5] = A[14]; sn[6] = sn[7] = T(0);
        }
    }
    __syncthreads();

    // 3. flux of item cell t (Eq. (advection)) from the published face values, then the stage
    //    algebra with the accumulator rows, tau and the parameters from shared memory
    // (double: not released early, see dep_launch)
    if (sizeof(T) == 4) dep_launch();
    double st[4] = {0.0, 0.0, 0.0, 0.0};
    if constexpr (sizeof(T) == 4) {
        if (mine) {
            T q[8], fi[kQ], acc[kQ], macv[3], uo = T(0), vo = T(0);
            V ac[4], fr[4];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = sn[k];
            if (!OFF) fv_normals(q, w[3] >= kFvNone, sn);
            fv_flux<T>(t, sn, w, sf, sv, ac);
            fv_load_row(sf, t, fr);
            fi[0] = sf0[t];
            acc[0] = T(0);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                fi[fv_first(p)] = fr[p].x;
                fi[fv_second(p)] = fr[p].y;
                acc[fv_first(p)] = ac[p].x;
                acc[fv_second(p)] = ac[p].y;
            }
            const InstParam &P = *reinterpret_cast<const InstParam *>(smem_raw + L::ip);
            if (STATS) {
                uo = mac[np + i];
                vo = mac[2 * np + i];
            }
            // C rows hold alpha = 1..8 (stage 2 after the nine of B, stage 3 first)
            const T *a1 = STAGE == 3 ? sacc - IT : sacc, *a2 = sacc + (STAGE == 1 ? kQ : kQ - 1) * IT;
            stage_algebra<T, STAGE, false, NT, IT, STAGE == 1>(i, np, fi, acc, P, STAGE == 3 ? T(1) : sacc[2 * kQ * IT + t],
                                                                 dt_i, a1, IT, t, a2, IT, t, fs_out, fn,
                                                                 Bacc + fv_acc_at<IT>(i, 0), Cacc + fv_acc_at<IT>(i, 0),
                                                                 mac, nullptr, G.area, T(0), macv);
            if (STATS) {
                const double un = double(macv[1]), vn = double(macv[2]), r = double(macv[0]);
                const bool bad = !(isfinite(un) && isfinite(vn) && isfinite(r));
                st[0] = (un - double(uo)) * (un - double(uo)) + (vn - double(vo)) * (vn - double(vo));
                st[1] = un * un + vn * vn;
                st[2] = r * double(G.area[i]);
                st[3] = bad ? 1.0 : 0.0;
            }
        }
    } else if (mine) {
        V ac[4];
        T *const Bi = Bacc + fv_acc_at<IT>(i, 0), *const Ci = Cacc + fv_acc_at<IT>(i, 0);
        fv_flux<T>(t, sn, w, sf, sv, ac);
        const T r0 = ipv<T>(reinterpret_cast<const InstParam *>(smem_raw + L::ip)->rho0,
                            reinterpret_cast<const InstParam *>(smem_raw + L::ip)->rho0_f);
        auto macros = [&](const V *f, T f0) {  // of the new f, and its statistics
            const FvMoments<T> M = fv_moments<T>(f, f0, r0);
            if (STATS) {
                const double un = double(M.u), vn = double(M.v), r = double(M.r);
                const double du = un - double(mac[np + i]), dv = vn - double(mac[2 * np + i]);
                const bool bad = !(isfinite(un) && isfinite(vn) && isfinite(r));
                st[0] = du * du + dv * dv;
                st[1] = un * un + vn * vn;
                st[2] = r * double(G.area[i]);
                st[3] = bad ? 1.0 : 0.0;
            }
            mac[i] = M.r;
            mac[np + i] = M.u;
            mac[2 * np + i] = M.v;
        };
        if (STAGE == 4) {
            // f^{n+1} = f^n + dt (Gamma^a + (f^eq - f^n) / tau)
            const double itau = dt_i / sacc[2 * kQ * IT + t];
            V f[4];
            fv_load_row(sf, t, f);
            const T f0 = sf0[t];
            const FvMoments<T> M = fv_moments<T>(f, f0, r0);
            T o[kQ];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const V eq = fv_feq<T>(M, p);
                const V d = PV::make(eq.x - f[p].x, eq.y - f[p].y);
                f[p] = PV::fma(PV::bcast(-dt_i), ac[p], PV::fma(PV::bcast(itau), d, f[p]));
                o[fv_first(p)] = f[p].x;
                o[fv_second(p)] = f[p].y;
            }
            o[0] = fma(itau, fv_feq0(M) - f0, f0);
            store9(fs_out, np, i, o);
            macros(f, o[0]);
        } else if (STAGE == 1 || STAGE == 2) {
            // X = f^n - dt/2 acc (stage 1), B - dt/2 acc (stage 2); f^(J+1) = f^eq(X) + a (X - f^eq(X))
            T a, g;
            fv_factors(dt_i, sacc[2 * kQ * IT + t], STAGE == 1 ? T(0.25) : T(1.0 / 3.0), a, g);
            const T hdt2 = T(-0.5) * dt_i, dt6 = dt_i * T(1.0 / 6.0);
            g *= T(-1.0 / 3.0);
            V X[4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
                X[p] = PV::fma(PV::bcast(hdt2), ac[p],
                               PV::make(sacc[fv_first(p) * IT + t], sacc[fv_second(p) * IT + t]));
            const T X0 = sacc[t];
            const FvMoments<T> M = fv_moments<T>(X, X0, r0);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const V eq = fv_feq<T>(M, p);
                const V d = PV::make(X[p].x - eq.x, X[p].y - eq.y);
                X[p] = PV::fma(PV::bcast(a), d, eq);
                const int f1 = fv_first(p), f2 = fv_second(p);
                if (STAGE == 1) {  // B = f^n + dt/2 Gamma^a(1) + dt/3 (Gamma^c(1) + Gamma^c(2)), C = -dt/6 Gamma^a(1)
                    const V pb = PV::make(sacc[(kQ + f1) * IT + t], sacc[(kQ + f2) * IT + t]);
                    const V b = PV::fma(PV::bcast(g), d, PV::fma(PV::bcast(hdt2), ac[p], pb));
                    Bi[f1 * IT] = b.x;
                    Bi[f2 * IT] = b.y;
                    Ci[f1 * IT] = dt6 * ac[p].x;
                    Ci[f2 * IT] = dt6 * ac[p].y;
                } else {
                    const V c = PV::fma(PV::bcast(dt6), ac[p],
                                        PV::make(sacc[(kQ + f1 - 1) * IT + t], sacc[(kQ + f2 - 1) * IT + t]));
                    Ci[f1 * IT] = c.x;
                    Ci[f2 * IT] = c.y;
                }
            }
            const T eq0 = fv_feq0(M), d0 = X0 - eq0;
            if (STAGE == 1) Bi[0] = fma(g, d0, sacc[kQ * IT + t]);
            fv_store_stage<T>(fs_out, np, i, fma(a, d0, eq0), X);
        } else {
            // f^{n+1} = f^(3) + C - dt/3 acc (Eq. (imextwo)); macros
            const T dt3 = -(dt_i * T(1.0 / 3.0));
            V f[4];
            fv_load_row(sf, t, f);
            T o[kQ];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int f1 = fv_first(p), f2 = fv_second(p);
                f[p] = PV::fma(PV::bcast(dt3), ac[p], PV::make(f[p].x + sacc[(f1 - 1) * IT + t],
                                                               f[p].y + sacc[(f2 - 1) * IT + t]));
                o[f1] = f[p].x;
                o[f2] = f[p].y;
            }
            o[0] = sf0[t];
            store9(fn, np, i, o);
            macros(f, o[0]);
        }
    }
    if (STATS) block_sum<4, NT>(st, partial + 4 * it);
}
