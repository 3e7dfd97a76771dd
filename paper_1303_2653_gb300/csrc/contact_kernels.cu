// Soft-sphere contact forces, the discrete-element alternative to the
// time-driven hard spheres that §2.2 names for dense beds (normal contact
// only).  Each pair closer than d and each face closer than r pushes with
//
//     F = max(0, k_n delta - eta v_n)      along the line of centres,
//
// delta the overlap and v_n the approach speed; eta is set at creation so that
// a contact without the max() would return the restitution e of Eq. 17-18.
// The forces come from the positions and velocities at the start of the step
// (after the previous sort) and enter Eq. 16 beside the drag and the pressure
// force, in the drag kernel.
//
// With friction (mu > 0) the contact point's tangential slip meets a viscous
// force capped at mu times the normal force (Coulomb), whose torque changes
// the particle spins; the spins after the step are written for the sort to
// carry, those of the start of the step are read.
//
// One thread per particle in sorted order: in sparse beds it walks the cells
// within reach (as the hard-sphere detection does), in crowded ones a block
// bins the particles around its own in shared memory.  The separation of a pair is formed in
// the arithmetic type from the cell indices and in-cell offsets; only a pair
// whose squared distance lies within a thin band around d^2 (wider than the
// rounding of the offsets) takes the exact FP64 test on the positions that
// the oracle uses, so that every contact decision is the exact one.  FP64 is
// slow on this part, and in FP32 this keeps it off all but a few pairs.  The
// overlap is taken as (d^2 - |dx|^2) / (d + |dx|), free of cancellation.
#include "particle_common.cuh"

namespace lbdpsk {

// blocks of 256 threads per SM the register allocation is held to
template <int D, class Real, bool FRIC> struct ContactOccupancy { static constexpr int value = 2; };
template <> struct ContactOccupancy<2, float, false> { static constexpr int value = 6; };
template <> struct ContactOccupancy<2, float, true> { static constexpr int value = 5; };

// w x n for the spin w (one component normal to the plane in 2D) and an
// in-plane (2D) or 3D vector n
template <int D, class Real>
__device__ __forceinline__ void spin_cross(const Real *w, const Real *n, Real *out)
{
    if (D == 2) {
        out[0] = -w[0] * n[1];
        out[1] = w[0] * n[0];
        out[2] = Real(0);
    } else {
        out[0] = w[1] * n[2] - w[2] * n[1];
        out[1] = w[2] * n[0] - w[0] * n[2];
        out[2] = w[0] * n[1] - w[1] * n[0];
    }
}

// One contact as it acts on particle i: unit normal n towards i and normal
// force f > 0; with friction also the tangential force Ft, the lever arm l from
// i's centre to the contact point (at -l n) and n x Ft (cr[0] holds the
// component normal to the plane in 2D), so that the torque is -l cr.
template <class Real, bool FRIC> struct Push;
template <class Real> struct Push<Real, false> { Real f, n[3]; };
template <class Real> struct Push<Real, true> { Real f, n[3], Ft[3], l, cr[3]; };

// Adds a contact to the force F and the torque T.
template <int D, class Real, bool FRIC>
__device__ __forceinline__ void add_push(const Push<Real, FRIC> &c, Real *F, Real *T)
{
#pragma unroll
    for (int a = 0; a < D; ++a) F[a] += c.f * c.n[a];
    if constexpr (FRIC) {
#pragma unroll
        for (int a = 0; a < D; ++a) F[a] += c.Ft[a];
#pragma unroll
        for (int k = 0; k < (D == 2 ? 1 : 3); ++k) T[k] -= c.l * c.cr[k];
    }
}

// Tangential (friction) part of a contact (c.f, c.n and c.l set), from the
// relative velocity vc of the contact point (i's minus the other body's, three
// components, z only used in 3D).  The slip v_t = vc - (vc.n) n meets
// -min(gamma_t |v_t|, mu f) v_t / |v_t|.
template <int D, class Real>
__device__ __forceinline__ void friction(const StepParams<Real> &p, const Real *vc,
                                         Push<Real, true> &c)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) c.Ft[a] = c.cr[a] = Real(0);
    Real vcn = Real(0);
#pragma unroll
    for (int a = 0; a < D; ++a) vcn += vc[a] * c.n[a];
    Real vt[3] = {Real(0), Real(0), Real(0)}, s2 = Real(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        vt[a] = vc[a] - vcn * c.n[a];
        s2 += vt[a] * vt[a];
    }
    if (!(s2 > Real(0))) return;
    const Real st = sqrt(s2);
    Real mag = p.gamma_t * st;
    const Real cap = p.mu_f * c.f;
    if (mag > cap) mag = cap;
    const Real k = -mag / st;
#pragma unroll
    for (int a = 0; a < D; ++a) c.Ft[a] = k * vt[a];
    if (D == 2) {
        c.cr[0] = c.n[0] * c.Ft[1] - c.n[1] * c.Ft[0];
    } else {
        c.cr[0] = c.n[1] * c.Ft[2] - c.n[2] * c.Ft[1];
        c.cr[1] = c.n[2] * c.Ft[0] - c.n[0] * c.Ft[2];
        c.cr[2] = c.n[0] * c.Ft[1] - c.n[1] * c.Ft[0];
    }
}

// The squared contact distance: squared distances beyond hi cannot be contacts,
// those below lo are; the band between covers the rounding of the offsets
// (about 1e-7 in FP32 on a separation of at most 2).  Formed once per thread:
// the conversion from FP64 (2 lanes per clock and SM), made anew for every pair
// tested, took the walk of 1,048,576 particles in 256 x 1024 cells 63 us instead
// of 57.
template <class Real> struct ContactReach {
    Real dd, lo, hi;
    __device__ __forceinline__ explicit ContactReach(const StepParams<Real> &p) : dd((Real)p.d2)
    {
        const Real band = sizeof(Real) == 4 ? Real(4e-6) : Real(1e-12);
        lo = dd - band;
        hi = dd + band;
    }
};

// The contact of particles i and j whose separation dx (i minus j, squared
// length d2 <= reach.hi) is known, as it acts on i.  False for a pair that
// does not push.  vi, wi: i's velocity and spin.
template <int D, class Real, bool FRIC>
__device__ __forceinline__ bool pair_push(const StepParams<Real> &p, const Particles<Real> &parts,
                                          int i, int j, const bool *per, const Real *dx, Real d2,
                                          const ContactReach<Real> &reach, const Real *vi, const Real *wi,
                                          Push<Real, FRIC> &c)
{
    const Real dd = reach.dd;
    if (!(d2 < reach.lo)) {
        // near the contact distance: the exact test of the oracle
        double e2 = 0.0;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            const double t = sep_axis(__ldg(parts.P[a] + i), __ldg(parts.P[a] + j), per[a], p.len[a]);
            e2 = __dadd_rn(e2, __dmul_rn(t, t));
        }
        if (!(e2 < p.d2)) return false;
        if (d2 >= dd) d2 = dd;   // the overlap is then below the rounding: zero
    }
    const Real dist = sqrt(d2);
    const Real delta = (dd - d2) / ((Real)p.d + dist);
    Real vr[3] = {Real(0), Real(0), Real(0)};
    Real vn = Real(0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        c.n[a] = dx[a] / dist;
        vr[a] = vi[a] - __ldg(parts.v[a] + j);
        vn += vr[a] * c.n[a];
    }
    c.f = p.kn * delta - p.eta * vn;
    if (!(c.f > Real(0))) return false;
    if constexpr (FRIC) {
        // contact point half way: vc = v_rel - l (w_i + w_j) x n
        c.l = Real(0.5) * dist;
        Real ws[3] = {Real(0), Real(0), Real(0)}, wxn[3], vc[3];
#pragma unroll
        for (int k = 0; k < (D == 2 ? 1 : 3); ++k) ws[k] = wi[k] + __ldg(parts.w[k] + j);
        spin_cross<D, Real>(ws, c.n, wxn);
#pragma unroll
        for (int a = 0; a < 3; ++a) vc[a] = vr[a] - c.l * wxn[a];
        friction<D, Real>(p, vc, c);
    }
    return true;
}

// The faces' part of particle i (only the first and last cell of an axis can
// be within r < 1/2 of one; the open outlet of a circulating bed makes no
// contact; the contact point lies on the face, at the centre's distance from
// it), added to F and T, and the step's results of the particle.
template <int D, class Real, bool FRIC>
__device__ __forceinline__ void finish_contacts(const StepParams<Real> &p,
                                                const Particles<Real> &parts, int i, const int *idx,
                                                const bool *per, const Real *vi, const Real *wi,
                                                Real *F, Real *T, Real *diag_fc, int np)
{
#pragma unroll
    for (int a = 0; a < D; ++a) {
        if (per[a]) continue;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            if (side == 0 ? idx[a] != 0 : (idx[a] != p.n[a] - 1 || (p.recirculate && a == D - 1)))
                continue;
            const double Pa = __ldg(parts.P[a] + i);
            const double gap = side == 0 ? Pa : __dsub_rn(p.len[a], Pa);
            if (!(gap < p.r64)) continue;
            const Real sg = side == 0 ? Real(1) : Real(-1);   // normal into the bed
            const Real f = p.kn * (Real)__dsub_rn(p.r64, gap) - p.eta_w * (sg * vi[a]);
            if (!(f > Real(0))) continue;
            F[a] += sg * f;
            if constexpr (FRIC) {
                Push<Real, true> c{};
                c.f = f;
                c.n[a] = sg;
                c.l = (Real)gap;
                Real wxn[3], vc[3];
                spin_cross<D, Real>(wi, c.n, wxn);
#pragma unroll
                for (int k = 0; k < 3; ++k) vc[k] = vi[k] - c.l * wxn[k];
                friction<D, Real>(p, vc, c);
#pragma unroll
                for (int k = 0; k < D; ++k) F[k] += c.Ft[k];
#pragma unroll
                for (int k = 0; k < (D == 2 ? 1 : 3); ++k) T[k] -= c.l * c.cr[k];
            }
        }
    }
#pragma unroll
    for (int a = 0; a < D; ++a) p.fc[a][i] = F[a];
    if (FRIC) {
        // I dw = T dt from the start-of-step state
#pragma unroll
        for (int k = 0; k < (D == 2 ? 1 : 3); ++k) p.spin_out[k][i] = wi[k] + T[k] * p.inv_inertia;
    }
    if (diag_fc) {
        const int id = parts.id[i];
#pragma unroll
        for (int a = 0; a < D; ++a) diag_fc[(size_t)a * np + id] = F[a];
    }
}

// The contacts of particle i by a walk over the cells within its own reach.
// FRIC: soft spheres with friction (spins read from parts.w, the new spins
// written to p.spin_out).
template <int D, class Real, bool FRIC>
__device__ __forceinline__ void walk_contacts(const StepParams<Real> &p, const Particles<Real> &parts,
                                              const CellList &cells, Real *diag_fc, int np, int i)
{
    int idx[3];
    cell_coords<D, Real>(p, __ldg(parts.cell + i), idx);
    float oi[3] = {0.f, 0.f, 0.f};
    Real oR[3] = {Real(0), Real(0), Real(0)};
    Real vi[3] = {Real(0), Real(0), Real(0)}, wi[3] = {Real(0), Real(0), Real(0)};
    bool per[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        per[a] = (a < D) && (p.bc[2 * a] == BC_PERIODIC);
        if (a < D) {
            oR[a] = __ldg(parts.off[a] + i);
            oi[a] = (float)oR[a];
            vi[a] = __ldg(parts.v[a] + i);
        }
    }
    if (FRIC) {
#pragma unroll
        for (int c = 0; c < (D == 2 ? 1 : 3); ++c) wi[c] = __ldg(parts.w[c] + i);
    }
    const float cut = (float)p.d + 1e-4f;   // reach of the walk
    const ContactReach<Real> reach(p);
    Real F[3] = {Real(0), Real(0), Real(0)}, T[3] = {Real(0), Real(0), Real(0)};

    auto pair = [&](int j, int rowbase, float sy, float sz) {
        if (j == i) return;
        const Real shift[3] = {(Real)x_shift(p, parts, idx, per[0], j, rowbase), (Real)sy, (Real)sz};
        Real dx[3] = {Real(0), Real(0), Real(0)};
        Real d2 = Real(0);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            dx[a] = oR[a] - __ldg(parts.off[a] + j) - shift[a];
            d2 += dx[a] * dx[a];
        }
        if (d2 > reach.hi) return;
        Push<Real, FRIC> c;
        if (pair_push<D, Real, FRIC>(p, parts, i, j, per, dx, d2, reach, vi, wi, c))
            add_push<D, Real, FRIC>(c, F, T);
    };
    visit_neighbours<D, Real>(p, cells, idx, per, oi, cut, pair);
    finish_contacts<D, Real, FRIC>(p, parts, i, idx, per, vi, wi, F, T, diag_fc, np);
}

// One thread per particle (sparse beds).
template <int D, class Real, bool FRIC>
__global__ void __launch_bounds__(256, ContactOccupancy<D, Real, FRIC>::value)
k_contacts(StepParams<Real> p, Particles<Real> parts, CellList cells, Real *diag_fc, int np)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    walk_contacts<D, Real, FRIC>(p, parts, cells, diag_fc, np, i);
}

// Crowded beds: one block per kBinThreads consecutive sorted particles, a
// thread each.  They lie in a few runs of cells along x; for each run the block
// reads every particle of the rows around it once, keeps those within reach of
// the run's box in shared memory, and bins them by subcells no smaller than the
// reach, so that a particle looks at 9 (27) subcells instead of at every
// particle of up to 4 (8) cells.  The pairs found are then evaluated one per
// lane, whatever particle they belong to, and each thread adds its own
// particle's forces in the order of the walk of k_contacts, so both kernels
// add the same forces in the same order.
//
// Why: the walk is bound by instruction issue.  Its lanes look through
// different sets of cells, so a warp runs as long as its slowest lane with a
// third of its lanes busy, at 22 (2D, 11 particles per cell) to 230 (3D, 84 per
// cell) candidates per particle, and evaluates each lane's few contacts alone.
// Block and shared-memory shape; blocks per SM in FP32 without and with friction
// (2D: 48 registers instead of 40 with spills, 99 -> 95 us on the bed of 256 x
// 1024 cells; with friction the shared memory holds 9); blocks that share the
// runs of a group of slots, and the runs that each of them takes at most (FP64:
// a walk costs five times the time there, so it is left to more runs: rows of
// 2 cells at 11 per cell 277 us with 8, 420 with 3, all runs binned 316, walk
// alone 486).
template <int D> struct BinShape;
template <> struct BinShape<2> {
    static constexpr int threads = 128, cap = 384, bins = 384, hits = 8, blocks_f32 = 10, blocks_fric = 9;
    static constexpr int share = 1, runs_f32 = 3, runs_f64 = 8;
};
template <> struct BinShape<3> {
    static constexpr int threads = 256, cap = 1024, bins = 1024, hits = 12, blocks_f32 = 3, blocks_fric = 3;
    static constexpr int share = 8, runs_f32 = 6, runs_f64 = 6;
};

// in-cell offsets (in 2D o[2] holds the y cell offset of the candidate's row
// from the run) and the unwrapped cell along x
template <class Real> struct alignas(16) BinSlot { Real o[3], x; };

template <int D, class Real, bool FRIC> struct ContactBins {
    // threads of a block, candidates held at a time, subcells, and pairs of
    // one particle listed at a time
    static constexpr int kBinThreads = BinShape<D>::threads, kBinCap = BinShape<D>::cap;
    static constexpr int kBinMax = BinShape<D>::bins, kBinHits = BinShape<D>::hits;
    static_assert(kBinCap <= 1024, "a candidate's number takes 10 bits");
    BinSlot<Real> cand[kBinCap];
    Real yz[D == 3 ? 2 * kBinCap : 1];          // 3D: y and z cell offsets
    int j[kBinCap], key[kBinCap];               // slot; place in the order of the walk
    unsigned short bin[kBinCap], rank[kBinCap], order[kBinCap];
    int start[kBinMax + 1];                     // counts, then first entries in order[]
    unsigned short hit[kBinThreads][kBinHits];  // candidates in contact, by key
    unsigned short flat[kBinThreads / 32][32 * kBinHits];   // a warp's (lane << 10 | candidate)
    Push<Real, FRIC> push[kBinThreads];         // f = 0: the pair does not push
    int seg0[27], cum[28], rowbase[27];
    int warp_tot[kBinThreads / 32], kept;
};

template <int D, class Real, bool FRIC>
__global__ void __launch_bounds__(BinShape<D>::threads, sizeof(Real) != 4 ? 1 : FRIC ? BinShape<D>::blocks_fric
                                                                                : BinShape<D>::blocks_f32)
k_contacts_binned(StepParams<Real> p, Particles<Real> parts, CellList cells, Real *diag_fc, int np)
{
    extern __shared__ __align__(16) unsigned char bins_smem[];
    using Bins = ContactBins<D, Real, FRIC>;
    constexpr int kBinThreads = Bins::kBinThreads, kBinCap = Bins::kBinCap, kBinMax = Bins::kBinMax;
    constexpr int kBinHits = Bins::kBinHits;
    Bins &t = *reinterpret_cast<Bins *>(bins_smem);
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kRowCells = D == 2 ? kBinMax / 3 - 2 : kBinMax / 9 - 2;   // longest run (m = 1)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int first = blockIdx.x * kBinThreads, end = min(first + kBinThreads, np);
    const int i = first + tid;
    int idx[3] = {0, 0, 0};
    Real oi[3] = {Real(0), Real(0), Real(0)};
    Real vi[3] = {Real(0), Real(0), Real(0)}, wi[3] = {Real(0), Real(0), Real(0)};
    bool per[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) per[a] = (a < D) && (p.bc[2 * a] == BC_PERIODIC);
    if (i < np) {
        cell_coords<D, Real>(p, __ldg(parts.cell + i), idx);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            oi[a] = __ldg(parts.off[a] + i);
            vi[a] = __ldg(parts.v[a] + i);
        }
        if (FRIC) {
#pragma unroll
            for (int k = 0; k < (D == 2 ? 1 : 3); ++k) wi[k] = __ldg(parts.w[k] + i);
        }
    }
    const float cut = (float)p.d + 1e-4f;
    const ContactReach<Real> reach(p);
    Real F[3] = {Real(0), Real(0), Real(0)}, T[3] = {Real(0), Real(0), Real(0)};

    // The thin top of a bed spreads a block over many rows, a run for each, at
    // 2-3 us a run in 2D and 5-15 in 3D.  In 3D gridDim.y blocks share the runs:
    // the 16 x 16 x 32 bed's launch grew from 120 to 366 us as its top loosened
    // with one, to 177 with four and 153 with eight; spare blocks leave at once (a
    // steady launch: 110.5 us with one, 109 with eight).  A row of n[0] cells
    // holds at most ceil(n[0] / kRowCells) runs, each of which starts kRowCells
    // cells or more after the one before.
    if (blockIdx.y > 0) {
        const int rows = p.by_row(__ldg(parts.cell + end - 1)) - p.by_row(__ldg(parts.cell + first)) + 1;
        if ((long long)rows * ((p.n[0] + kRowCells - 1) / kRowCells) <= (int)blockIdx.y) return;
    }
    // The slots past the first share * runs runs are walked a thread each, as in
    // k_contacts: so few particles to a run have few candidates.  64 x 512 cells,
    // the lower half at 11 per cell, one particle in each row above: 294 us with
    // every run binned, 25.7 so (walk alone 33; at most 2, 4 and 8 runs: 25.7, 27.7
    // and 36); 16 x 16 x 32, a third at 30 per cell, one in each row above, friction:
    // 164 us, 54 so (walk alone 70; at most 32 and 64 runs: 46 and 64; but 32 cost
    // 3 x 40 x 40 cells, half filled at 50, 119 us a step against 111).
    constexpr int kRuns = BinShape<D>::share * (sizeof(Real) == 4 ? BinShape<D>::runs_f32 : BinShape<D>::runs_f64);
    int rest = end;
    bool taken = false;   // the thread's particle was in one of this block's runs
    for (int s = first, e, run = 0; s < end; s = e, ++run) {
        if (run == kRuns) {
            rest = s;
            break;
        }
        // the run [s, e): the particles left in the row of slot s (at most kRowCells cells)
        const int c0 = __ldg(parts.cell + s), xa = c0 - p.by_row(c0) * p.n[0], row = c0 - xa;
        e = min(end, cells.begin(row + min(p.n[0], xa + kRowCells)));
        if (run % BinShape<D>::share != (int)blockIdx.y) continue;
        const int xb = __ldg(parts.cell + e - 1) - row;
        const int ncx = xb - xa + 1;
        int ri[3];
        cell_coords<D, Real>(p, row, ri);
        // m subcells per cell along each axis, none smaller than the reach
        int m = max(1, (int)(0.9999f / cut));
        while (m > 1 && (ncx * m + 2) * (m + 2) * (D == 3 ? m + 2 : 1) > kBinMax) --m;
        const int nxs = ncx * m + 2, nys = m + 2, nb = nxs * nys * (D == 3 ? nys : 1);
        const bool mine = i >= s && i < e;
        taken = taken || mine;
        // subcell of an in-cell offset
        auto sub = [&](Real o) { return min((int)(o * (Real)m), m - 1); };
        const int bx = (idx[0] - xa) * m + sub(oi[0]), by = sub(oi[1]), bz = D == 3 ? sub(oi[2]) : 0;

        // The slots to read: per plane the rows below, at and above the run,
        // then, for a run that ends at a periodic x face, the cell across it
        // in each row (the order of the walk).
        const int x0 = max(xa - 1, 0), x1 = min(xb + 1, p.n[0] - 1);
        const int per_plane = per[0] && (xa == 0 || xb == p.n[0] - 1) ? 9 : 3;
        const int nseg = per_plane * (D == 3 ? 3 : 1);
        if (warp == 0) {
            int len = 0;
            if (lane < nseg) {
                const int g = lane % per_plane, oz = D == 3 ? lane / per_plane - 1 : 0;
                const int r = g < 3 ? g : (g - 3) >> 1;
                int qy = ri[1] + r - 1, qz = ri[2] + oz;
                bool ok = true;
                if (qy < 0 || qy >= p.n[1]) {
                    ok = per[1];
                    qy = qy < 0 ? qy + p.n[1] : qy - p.n[1];
                }
                if (D == 3 && (qz < 0 || qz >= p.n[2])) {
                    ok = ok && per[2];
                    qz = qz < 0 ? qz + p.n[2] : qz - p.n[2];
                }
                int lo = x0, hi = x1;
                if (g >= 3) {   // across the low face (the last cell) or the high one
                    lo = hi = (g & 1) ? p.n[0] - 1 : 0;
                    ok = ok && ((g & 1) ? xa == 0 : xb == p.n[0] - 1);
                }
                const int base = p.n[0] * (qy + p.n[1] * qz);
                const int b0 = ok ? cells.begin(base + lo) : 0;
                len = ok ? cells.begin(base + hi + 1) - b0 : 0;
                t.seg0[lane] = b0;
                // subtracted from a cell index: its unwrapped cell along x
                t.rowbase[lane] = g < 3 ? base : ((g & 1) ? base + p.n[0] : base - p.n[0]);
            }
            int inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(kAll, inc, o);
                if (lane >= o) inc += u;
            }
            if (lane < nseg) t.cum[lane + 1] = inc;
            if (lane == 0) {
                t.cum[0] = 0;
                t.kept = 0;
            }
        }
        for (int b = tid; b < nb; b += kBinThreads) t.start[b] = 0;
        __syncthreads();
        const int total = t.cum[nseg];
        int sg = 0;
        for (int e0 = 0; e0 < total;) {
            // read on until the next kBinThreads might not fit
            int kept = 0;
            for (; e0 < total && kept + kBinThreads <= kBinCap; e0 += kBinThreads) {
                const int at = e0 + tid;
                bool keep = at < total;
                BinSlot<Real> c{};
                int j = 0, sy = 0, sz = 0;
                if (keep) {
                    while (at >= t.cum[sg + 1]) ++sg;
                    const int g = sg % per_plane;
                    sy = (g < 3 ? g : (g - 3) >> 1) - 1;
                    sz = D == 3 ? sg / per_plane - 1 : 0;
                    j = t.seg0[sg] + at - t.cum[sg];
#pragma unroll
                    for (int a = 0; a < D; ++a) c.o[a] = __ldg(parts.off[a] + j);
                    const int x = __ldg(parts.cell + j) - t.rowbase[sg];
                    c.x = (Real)x;
                    // within reach of the run's box
                    const float fx = (float)c.o[0], fy = (float)c.o[1];
                    if (x < xa) keep = fx > 1.f - cut;
                    if (x > xb) keep = keep && fx < cut;
                    if (sy < 0) keep = keep && fy > 1.f - cut;
                    if (sy > 0) keep = keep && fy < cut;
                    if (D == 3) {
                        const float fz = (float)c.o[2];
                        if (sz < 0) keep = keep && fz > 1.f - cut;
                        if (sz > 0) keep = keep && fz < cut;
                    }
                }
                const unsigned b = __ballot_sync(kAll, keep);
                int base = 0;
                if (lane == 0 && b) base = atomicAdd(&t.kept, __popc(b));
                base = __shfl_sync(kAll, base, 0);
                if (keep) {
                    const int k = base + __popc(b & ((1u << lane) - 1u));
                    const int x = (int)c.x;
                    int bin = (x - xa) * m + sub(c.o[0]) + 1 + nxs * (sy * m + sub(c.o[1]) + 1);
                    if (D == 3) bin += nxs * nys * (sz * m + sub(c.o[2]) + 1);
                    if (D == 2) c.o[2] = (Real)sy;
                    t.cand[k] = c;
                    if (D == 3) {
                        t.yz[2 * k] = (Real)sy;
                        t.yz[2 * k + 1] = (Real)sz;
                    }
                    t.j[k] = j;
                    t.key[k] = at;
                    t.bin[k] = (unsigned short)bin;
                    t.rank[k] = (unsigned short)atomicAdd(&t.start[bin], 1);
                }
                __syncthreads();
                kept = t.kept;
                __syncthreads();
            }
            // exclusive scan of the counts, in place
            {
                constexpr int kPer = kBinMax / kBinThreads;
                const int lo = tid * kPer;
                int v[kPer], sum = 0;
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    v[k] = lo + k < nb ? t.start[lo + k] : 0;
                    sum += v[k];
                }
                int inc = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int u = __shfl_up_sync(kAll, inc, o);
                    if (lane >= o) inc += u;
                }
                if (lane == 31) t.warp_tot[warp] = inc;
                __syncthreads();
                int at = inc - sum;
#pragma unroll
                for (int w = 0; w < kBinThreads / 32; ++w)
                    if (w < warp) at += t.warp_tot[w];
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    if (lo + k < nb) t.start[lo + k] = at;
                    at += v[k];
                }
                if (tid == 0) {
                    t.start[nb] = kept;
                    t.kept = 0;
                }
            }
            __syncthreads();
            for (int k = tid; k < kept; k += kBinThreads)
                t.order[t.start[t.bin[k]] + t.rank[k]] = (unsigned short)k;
            __syncthreads();

            // separation of the thread's particle from candidate c
            auto separation = [&](const BinSlot<Real> &q, int c, const Real *o, Real x, Real *dx) {
                const Real s3[3] = {q.x - x, D == 2 ? q.o[2] : t.yz[D == 3 ? 2 * c : 0],
                                    D == 3 ? t.yz[2 * c + 1] : Real(0)};
                Real d2 = Real(0);
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    dx[a] = o[a] - q.o[a] - s3[a];
                    d2 += dx[a] * dx[a];
                }
                return d2;
            };
            // calls f(c) for the candidates in contact range of the thread's
            // particle (an image farther than a cell away along x is another
            // candidate's business)
            auto look = [&](auto &&f) {
                const Real x = (Real)idx[0];
#pragma unroll 1
                for (int dz = 0; dz < (D == 3 ? 3 : 1); ++dz) {
#pragma unroll 1
                    for (int dy = 0; dy < 3; ++dy) {
                        const int b = bx + nxs * (by + dy + (D == 3 ? nys * (bz + dz) : 0));
                        const int k1 = t.start[b + 3];
                        for (int k = t.start[b]; k < k1; ++k) {
                            const int c = t.order[k];
                            const BinSlot<Real> q = t.cand[c];
                            Real dx[3];
                            const Real d2 = separation(q, c, oi, x, dx);
                            if (!(d2 > reach.hi) && t.j[c] != i && !(fabs(q.x - x) > Real(1))) f(c);
                        }
                    }
                }
            };
            int hits = 0;
            if (mine) {
                look([&](int c) {
                    int at = hits++;
                    if (at >= kBinHits) return;
                    const int key = t.key[c];
                    for (; at > 0 && t.key[t.hit[tid][at - 1]] > key; --at) t.hit[tid][at] = t.hit[tid][at - 1];
                    t.hit[tid][at] = (unsigned short)c;
                });
            }
            if (hits > kBinHits) {
                // more than the list holds (spheres pressed far into each
                // other): one pass of the walk per pair, in order
                for (int done = -1;;) {
                    int next = INT_MAX, nc = 0;
                    look([&](int c) {
                        const int key = t.key[c];
                        if (key > done && key < next) {
                            next = key;
                            nc = c;
                        }
                    });
                    if (next == INT_MAX) break;
                    done = next;
                    Real dx[3];
                    const Real d2 = separation(t.cand[nc], nc, oi, (Real)idx[0], dx);
                    Push<Real, FRIC> c;
                    if (pair_push<D, Real, FRIC>(p, parts, i, t.j[nc], per, dx, d2, reach, vi, wi, c))
                        add_push<D, Real, FRIC>(c, F, T);
                }
                hits = 0;
            }
            // the warp's pairs in one list, particle by particle
            int h1 = hits;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(kAll, h1, o);
                if (lane >= o) h1 += u;
            }
            const int h0 = h1 - hits, nh = __shfl_sync(kAll, h1, 31);
            for (int k = 0; k < hits; ++k)
                t.flat[warp][h0 + k] = (unsigned short)(lane << 10 | t.hit[tid][k]);
            __syncwarp();
            Push<Real, FRIC> *push = t.push + 32 * warp;
            for (int b0 = 0; b0 < nh; b0 += 32) {
                // one pair per lane; its particle's state comes from the owning lane
                const bool have = b0 + lane < nh;
                const int fl = have ? t.flat[warp][b0 + lane] : 0, own = fl >> 10, c = fl & 1023;
                Real om[3] = {Real(0), Real(0), Real(0)};
                Real vm[3] = {Real(0), Real(0), Real(0)}, wm[3] = {Real(0), Real(0), Real(0)};
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    om[a] = __shfl_sync(kAll, oi[a], own);
                    vm[a] = __shfl_sync(kAll, vi[a], own);
                }
                const int xm = __shfl_sync(kAll, idx[0], own);
                if (FRIC) {
#pragma unroll
                    for (int k = 0; k < (D == 2 ? 1 : 3); ++k) wm[k] = __shfl_sync(kAll, wi[k], own);
                }
                if (have) {
                    Real dx[3];
                    const Real d2 = separation(t.cand[c], c, om, (Real)xm, dx);
                    if (!pair_push<D, Real, FRIC>(p, parts, i - lane + own, t.j[c], per, dx, d2, reach, vm, wm,
                                                  push[lane]))
                        push[lane].f = Real(0);
                }
                __syncwarp();
                const int k1 = min(h1, b0 + 32);
                for (int k = max(h0, b0); k < k1; ++k)
                    if (push[k - b0].f > Real(0)) add_push<D, Real, FRIC>(push[k - b0], F, T);
                __syncwarp();
            }
            __syncthreads();
            if (e0 < total) {
                for (int b = tid; b < nb; b += kBinThreads) t.start[b] = 0;
                __syncthreads();
            }
        }
        __syncthreads();
    }
    if (taken) finish_contacts<D, Real, FRIC>(p, parts, i, idx, per, vi, wi, F, T, diag_fc, np);
    else if (blockIdx.y == 0 && i >= rest && i < np) walk_contacts<D, Real, FRIC>(p, parts, cells, diag_fc, np, i);
}

// Whether the binned kernel is taken.  It pays by the particles per cell, and the
// narrower the rows, the more runs a block has.  Both sides on a GB300, d = 0.2
// (us; even: spread evenly, half: the lower half filled, particles per cell of
// the whole bed), walk / binned:
//     2D      even 5     even 5.5   even 7      even 9      half 5.6
//     512^2   80 / 87    92 / 91    135 / 113   206 / 140   158 / 108
//     256^2   29 / 32    33 / 34    45 / 40     63 / 49     51 / 38
//     64^2    16 / 20    16 / 20    19 / 20     21 / 20     23 / 20
//     2D rows of   16          12         10         8          6          4 cells
//     even 8       41 / 42     42 / 47    42 / 47    41 / 53    42 / 65    41 / 68
//     even 11      67 / 52     66 / 55    66 / 59    66 / 63    67 / 70    65 / 99
//     half 5.6     51 / 40     51 / 42    52 / 45    53 / 48    51 / 52    51 / 72
//     3D                 even 8      even 10    even 12    even 20    half 25, friction
//     48 x 48 x 64       295 / 280
//     20 x 20 x 40       46 / 50     66 / 55
//     8 x 40 x 40        44 / 56                60 / 64    149 / 85   428 / 118
//     4 x 40 x 40        29 / 46                35 / 52    83 / 62    247 / 72
//     2 x 40 x 40        26 / 38                32 / 42    46 / 54    153 / 52
// 2D: 5.5 per cell lies between the two fillings' own lines, and 66 per row holds
// both.  3D: 8 per cell in wide beds, the more the narrower the rows.  In FP64 a
// pair tested costs the walk more (the FP64 pipe) and the lines lie lower: 256 x
// 256 even 5.1 288 / 175; rows of 4 cells, 2D, even 5.1 130 / 153 and 8 276 / 182;
// of 2 cells even 8 271 / 279, 11 486 / 316; 3D rows of 1 cell even 12 91 / 107,
// 20 137 / 123, of 2 cells even 8.1 104 / 97.
template <int D, class Real> static bool bins_pay(long long np, long long ncell, long long n0)
{
    const long long rows = ncell / n0;
    constexpr bool f32 = sizeof(Real) == 4;
    if (D == 2) return 2 * np >= (f32 ? 11 : 10) * ncell && np >= (f32 ? 66 : 22) * rows;
    return f32 ? np >= 8 * ncell + 20 * rows : np >= 8 * ncell && np >= 16 * rows;
}

template <int D, class Real, bool FRIC>
static void launch_contacts_fric(const StepParams<Real> &p, Particles<Real> parts, CellList cells,
                                 Real *diag_fc, int np, cudaStream_t st)
{
    if (bins_pay<D, Real>(np, p.ncell, p.n[0])) {
        constexpr size_t smem = sizeof(ContactBins<D, Real, FRIC>);
        constexpr int kBinThreads = BinShape<D>::threads;
        // a refusal shows as the launch's error
        cudaFuncSetAttribute(k_contacts_binned<D, Real, FRIC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
        const dim3 grid((np + kBinThreads - 1) / kBinThreads, BinShape<D>::share);
        k_contacts_binned<D, Real, FRIC><<<grid, kBinThreads, smem, st>>>(
            p, parts, cells, diag_fc, np);
    } else {
        const int b = wave_block(k_contacts<D, Real, FRIC>, np);
        k_contacts<D, Real, FRIC><<<(np + b - 1) / b, b, 0, st>>>(p, parts, cells, diag_fc, np);
    }
}

template <int D, class Real>
void launch_contacts(const StepParams<Real> &p, Particles<Real> parts, CellList cells,
                     Real *diag_fc, int np, cudaStream_t st)
{
    if (np == 0) return;
    if (p.spin_out[0]) launch_contacts_fric<D, Real, true>(p, parts, cells, diag_fc, np, st);
    else launch_contacts_fric<D, Real, false>(p, parts, cells, diag_fc, np, st);
}

#define LBDPS_INST_C(D, R)                                                                          \
    template void launch_contacts<D, R>(const StepParams<R> &, Particles<R>, CellList, R *, int,    \
                                        cudaStream_t);
LBDPS_INST_C(2, double)
LBDPS_INST_C(2, float)
LBDPS_INST_C(3, double)
LBDPS_INST_C(3, float)

}  // namespace lbdpsk
