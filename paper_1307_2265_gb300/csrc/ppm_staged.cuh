// The split PPM sweep by stages: one thread per zone, then per face, then per
// cell, of a tile of whole pencils held in shared memory.
//
// The marching kernel (ppm_device.cuh) keeps one pencil per thread: its
// parallelism is the number of pencils, its time the length of one, and its
// loop body is longer than the instruction cache, which every warp walks on its
// own.  Here a tile of at most THREADS zones goes through the steps of the
// method together: primitives; slopes; interface values; parabolas and traced
// states; Riemann problems; update.  Each step reads its neighbours from shared
// memory, and its zones, faces or cells are dealt out to consecutive threads,
// so no lane of a warp idles in a ghost zone where ghosts have no part.  Every
// value is formed by the same functions as in the march, so results agree bit
// for bit (FP32 through the functions' stated roundings; the HLLC flux's are the
// compiler's, the same in both kernels as far as the tests compare them).
//
// Measured, a step against the march with the same arithmetic: FP64, where the
// pipe is the bound, 82% busy instead of 49% (the march's warps wait for
// instructions): 400 patches (2e7 cells) 142 -> 84 ms, a walled 100x75x50 grid
// 10.0 -> 1.55 ms, a 32^3 grid 4.2 -> 0.20 ms.  FP32, for batches of few pencils
// only (a march that fills the chip issues 35% fewer instructions per cell): a
// 32^3 grid 324 -> 76 us, a walled 240x125x61 grid with the reconstruction options
// 1730 -> 754 us.  (Dealing items by a reciprocal instead of integer divisions is
// 2% of that.)
//
// A pencil longer than the tile goes in windows of W positions.  A window
// updates cells [lo, hi), reads the four positions on either side (the
// fallback test of the neighbouring cell needs its two faces), and hands the
// last eight positions, as they were before any update, to the next window
// through shared memory.
#pragma once
#include "ppm_device.cuh"

namespace enzo {

template <class R, int THREADS, int EXT>
struct StagedSmem {
    static constexpr int NV = EXT == 2 ? 6 : 5;        // traced variables (eps with dual energy)
    static constexpr int NX = EXT == 2 ? THREADS : 1;
    double U[5][THREADS];           // raw conserved values (rho, m_n, m_t1, m_t2, E)
    double ge[NX], En[NX];          // gas energy, E after the update
    R q[NV + 1][THREADS];           // zone primitives r, u, p, t1, t2, c (and eps)
    R A[NV][THREADS];               // slopes, then right states of the zones' left edges
    R B[NV][THREADS];               // interface values at s+1/2, then fluxes
    R C[NV][THREADS];               // left states of the zones' right edges
    R uf[NX];                       // interface velocities (gas energy)
    R ds[EXT ? THREADS : 1];        // density slopes (contact steepening)
    R save[NV + 1][3][kStagedMaxPencils];   // windowed wrapped pencils: the first three active zones
    double save_E[kStagedMaxPencils];       // and the first one's E
    // windowed pencils with dual energy: the last updated cell, whose
    // resynchronisation waits for its right neighbour's new E
    double pend[4][kStagedMaxPencils];      // advected ge, E - KE, E, left neighbour's E
    bool pend_ok[kStagedMaxPencils];
    unsigned char bad[THREADS];
    int64_t base[THREADS / 7 + 1];  // storage index of each pencil's position 0 (a pencil has at least 7)
};

template <class R, int DIR, int THREADS, bool REG, int EXT>
struct Staged {
    static constexpr int A1 = DIR == 0 ? 1 : 0;
    static constexpr int A2 = DIR == 2 ? 1 : 2;
    using Smem = StagedSmem<R, THREADS, EXT>;
    static constexpr int NV = Smem::NV;
    static constexpr bool dual = EXT == 2;
    static_assert(!dual || sizeof(R) == 8, "FP32 dual-energy sweeps march");
    const SweepArgs &a;
    const enzo_patch &P;
    Smem &S;
    const Consts<R> &k;
    Counters &cnt;
    R dtdx;
    double dtdx64, dt64;
    int np, W, L, n, ng;       // pencils of this tile, window, pencil length, active cells, ghosts
    int pen0, cnt1, r1, r2;    // first pencil, pencils per row of the cross-section, its origin
    int64_t st1, st2, sd;
    bool wrap;
    int patch;
    int j0, p0;                // y and z pencils: this thread's position and pencil at every step

    // Storage index of position 0 of pencil p of the tile.
    __device__ __forceinline__ int64_t base(int p) const
    {
        const int pe = pen0 + p;
        const int i2 = pe / cnt1, i1 = pe - i2 * cnt1;
        return P.off + (int64_t)(r1 + i1) * st1 + (int64_t)(r2 + i2) * st2;
    }
    // Deal item t of m per pencil: pencil p and item j; x pencils item-fastest,
    // y and z pencils pencil-fastest (neighbouring x), so global accesses run
    // along x.
    __device__ __forceinline__ void deal(int t, int m, int &p, int &j) const
    {
        static_assert(THREADS <= 256, "items are dealt by a reciprocal");
        if (DIR == 0) {
            // t / m from a reciprocal: exact for t < 256, as (t + 1/2) / m is at
            // least 1/(2m) from a whole number
            p = (int)(((float)t + 0.5f) * rcp_approx((float)m));
            j = t - p * m;
        } else {
            j = j0;
            p = p0;
        }
    }
    // Slot of window position w of pencil p; the slot one position on.
    __device__ __forceinline__ int slot(int p, int w) const { return DIR == 0 ? p * W + w : w * np + p; }
    __device__ __forceinline__ int next() const { return DIR == 0 ? 1 : np; }

    __device__ __forceinline__ Zone<R> zone(int z) const
    {
        return Zone<R>{S.q[0][z], S.q[1][z], S.q[2][z], S.q[3][z], S.q[4][z], S.q[5][z]};
    }

    __device__ __forceinline__ double widen(R F) const
    {
        return sizeof(R) == 8 ? (double)F : f2d_exact((float)(dtdx * F));
    }

    // Gas energy of a cell after its resynchronisation (Sec. 4.1.1): E - KE
    // where that exceeds a tenth of the largest E of the cell and its neighbours.
    __device__ __forceinline__ static double resync(double g, double e, double E, double El, double Er, bool ok)
    {
        double emax = El;
        if (x64::less(emax, E)) emax = E;
        if (x64::less(emax, Er)) emax = Er;
        return ok && x64::less(0.1 * emax, e) ? e : g;
    }

    // Flux registers of face f (left of active cell f) of pencil p, as the
    // march records them (a sixth component with dual energy).
    __device__ __forceinline__ void record(int p, int f, const double G[5], double gG) const
    {
        if (!REG || !a.freg) return;
        const int pe = pen0 + p, i2 = pe / cnt1, i1 = pe - i2 * cnt1;
        const int j1 = r1 + i1 - ng, j2 = r2 + i2 - ng;
        const int na1 = P.n[A1], na2 = P.n[A2];
        if (j1 < 0 || j1 >= na1 || j2 < 0 || j2 >= na2) return;
        int64_t oall = 0, obnd = 0;
        for (int d = 0; d < DIR; ++d) {
            const int b1 = d == 0 ? 1 : 0, b2 = d == 2 ? 1 : 2;
            oall += (int64_t)(P.n[d] + 1) * P.n[b1] * P.n[b2] * NV;
            obnd += (int64_t)2 * P.n[b1] * P.n[b2] * NV;
        }
        const int64_t row = (int64_t)j2 * na1 + j1;
        if (P.freg_all >= 0) {
            double *o = a.freg + P.freg_all + oall + (row * (n + 1) + f) * NV;
            _Pragma("unroll") for (int v = 0; v < 5; ++v) o[v] = G[v];
            if constexpr (dual) o[5] = gG;
        }
        if (P.freg_bnd >= 0 && (f == 0 || f == n)) {
            double *o = a.freg + P.freg_bnd + obnd + (row * 2 + (f == 0 ? 0 : 1)) * NV;
            _Pragma("unroll") for (int v = 0; v < 5; ++v) o[v] = o[v] + (sizeof(R) == 8 ? dt64 * G[v] : G[v]);
            if constexpr (dual) o[5] = o[5] + dt64 * gG;
        }
    }

    __device__ __forceinline__ void log_states(int p, int s, const R l[3], const R r[3]) const
    {
        // the march's key and step: pencil identity, and the step that solves
        // the interface right of position s
        const int kk = s + 3;
        const unsigned key = (unsigned)patch * 7919u + (unsigned)(pen0 + p);
        const unsigned h = (key * 2654435761u) ^ ((unsigned)kk * 40503u);
        if ((h % (unsigned)a.log_stride) != 0u) return;
        const unsigned long long i = atomicAdd(a.log_count, 1ull);
        if ((long long)i >= a.log_cap) return;
        float *o = a.log + 6 * i;
        _Pragma("unroll") for (int v = 0; v < 3; ++v)
        {
            o[v] = (float)l[v];
            o[3 + v] = (float)r[v];
        }
    }

    // One window: positions [w0, w0 + m), cells [lo, hi) updated.  fresh: first
    // window position not handed over by the window before.
    __device__ __forceinline__ void window(int w0, int m, int lo, int hi, int fresh)
    {
        const int t = threadIdx.x;
        const bool first = w0 == 0, last = hi == L - ng;
        const bool windowed = W < L;
        const int map[5] = {0, 1 + DIR, 1 + A1, 1 + A2, 4};
        int p, j;
        // zones: load and primitives
        deal(t, m - fresh, p, j);
        if (p < np && j < m - fresh) {
            const int w = fresh + j, s = w0 + w, z = slot(p, w);
            const int64_t b = base(p);
            if (j == 0) S.base[p] = b;
            bool count = true, saved = false;
            int64_t idx = b + (int64_t)s * sd;
            if (wrap) {
                const int c = s - ng;
                if (c < 0 || c >= n) idx = b + (int64_t)(ng + (c % n + n) % n) * sd;
                count = c < n;
                saved = windowed && c >= n;
            }
            Zone<R> q;
            R eps = (R)0;
            if (saved) {
                const int i = s - ng - n;
                q = Zone<R>{S.save[0][i][p], S.save[1][i][p], S.save[2][i][p],
                            S.save[3][i][p], S.save[4][i][p], S.save[5][i][p]};
                if constexpr (dual) {
                    eps = S.save[6][i][p];
                    if (i == 0) S.U[4][z] = S.save_E[p];
                }
            } else {
                double u[5];
                _Pragma("unroll") for (int v = 0; v < 5; ++v) u[v] = a.U[map[v]][idx];
                Counters c;
                c.st = count ? cnt.st : nullptr;
                if constexpr (dual) {
                    const double g = a.ge[idx];
                    q = prim_dual<true>(u[0], u[1], u[2], u[3], u[4], g, k, c, eps);
                    cnt.gep += count ? c.gep : 0u;
                    S.ge[z] = g;
                } else if constexpr (sizeof(R) == 4) q = prim_f<true, true>(u[0], u[1], u[2], u[3], u[4], k, c);
                else q = prim<R, true>(u[0], u[1], u[2], u[3], u[4], k, c);
                _Pragma("unroll") for (int v = 0; v < 5; ++v) S.U[v][z] = u[v];
                if (windowed && wrap && s >= ng && s < ng + 3) {
                    const int i = s - ng;
                    S.save[0][i][p] = q.r;
                    S.save[1][i][p] = q.u;
                    S.save[2][i][p] = q.p;
                    S.save[3][i][p] = q.t1;
                    S.save[4][i][p] = q.t2;
                    S.save[5][i][p] = q.c;
                    if constexpr (dual) {
                        S.save[6][i][p] = eps;
                        if (i == 0) S.save_E[p] = u[4];
                    }
                }
            }
            S.q[0][z] = q.r;
            S.q[1][z] = q.u;
            S.q[2][z] = q.p;
            S.q[3][z] = q.t1;
            S.q[4][z] = q.t2;
            S.q[5][z] = q.c;
            if constexpr (dual) S.q[6][z] = eps;
        }
        __syncthreads();
        const int e = next();
        // slopes of positions 1 .. m-2
        deal(t, m - 2, p, j);
        if (p < np && j < m - 2) {
            const int z = slot(p, 1 + j);
            _Pragma("unroll") for (int v = 0; v < NV; ++v)
            {
                const int w = v < 5 ? v : 6;
                S.A[v][z] = limited_slope<R>(S.q[w][z - e], S.q[w][z], S.q[w][z + e]);
            }
            if constexpr (EXT) S.ds[z] = S.A[0][z];
        }
        __syncthreads();
        // interface values right of positions 1 .. m-3
        deal(t, m - 3, p, j);
        if (p < np && j < m - 3) {
            const int z = slot(p, 1 + j);
            _Pragma("unroll") for (int v = 0; v < NV; ++v)
            {
                const int w = v < 5 ? v : 6;
                S.B[v][z] = face_value<R, true>(S.q[w][z], S.q[w][z + e], S.A[v][z], S.A[v][z + e]);
            }
        }
        __syncthreads();
        // parabolas and traced states of positions 2 .. m-3
        deal(t, m - 4, p, j);
        if (p < np && j < m - 4) {
            const int z = slot(p, 2 + j);
            R pL[5], pR[5], pd[5], p6[5], sR[5], sL[5];
            if constexpr (EXT) {
                R el[5], er[5], elx = (R)0, erx = (R)0;
                _Pragma("unroll") for (int v = 0; v < 5; ++v)
                {
                    el[v] = S.B[v][z - e];
                    er[v] = S.B[v][z];
                }
                if constexpr (dual) {
                    elx = S.B[5][z - e];
                    erx = S.B[5][z];
                }
                dissipate<R, true>(k, a.mp, zone(z - e), zone(z), zone(z + e), zone(z + 2 * e), S.q[0][z - 2 * e],
                                   S.q[2][z - 2 * e], S.ds[z - e], S.ds[z + e], el, er, dual ? S.q[NV][z] : (R)0,
                                   dual ? &elx : nullptr, dual ? &erx : nullptr);
                _Pragma("unroll") for (int v = 0; v < 5; ++v)
                    parabola<R, true>(S.q[v][z], el[v], er[v], pL[v], pR[v], pd[v], p6[v]);
                if constexpr (dual) {
                    R xL, xR, xd, x6;
                    parabola<R, true>(S.q[6][z], elx, erx, xL, xR, xd, x6);
                    S.A[5][z] = trace_passive<R, -1>(xL, xR, xd, x6, S.q[1][z], dtdx);
                    S.C[5][z] = trace_passive<R, +1>(xL, xR, xd, x6, S.q[1][z], dtdx);
                }
            } else {
                _Pragma("unroll") for (int v = 0; v < 5; ++v)
                    parabola<R, true>(S.q[v][z], S.B[v][z - e], S.B[v][z], pL[v], pR[v], pd[v], p6[v]);
            }
            trace<R, true>(pL, pR, pd, p6, S.q[1][z], S.q[5][z], dtdx, k, sR, sL);
            _Pragma("unroll") for (int v = 0; v < 5; ++v)
            {
                S.A[v][z] = sR[v];
                S.C[v][z] = sL[v];
            }
        }
        __syncthreads();
        // Riemann problems right of positions 2 .. m-4; this window answers for
        // the faces left of its cells and, at the pencil's end, the last one
        deal(t, m - 5, p, j);
        if (p < np && j < m - 5) {
            const int w = 2 + j, s = w0 + w, z = slot(p, w);
            const bool own = s >= lo - 1 && (s < hi - 1 || last);
            R l[5], r[5], F[5], gF = (R)0;
            _Pragma("unroll") for (int v = 0; v < 5; ++v)
            {
                l[v] = S.C[v][z];
                r[v] = S.A[v][z + e];
            }
            if (a.log && own) log_states(p, s, l, r);
            if (a.mp.solver == ENZO_SOLVER_TWOSHOCK) {
                const RiemannOut<R> o = riemann<R, true>(l[0], l[1], l[2], r[0], r[1], r[2], (R)-1, k, cnt);
                if (own) {
                    cnt.iters += (unsigned)o.iters;
                    if (!o.conv) cnt.rare(ENZO_ST_NEWTON_NONCONV);
                }
                const bool up = o.ustar >= (R)0;
                phys_flux<R, true>(o.rho, o.u, o.p, up ? l[3] : r[3], up ? l[4] : r[4], k, F);
                if constexpr (dual) {
                    gF = F[0] * (up ? S.C[5][z] : S.A[5][z + e]);
                    S.uf[z] = o.u;
                }
            } else if (a.mp.solver == ENZO_SOLVER_HLLC) {
                hllc_states<R>(l, r, k, F);
            } else {
                hll_states<R>(l, r, k, F);
            }
            if constexpr (EXT) {
                if (a.mp.options & ENZO_OPT_DIFFUSE)
                    diffuse<R, true>(k, zone(z), zone(z + e), F, dual ? S.q[NV][z] : (R)0,
                                     dual ? S.q[NV][z + e] : (R)0, dual ? &gF : nullptr);
            }
            _Pragma("unroll") for (int v = 0; v < 5; ++v) S.B[v][z] = F[v];
            if constexpr (dual) S.B[5][z] = gF;
        }
        __syncthreads();
        // does the Godunov update leave rho > 0?  Cells [lo - 1, hi] of the
        // pencil's active ones (the neighbours' answers decide shared faces)
        const bool fb = a.mp.fallback != 0;
        if (fb) {
            bool any = false;
            const int c0 = first ? lo : lo - 1, c1 = last ? hi : hi + 1;
            deal(t, c1 - c0, p, j);
            if (p < np && j < c1 - c0) {
                const int s = c0 + j, z = slot(p, s - w0);
                const R fm = S.B[0][z - e], fp = S.B[0][z];
                bool bad = false;
                if (EXT && a.mp.fallback == 2) {
                    // FP32: a screen on the zone's own primitives with wide margins; unclear
                    // cells take the exact test on the update they would get
                    R Fm[5], Fp[5];
                    _Pragma("unroll") for (int v = 0; v < 5; ++v)
                    {
                        Fm[v] = S.B[v][z - e];
                        Fp[v] = S.B[v][z];
                    }
                    if (sizeof(R) == 8 || !clearly_ok<R>(k, zone(z), Fm, Fp, dtdx)) {
                        double u[5];
                        _Pragma("unroll") for (int v = 0; v < 5; ++v)
                            u[v] = sizeof(R) == 8 ? cell_update(S.U[v][z], dtdx64, (double)Fm[v], (double)Fp[v])
                                                  : (S.U[v][z] + widen(Fm[v])) - widen(Fp[v]);
                        bad = fails_state(u);
                    }
                } else if (sizeof(R) == 8) {
                    bad = !x64::gt0(cell_update(S.U[0][z], dtdx64, (double)fm, (double)fp));
                } else {
                    // FP32 screen; cells near zero are decided in FP64
                    const R r0 = S.q[0][z];
                    if (!(r0 + dtdx * (fm - fp) > (R)1e-3 * r0))
                        bad = !((S.U[0][z] + f2d_exact((float)(dtdx * fm))) - f2d_exact((float)(dtdx * fp)) > 0.0);
                }
                if (bad && s >= lo && s < hi) cnt.rare(ENZO_ST_HLL_CELLS);
                S.bad[z] = bad;
                any = bad;
            }
            if (__syncthreads_or(any)) {
                // a face beside a failing cell takes HLL from the zone states
                // (Sec. 4.1.2), its gas-energy flux the mass flux times the upwind
                // eps, its interface velocity the mean zone velocity; formed here
                // once, for both of its cells and the flux register
                deal(t, hi - lo + 1, p, j);
                if (p < np && j < hi - lo + 1) {
                    const int s = lo - 1 + j, z = slot(p, s - w0);
                    if ((s >= ng && S.bad[z]) || (s + 1 < L - ng && S.bad[z + e])) {
                        const Zone<R> l = zone(z), r = zone(z + e);
                        R F[5];
                        hll_flux<R>(l, r, k, F);
                        _Pragma("unroll") for (int v = 0; v < 5; ++v) S.B[v][z] = F[v];
                        if constexpr (dual) {
                            S.B[5][z] = F[0] * (F[0] >= (R)0 ? S.q[6][z] : S.q[6][z + e]);
                            S.uf[z] = (R)0.5 * (l.u + r.u);
                        }
                    }
                }
                __syncthreads();
            }
        }
        // update of cells [lo, hi)
        deal(t, hi - lo, p, j);
        const bool mine = p < np && j < hi - lo;
        const int s = lo + j, z = mine ? slot(p, s - w0) : 0;
        const int64_t idx = mine ? S.base[p] + (int64_t)s * sd : 0;
        double u[5], gnew = 0.0, enew = 0.0;
        bool ok = false;
        if (mine) {
            R Fm[5], Fp[5], gm = (R)0, gp = (R)0, um = (R)0, up = (R)0;
            double Gm[5], Gp[5];
            _Pragma("unroll") for (int v = 0; v < 5; ++v)
            {
                Fm[v] = S.B[v][z - e];
                Fp[v] = S.B[v][z];
            }
            if constexpr (dual) {
                gm = S.B[5][z - e];
                gp = S.B[5][z];
                um = S.uf[z - e];
                up = S.uf[z];
            }
            _Pragma("unroll") for (int v = 0; v < 5; ++v)
            {
                Gm[v] = widen(Fm[v]);
                Gp[v] = widen(Fp[v]);
            }
            const double ggm = (double)gm, ggp = (double)gp;
            if (REG) {
                record(p, s - ng, Gm, ggm);
                if (s == L - ng - 1) record(p, n, Gp, ggp);
            }
            _Pragma("unroll") for (int v = 0; v < 5; ++v)
            {
                const double U = S.U[v][z];
                u[v] = sizeof(R) == 8 ? cell_update(U, dtdx64, Gm[v], Gp[v]) : (U + Gm[v]) - Gp[v];
            }
            if constexpr (dual) {
                const double g0 = S.ge[z];
                const R pz = S.q[2][z];
                gnew = (g0 + dtdx64 * (ggm - ggp)) - dtdx64 * (double)pz * ((double)up - (double)um);
                ok = x64::gt0(u[0]);
                if (ok) enew = u[4] - x64::div<-1>((u[1] * u[1] + u[2] * u[2]) + u[3] * u[3], u[0], x64::recip(u[0]));
            }
            if (fb && (EXT && a.mp.fallback == 2 ? fails_state(u) : !x64::gt0(u[0]))) cnt.rare(ENZO_ST_NEG_AFTER);
            if (x64::is_nan(u[0]) || x64::is_nan(u[4])) cnt.rare(ENZO_ST_NAN);
            _Pragma("unroll") for (int v = 0; v < 5; ++v) a.U[map[v]][idx] = u[v];
        }
        if constexpr (dual) {
            // resynchronisation: neighbours' new E; ghosts beside the pencil's
            // ends keep theirs from the start of the sweep
            double keep[4] = {0.0, 0.0, 0.0, 0.0};
            bool keep_ok = false;
            if (mine) S.En[z] = u[4];
            __syncthreads();
            if (mine) {
                double El = s > lo ? S.En[z - e] : S.U[4][z - e];
                if (!first && s == lo) {
                    // the window before left its last cell pending
                    _Pragma("unroll") for (int i = 0; i < 4; ++i) keep[i] = S.pend[i][p];
                    keep_ok = S.pend_ok[p];
                    El = keep[2];
                    a.ge[idx - sd] = resync(keep[0], keep[1], keep[2], keep[3], u[4], keep_ok);
                }
                if (s == hi - 1 && !last) {
                    keep[0] = gnew;
                    keep[1] = enew;
                    keep[2] = u[4];
                    keep[3] = El;
                    keep_ok = ok;
                } else {
                    a.ge[idx] = resync(gnew, enew, u[4], El, s < hi - 1 ? S.En[z + e] : S.U[4][z + e], ok);
                }
            }
            if (!last) {
                __syncthreads();
                if (mine && s == hi - 1) {
                    _Pragma("unroll") for (int i = 0; i < 4; ++i) S.pend[i][p] = keep[i];
                    S.pend_ok[p] = keep_ok;
                }
            }
        }
    }

    __device__ void run()
    {
        if (W >= L) {
            window(0, L, ng, L - ng, 0);
            return;
        }
        int w0 = 0, lo = ng, fresh = 0;
        for (;;) {
            const bool last = w0 + W >= L;
            const int m = last ? L - w0 : W, hi = last ? L - ng : w0 + W - 4;
            window(w0, m, lo, hi, fresh);
            if (last) return;
            // the next window starts four positions left of its first cell
            const int nw = hi - 4;
            int p, j;
            deal(threadIdx.x, 8, p, j);
            const bool mine = p < np && j < 8;
            R q[NV + 1];
            double u[5], g = 0.0;
            if (mine) {
                const int z = slot(p, nw - w0 + j);
                _Pragma("unroll") for (int v = 0; v < NV + 1; ++v) q[v] = S.q[v][z];
                _Pragma("unroll") for (int v = 0; v < 5; ++v) u[v] = S.U[v][z];
                if constexpr (dual) g = S.ge[z];
            }
            __syncthreads();
            if (mine) {
                const int z = slot(p, j);
                _Pragma("unroll") for (int v = 0; v < NV + 1; ++v) S.q[v][z] = q[v];
                _Pragma("unroll") for (int v = 0; v < 5; ++v) S.U[v][z] = u[v];
                if constexpr (dual) S.ge[z] = g;
            }
            w0 = nw;
            lo = hi;
            fresh = 8;
        }
    }
};

// This CTA's own work list of a small batch, and the zones per tile: of 256,
// 224 .. 128 the one that gives the busiest SM the smallest share (a 32^3 grid in
// FP64 has 171 tiles of 256 zones, two on some SMs and one on most).
template <int DIR, int THREADS>
__device__ __forceinline__ int staged_list(const SweepArgs &a, int *pre, int &zones)
{
    static_assert(THREADS == kListPatches, "one patch per thread");
    constexpr int A1 = DIR == 0 ? 1 : 0, A2 = DIR == 2 ? 1 : 2, kCand = 5;
    __shared__ int sum[kCand];
    const int t = threadIdx.x;
    int pen = 0, L = 1;
    if (t < a.npatch) {
        const enzo_patch &P = a.patches[t];
        if (patch_ok(P, a.field_len)) {
            int lo[3], hi[3];
            sweep_ranges(P, DIR, a.cover_mask, lo, hi);
            pen = (hi[A1] - lo[A1]) * (hi[A2] - lo[A2]);
            L = P.n[DIR] + 2 * P.ng;
        } else if (blockIdx.x == 0) {
            atomicAdd(a.status + ENZO_ST_BAD_PATCH, 1ull);
        }
    }
    if (t < kCand) sum[t] = 0;
    __syncthreads();
    int tiles[kCand];
    for (int c = 0; c < kCand; ++c) {
        int per = 1, window = 0;
        if (pen) staged_shape(L, THREADS * (8 - c) / 8, per, window);
        tiles[c] = (pen + per - 1) / per;
        const int w = __reduce_add_sync(0xffffffffu, tiles[c]);
        if ((t & 31) == 0) atomicAdd(&sum[c], w);
    }
    __syncthreads();
    // the busiest SM's share of the zones, and 4% for each step down in size
    int best = 0, mine = 0;
    float cost = 1e30f;
    for (int c = 0; c < kCand; ++c) {
        const float z = (float)((sum[c] + a.sms - 1) / a.sms) / (float)max(sum[c], 1) * (1.0f + 0.04f * (float)c);
        if (z < cost) {
            cost = z;
            best = c;
            mine = tiles[c];
        }
    }
    zones = THREADS * (8 - best) / 8;
    return list_scan(mine, pre);
}

// Persistent kernel: CTAs take (patch, tile) items from a device counter, or in
// a fixed stride from their own list of a small batch.
template <class R, int DIR, int THREADS, bool REG, int EXT, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) ppm_staged_kernel(const __grid_constant__ SweepArgs a)
{
    extern __shared__ __align__(16) unsigned char dsmem[];
    // the tile at hand, found by one thread: its patch, dt/dx (a division each
    // thread made for itself cost FP32 sweeps more of the FP64 pipe than their
    // updates)
    __shared__ enzo_patch s_patch;
    __shared__ double s_dtdx;
    __shared__ int s_tile, s_index, s_per, s_window, s_pre[kListPatches + 1];
    StagedSmem<R, THREADS, EXT> &S = *reinterpret_cast<StagedSmem<R, THREADS, EXT> *>(dsmem);
    constexpr int A1 = DIR == 0 ? 1 : 0, A2 = DIR == 2 ? 1 : 2;
    Counters cnt;
    cnt.st = a.status;
    const Consts<R> k = make_consts<R>(a.mp);
    const double dt = a.dt_ptr ? *a.dt_ptr : a.dt;
    unsigned long long interfaces = 0;
    const int *prefix = a.prefix;
    int zones = THREADS, total;
    if (prefix) total = prefix[a.npatch];
    else {
        total = staged_list<DIR, THREADS>(a, s_pre, zones);
        prefix = s_pre;
    }
    for (int turn = blockIdx.x;; turn += gridDim.x) {
        if (threadIdx.x == 0) {
            int tile = a.prefix ? (int)atomicAdd(a.tile_counter, 1u) : turn;
            if (tile >= total) tile = -1;
            else {
                const int lo = find_patch(prefix, a.npatch, tile);
                s_patch = a.patches[lo];
                s_index = lo;
                s_dtdx = x64::div(dt, a.patches[lo].dx[DIR]);
                int per, window;
                staged_shape(a.patches[lo].n[DIR] + 2 * a.patches[lo].ng, zones, per, window);
                s_per = per;
                s_window = window;
                tile -= prefix[lo];
            }
            s_tile = tile;
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const enzo_patch &P = s_patch;
        int rlo[3], rhi[3];
        sweep_ranges(P, DIR, a.cover_mask, rlo, rhi);
        const int cnt1 = rhi[A1] - rlo[A1], cnt2 = rhi[A2] - rlo[A2];
        const int64_t N0 = P.n[0] + 2 * P.ng, N1 = P.n[1] + 2 * P.ng;
        const int64_t stride[3] = {1, N0, N0 * N1};
        const int L = P.n[DIR] + 2 * P.ng;
        const int per = s_per, W = s_window;
        const int pen0 = tile * per;
        const int np = min(per, cnt1 * cnt2 - pen0);
        const double dtdx64 = s_dtdx;
        if (threadIdx.x == 0) interfaces += (unsigned long long)np * (P.n[DIR] + 1);
        Staged<R, DIR, THREADS, REG, EXT> t{a,  P,    S,  k,  cnt,  (R)dtdx64, dtdx64, dt, np, W, L, P.n[DIR], P.ng, pen0,
                                       cnt1, rlo[A1], rlo[A2], stride[A1], stride[A2], stride[DIR],
                                       (P.flags & ENZO_PATCH_PERIODIC) != 0, s_index,
                                       (int)(threadIdx.x / (unsigned)np), (int)(threadIdx.x % (unsigned)np)};
        t.run();
        __syncthreads();
    }
    warp_flush(a.status, interfaces, ENZO_ST_INTERFACES);
    warp_flush(a.status, cnt.iters, ENZO_ST_NEWTON_ITERS);
    warp_flush(a.status, cnt.restarts, ENZO_ST_GUESS_RESTARTS);
    if constexpr (EXT == 2) warp_flush(a.status, cnt.gep, ENZO_ST_GE_PRESSURE);
}

template <class R, int DIR, int THREADS, bool REG, int EXT, int MINB>
cudaError_t launch_staged_one(const SweepArgs &a, cudaStream_t s)
{
    auto kern = ppm_staged_kernel<R, DIR, THREADS, REG, EXT, MINB>;
    constexpr int bytes = (int)sizeof(StagedSmem<R, THREADS, EXT>);
    static int cached[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!cached[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, THREADS, bytes);
        cached[dev] = (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
    }
    kern<<<cached[dev], THREADS, bytes, s>>>(a);
    return cudaGetLastError();
}

template <class R, int THREADS, int EXT, int MINB>
cudaError_t launch_staged(const SweepArgs &a, cudaStream_t s)
{
    if (a.freg) {
        switch (a.dir) {
        case 0: return launch_staged_one<R, 0, THREADS, true, EXT, MINB>(a, s);
        case 1: return launch_staged_one<R, 1, THREADS, true, EXT, MINB>(a, s);
        default: return launch_staged_one<R, 2, THREADS, true, EXT, MINB>(a, s);
        }
    }
    switch (a.dir) {
    case 0: return launch_staged_one<R, 0, THREADS, false, EXT, MINB>(a, s);
    case 1: return launch_staged_one<R, 1, THREADS, false, EXT, MINB>(a, s);
    default: return launch_staged_one<R, 2, THREADS, false, EXT, MINB>(a, s);
    }
}

}  // namespace enzo
