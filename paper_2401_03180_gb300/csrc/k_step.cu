// Per-atom part of one timestep: velocity kick + drift (Sec. II.B, Eq. 12,
// velocity Verlet), the stochastic collisional-radiative charge update
// (Sec. II.A), and the free-electron-gas reduction that sets the Debye length
// (Sec. II.A, Eq. 3) together with the next cell grid.
//
// The charge update must reproduce the CPU oracle bit for bit, so its
// floating-point work uses only IEEE double basic operations written with
// explicit round-to-nearest intrinsics (no fused multiply-add), and this file
// is compiled with -fmad=false as a second guard.
#include "md_internal.cuh"

namespace mdg {

constexpr int kAccCopies = 16;   // accumulator copies per replica (spread contention)
// kStepAtoms atoms per block of the step kernel: one warp of each role.  Blocks this
// small wait at their barriers for two warps only, so the SM keeps issuing
// from the other blocks (water box: 1.8 us less per step than 128 atoms per
// block; 2 M-atom droplet: 87 us less)
constexpr int kStepThreads = 2 * kStepAtoms;   // two threads per atom: kick/drift and charge update

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): 10 rounds, multipliers M0, M1 on
// words 0 and 2, Weyl key schedule W0, W1.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// The 53-bit uniform ((a >> 5) 2^26 + (b >> 6)) 2^-53.  Its value is the
// integer m times a power of two, exactly, so the double is assembled from m
// in the integer pipe (GB300 issues FP64 at 2 lanes per SM per clock): the
// exponent from the leading one of m, the 52 bits below it as the mantissa.
__device__ __forceinline__ double u53(unsigned a, unsigned b)
{
    const unsigned long long m = ((unsigned long long)(a >> 5) << 26) | (unsigned long long)(b >> 6);
    if (m == 0ull) return 0.0;
    const int lz = __clzll((long long)m);                           // 11 .. 63
    const unsigned long long mant = ((m << lz) << 1) >> 12;         // the bits below the leading one
    const unsigned long long ex = (unsigned long long)(1033 - lz);  // 1023 + (63 - lz) - 53
    return __longlong_as_double((long long)((ex << 52) | mant));
}

// 1 - e^{-x}: x = k/16 + r, (1 - E_k) + E_k (1 - e^{-r}), degree-12 Taylor
// polynomial of 1 - e^{-r} in nested form; E_k and 1/m come from host tables.
__device__ __forceinline__ double one_minus_exp_neg(double x, const double* etab,
                                                    const double* inv)
{
    if (!(x > 0.0)) return 0.0;
    double xs = __dmul_rn(x, 16.0);
    if (xs >= (double)kNEtab) return 1.0;
    int k = (int)xs;
    double r = __dsub_rn(x, __dmul_rn((double)k, 0.0625));
    double t = 1.0;
#pragma unroll
    for (int m = 12; m >= 2; --m) t = __dsub_rn(1.0, __dmul_rn(__dmul_rn(r, inv[m]), t));
    double g = __dmul_rn(r, t);
    if (k == 0) return g;
    double ek = etab[k];
    return __dadd_rn(__dsub_rn(1.0, ek), __dmul_rn(ek, g));
}

__device__ __forceinline__ double interp(const double* K, int i0, double w)
{
    return __dadd_rn(K[i0], __dmul_rn(w, __dsub_rn(K[i0 + 1], K[i0])));
}

// Adaptive skin: whether this step rebuilds (x) and whether the list it builds
// carries the skin (y), from the step's largest displacement and the current
// list.  A pure function, so that the warps sizing the grids and the thread
// that records the decision agree.
__device__ __forceinline__ int2 adapt_decision(const Params& p, unsigned maxd2)
{
    const ListCtl& c = *p.lc;
    if (c.buffered) {
        const int rebuild = maxd2 > __float_as_uint(c.half_skin2) ? 1 : 0;
        return make_int2(rebuild, rebuild && c.since_build + 1 < kAdaptOffLife ? 0 : 1);
    }
    // one step since the last build: maxd2 is the largest one-step
    // displacement d, and a buffered list would last (skin/2) / d steps
    return make_int2(1, __uint_as_float(maxd2) * (float)(kAdaptOnLife * kAdaptOnLife) <= p.half_skin2 ? 1 : 0);
}

// Radius of the list this step builds: the cells' smallest edge.
template <bool SETCOND>
__device__ __forceinline__ double next_rlist(const Params& p, unsigned maxd2)
{
    if (SETCOND && p.lc) return adapt_decision(p, maxd2).y ? p.r_list : p.r_cut;
    return list_rlist(p);
}

// Velocity increment of a half kick, (dt/2m) F.  The mixed path forms it in
// FP32 (it is ~1e-4 of v, so its rounding is far below the FP32 force error);
// the FP64 path in FP64.  Every kernel that applies or reports a half kick
// uses this function, so stepping and state read-out round identically.
__device__ __forceinline__ void half_kick(const Params& p, int s, int slot, double& ax, double& ay,
                                          double& az)
{
    const double c = p.hdtm[s];
    if (p.precision == 0) {
        const float cf = p.hdtm_f[s];   // (float)(c 2^-32), formed on the host
        ax = (double)(cf * (float)p.fx[slot]);
        ay = (double)(cf * (float)p.fy[slot]);
        az = (double)(cf * (float)p.fz[slot]);
    } else {
        ax = c * ((double)p.fx[slot] * kFixInv);
        ay = c * ((double)p.fy[slot] * kFixInv);
        az = c * ((double)p.fz[slot] * kFixInv);
    }
}

// ---------------------------------------------------------------------------
// k_step_a: one thread per atom (original order).
// ---------------------------------------------------------------------------
constexpr int kInlineReps = 4;   // up to this many replicas (eight lanes of a warp each) the step kernel's last block reduces them

// Three standard normal numbers for the Langevin force (Sec. II.B, Eq. 14)
// from four Philox words: Box-Muller on u = (w + 1/2) 2^-32 for the pairs
// (w0, w1) and (w2, w3), of which the first three results are used.  The
// mixed path works in FP32 (u rounded to 24 bits, relative error 6e-8 down to
// the smallest u, which rounds up to 1 at most), the FP64 path in FP64.
__device__ __forceinline__ void gauss3(uint4 w, bool fp32, double& g0, double& g1, double& g2)
{
    if (fp32) {
        const float ua = __fmul_rn(__fadd_rn((float)w.x, 0.5f), 2.3283064e-10f);
        const float ub = __fmul_rn(__fadd_rn((float)w.y, 0.5f), 2.3283064e-10f);
        const float uc = __fmul_rn(__fadd_rn((float)w.z, 0.5f), 2.3283064e-10f);
        const float ud = __fmul_rn(__fadd_rn((float)w.w, 0.5f), 2.3283064e-10f);
        const float ra = sqrtf(-2.0f * logf(ua)), rb = sqrtf(-2.0f * logf(uc));
        float sb, cb;
        sincospif(2.0f * ub, &sb, &cb);
        g0 = (double)(ra * cb);
        g1 = (double)(ra * sb);
        g2 = (double)(rb * cospif(2.0f * ud));
    } else {
        const double s = 2.3283064365386963e-10;   // 2^-32
        const double ua = ((double)w.x + 0.5) * s, ub = ((double)w.y + 0.5) * s;
        const double uc = ((double)w.z + 0.5) * s, ud = ((double)w.w + 0.5) * s;
        const double ra = sqrt(-2.0 * log(ua)), rb = sqrt(-2.0 * log(uc));
        double sb, cb;
        sincospi(2.0 * ub, &sb, &cb);
        g0 = ra * cb;
        g1 = ra * sb;
        g2 = rb * cospi(2.0 * ud);
    }
}

// Hybrid ion-sphere / Debye electrostatics of every charge state at the
// plasma state just computed (Sec. II.A, Eqs. 4-7), by the warp that reduced
// replica rr.  An ion of charge Q has R = (3Q / (4 pi n_e))^{1/3} (Eq. 4) and
// the transition radius r' of Eq. 7, evaluated as s^3 / (kappa (t^2 + t + 1))
// with s = kappa R and t = (1 + s^3)^{1/3} (no cancellation).  Its potential
// is Q/r + c1 - c2 r^2 inside r' and G e^{-kappa r}/r outside; the continuity
// of the potential and its first two derivatives at r' gives, with
// x = kappa r' and D = 3 + 3x + x^2, G = 3 Q e^x / D,
// c1 = -Q kappa (3 + 3x/2) / D and c2 = -2 pi n_e / 3 for every Q.
// Without an ion sphere (Q = 0, n_e = 0 or kappa = 0): r' = 0, G = Q.
// R itself is not needed, (kappa R)^3 is; the neutral atom skips the divisions,
// whose slow path a zero numerator takes for the whole warp (hybrid box of 12,003
// atoms: step kernel 16.1 -> 15.0 us).
__device__ void hyb_table(const Params& p, int rr, int lane, double kap, double ne)
{
    HybQ* rows = p.hq + (size_t)rr * kHybQ;
    const double c2 = -2.0 * kPi * ne / 3.0;
    const double rc = p.r_cut;
    double rpm = 0.0;
    for (int q = lane; q <= p.z_max; q += 32) {   // the charge states the species can reach
        const double Q = (double)q;
        double G = Q, rp = 0.0, c1 = 0.0;
        const bool ion = q > 0 && ne > 0.0 && kap > 0.0;
        double phirc = 0.0;
        if (ion) {
            const double s3 = 3.0 * Q / (4.0 * kPi * ne) * kap * kap * kap;   // (kappa R)^3
            const double t = cbrt(1.0 + s3);
            rp = s3 / (kap * (t * t + t + 1.0));
            const double x = kap * rp;
            const double D = 3.0 + 3.0 * x + x * x;
            c1 = -Q * kap * (3.0 + 1.5 * x) / D;
            G = 3.0 * Q * exp(x) / D;
        }
        if (q > 0) {
            const bool in = rc < rp;
            const double ph = (in ? Q : G * exp(-kap * rc)) / rc;
            phirc = in ? ph + c1 - c2 * rc * rc : ph;
        }
        HybQ h;
        h.G = G; h.rp = rp; h.c1 = c1; h.phirc = phirc;
        h.Gf = (float)fmin(G, 1.0e30); h.rpf = (float)rp; h.c1f = (float)c1; h.phircf = (float)phirc;
        rows[q] = h;
        rpm = fmax(rpm, rp);
    }
    for (int o = 16; o; o >>= 1) rpm = fmax(rpm, __shfl_xor_sync(0xffffffffu, rpm, o));
    if (lane == 0) {
        HybRep r;
        r.c2 = c2; r.rpm2 = rpm * rpm; r.c2f = (float)c2; r.rpm2f = (float)(rpm * rpm);
        p.hrep[rr] = r;
    }
}

// The per-step reduction of up to four replicas (base .. base + nr - 1, eight
// lanes each) and the plasma scalars of their next step (Eq. 3 and the helpers of
// the charge update), by one warp.
//
// It runs at the end of every step with nothing else on the GPU, so its chain of
// dependent operations counts: lane f < 6 of a replica loads field f of all
// accumulator copies at once and reduces (and clears) them; the FP64 divisions and
// roots, each some hundreds of cycles on GB300's FP64 pipe, are issued once for
// several lanes: T_e on lane 0 with n_e on lane 1, kappa on lane 0 with the
// species' Langevin widths on the lanes from 1.  The cell grids are sized by
// finalize_grid on another warp meanwhile.  With
// one chain for everything (thirteen divisions and a square root) the step kernel
// took 15.9 us for 1,500 methane atoms in vacuum, 18.5 for 12,003 atoms of water
// with hybrid screening and 19.4 for the 45k-atom droplet; with this, the box
// reduced without contention, the records packed while the charge-update warp
// flushes, and the rate bounds below: 9.4, 15.0 and 13.3 us (water box of 30,000
// atoms 14.5 -> 10.7).
__device__ void finalize_plasma(const Params& p, int base, int nr, int lane, long long next)
{
    constexpr unsigned kFull = 0xffffffffu;
    static_assert(sizeof(RepAccum) == 12 * sizeof(long long), "twelve fields of eight bytes");
    const int sub = lane & 7;
    const bool on = (lane >> 3) < nr;
    const int rr = on ? base + (lane >> 3) : base;
    const bool head = on && sub == 0;
    RepState st{};
    double vol = 1.0, pne = 0.0, pte = 0.0;
    if (head) {   // issued before the accumulators are read and cleared
        st = p.rs[rr];
        if (p.plasma_mode == 1) {
            const long long idx = (long long)rr * (p.max_steps + 1) + (next <= p.max_steps ? next : p.max_steps);
            pne = p.pres_ne[idx];
            pte = p.pres_te[idx];
        }
    }
    if (on && sub == 1) vol = p.volume[rr];
    unsigned long long sum = 0ull;
    if (on && sub < 6) {
        unsigned long long* f = reinterpret_cast<unsigned long long*>(p.acc + (size_t)rr * kAccCopies) + sub;
        unsigned long long v[kAccCopies];
#pragma unroll
        for (int c = 0; c < kAccCopies; ++c) v[c] = __ldcg(f + 12 * c);
#pragma unroll
        for (int c = 0; c < kAccCopies; ++c) f[12 * c] = 0ull;
#pragma unroll
        for (int o = kAccCopies / 2; o; o >>= 1)
#pragma unroll
            for (int c = 0; c < o; ++c) v[c] += v[c + o];
        sum = v[0];
    }
    const long long dE = (long long)__shfl_sync(kFull, sum, 1, 8);
    long long dc[4];
    for (int k = 0; k < 4; ++k) dc[k] = (long long)__shfl_sync(kFull, sum, 2 + k, 8);
    if (sub == 0) {
        st.n_e += (long long)sum;
        st.e_gas += dE;
        if (st.e_gas < 0) st.e_gas = 0;
        for (int k = 0; k < 4; ++k) st.counts[k] += dc[k];
    }
    const long long n_e = __shfl_sync(kFull, st.n_e, 0, 8);
    double num = 1.0, den = 1.0;
    if (sub == 0 && n_e > 0) {
        num = (double)st.e_gas;
        den = __dmul_rn(1500.0, (double)n_e);
    } else if (sub == 1 && n_e > 0) {
        num = (double)n_e;
        den = vol;
    }
    double quo = __ddiv_rn(num, den);
    const double n_dens = __shfl_sync(kFull, quo, 1, 8);
    double te = 0.0, ne = 0.0;
    if (p.plasma_mode == 1) {
        ne = pne;
        te = pte;
    } else if (n_e > 0) {
        te = quo;
        ne = n_dens;
    }
    te = __shfl_sync(kFull, te, 0, 8);
    ne = __shfl_sync(kFull, ne, 0, 8);
    num = den = 1.0;
    // Langevin update of the next step per species (Eqs. 13-14): gamma =
    // n_e g_s, c = e^{-gamma dt}, sigma = sqrt((1 - c^2) k_B T_e / m_s); species s
    // on lane s + 1, the last of eight after the others
    double lc = 0.0;
    const int ls = sub - 1;
    const bool lgv = p.langevin && on && ls >= 0 && ls < p.n_species;
    if (lgv) {
        lc = exp(-(ne * p.lgv_g[ls]) * p.dt);
        num = (1.0 - lc * lc) * (te * kEvKJmol);
        den = p.mass[ls];
    } else if (head && ne > 0.0) {
        const double tc = te > p.te_floor ? te : p.te_floor;
        num = __dmul_rn(p.four_pi_f, ne);
        den = __dmul_rn(tc, kEvKJmol);
    }
    const double root = __dsqrt_rn(__ddiv_rn(num, den));
    if (lgv) p.lgv[(size_t)rr * kMaxSpecies + ls] = make_double2(lc, root);
    if (head) {
        const double kap = ne > 0.0 ? root : 0.0;
        st.te_ev = te;
        st.n_dens = ne;
        st.kappa = kap;
        st.ne_dt = __dmul_rn(ne, p.dt);
        double x = __dmul_rn(te, p.inv_dte);
        if (x > (double)(p.n_te - 1)) x = (double)(p.n_te - 1);
        if (x < 0.0) x = 0.0;
        int i0 = (int)x;
        if (i0 > p.n_te - 2) i0 = p.n_te - 2;
        st.it0 = i0;
        st.wt = __dsub_rn(x, (double)i0);
        const double kf = p.kappa_fixed >= 0.0 ? p.kappa_fixed : kap;
        st.kappa_force = kf;
        st.kappa_f = (float)kf;
        p.rs[rr] = st;
        if (p.langevin && p.n_species == kMaxSpecies) {
            const int s = kMaxSpecies - 1;
            const double c = exp(-(ne * p.lgv_g[s]) * p.dt);
            p.lgv[(size_t)rr * kMaxSpecies + s] =
                make_double2(c, __dsqrt_rn(__ddiv_rn((1.0 - c * c) * (te * kEvKJmol), p.mass[s])));
        }
    }
    if (p.screening)
        for (int k = 0; k < nr; ++k)
            hyb_table(p, base + k, lane, __shfl_sync(kFull, st.kappa_force, 8 * k), __shfl_sync(kFull, st.n_dens, 8 * k));
}

// The bounding boxes of up to four replicas (eight lanes each) and, for a vacuum
// replica, the cell grid of the positions reduced into it; rl: the radius of the
// list built on the grid.
__device__ void finalize_grid(const Params& p, int base, int nr, int lane, double rl)
{
    constexpr unsigned kFull = 0xffffffffu;
    const int sub = lane & 7;
    const bool on = (lane >> 3) < nr;
    const int rr = on ? base + (lane >> 3) : base;
    Grid& g = p.grid[rr];
    const int periodic = g.periodic, cell_cap = g.cell_cap;
    // lower ends on lanes 0 to 2, upper ends on 3 to 5, both as maxima (of complements)
    unsigned long long mx = 0ull;
    if (on && sub < 6 && !periodic) {
        unsigned long long* f = reinterpret_cast<unsigned long long*>(p.acc + (size_t)rr * kAccCopies) + 6 + sub;
        const unsigned long long flip = sub < 3 ? ~0ull : 0ull;
        unsigned long long m[kAccCopies];
#pragma unroll
        for (int c = 0; c < kAccCopies; ++c) m[c] = __ldcg(f + 12 * c);
#pragma unroll
        for (int c = 0; c < kAccCopies; ++c) {
            m[c] ^= flip;
            f[12 * c] = flip;
        }
#pragma unroll
        for (int o = kAccCopies / 2; o; o >>= 1)
#pragma unroll
            for (int c = 0; c < o; ++c) m[c] = max(m[c], m[c + o]);
        mx = m[0] ^ flip;
    }
    if (__all_sync(kFull, !on || periodic)) return;
    const int d = sub < 3 ? sub : 0;   // lane d: dimension d
    const unsigned long long mn = __shfl_sync(kFull, mx, d, 8);
    mx = __shfl_sync(kFull, mx, 3 + d, 8);
    double lo = mn == ~0ull ? 0.0 : from_ordered(mn), hi = mx == 0ull ? 0.0 : from_ordered(mx);
    if (!(hi >= lo)) lo = hi = 0.0;
    const bool size = on && !periodic;
    const double ext = size ? hi - lo : 1.0;   // (a zero numerator takes the division's slow path)
    double f = 1.0;
    int n = 1;
    bool done = !size;
    for (int it = 0; it < 400; ++it) {
        const double m = floor(__ddiv_rn(ext, rl * f));
        const int nn = m < 1.0 ? 1 : (m > 1.0e6 ? 1000000 : (int)m);
        if (!done) n = nn;
        const long long prod = (long long)__shfl_sync(kFull, n, 0, 8) * __shfl_sync(kFull, n, 1, 8) * __shfl_sync(kFull, n, 2, 8);
        done |= prod <= cell_cap;
        if (__all_sync(kFull, done)) break;
        f *= 1.125;
    }
    const double quo = __ddiv_rn(ext, (double)n);
    if (size && sub < 3) {
        const double e = n == 1 ? (ext > rl ? ext : rl) : quo;
        g.origin[d] = lo;
        g.edge[d] = e;
        g.inv_edge[d] = 1.0 / e;
        g.edge_f[d] = (float)e;
        g.dims[d] = n;
    }
}

// Once per step, after every replica: counters, step number and, with the
// Verlet buffer, the rebuild decision and the graph condition.
template <bool SETCOND>
__device__ void finalize_step(const Params& p, int mode, long long next, unsigned maxd2)
{
    p.counters[3] = 0;
    if (mode & STEP_ADVANCE) *p.step = next;
    if (mode & STEP_KICK_DRIFT) *p.kick_full = 1;
    if constexpr (SETCOND) {
        p.counters[2] = 0;   // work counter of the force kernel (also reset by a build)
        // rebuild once some atom may have closed half of the skin: pairs
        // within r_cut now were within r_cut + skin at the build
        *p.maxd2 = 0u;
        int rebuild;
        if (p.lc) {
            // adaptive skin: the buffer stays only while lists live long enough to pay
            ListCtl& c = *p.lc;
            const int2 d = adapt_decision(p, maxd2);
            rebuild = d.x;
            if (d.y != c.buffered) {
                c.buffered = d.y;
                c.rlist_f = d.y ? p.rlist_f : p.rc_f;
                c.r_list = d.y ? p.r_list : p.r_cut;
                c.half_skin2 = d.y ? p.half_skin2 : 0.0f;
            }
            if (rebuild && !d.y) c.unbuffered_builds += 1;
            c.since_build = rebuild ? 0 : c.since_build + 1;
        } else {
            rebuild = maxd2 > __float_as_uint(p.half_skin2) ? 1 : 0;
        }
        p.builds[0] += rebuild;
        p.builds[1] = rebuild;
        cudaGraphSetConditional(p.cond, (unsigned)rebuild);
    }
}

// Smallest (largest) of the lanes' 64-bit keys: the high words by one warp
// reduction, then the low words of the lanes that hold it.
template <bool MAX>
__device__ __forceinline__ unsigned long long warp_extreme(unsigned long long v)
{
    constexpr unsigned kFull = 0xffffffffu;
    const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
    const unsigned h = MAX ? __reduce_max_sync(kFull, hi) : __reduce_min_sync(kFull, hi);
    const unsigned c = hi == h ? lo : (MAX ? 0u : 0xffffffffu);
    const unsigned l = MAX ? __reduce_max_sync(kFull, c) : __reduce_min_sync(kFull, c);
    return ((unsigned long long)h << 32) | l;
}

// Half kicks, Langevin update, drift and periodic wrap of atom i: (ax, ay, az)
// is the half kick's velocity increment.
__device__ __forceinline__ void kick_drift(const Params& p, const Grid& g, int r, int s, int i, long long step, int kick_full,
                                           double ax, double ay, double az, double& vx, double& vy, double& vz, double& x,
                                           double& y, double& z)
{
    // the state holds v_{n-1/2} once stepping has started: finish the
    // previous step's half kick, then this step's (two separate adds,
    // exactly as velocity Verlet rounds them)
    if (kick_full) { vx = vx + ax; vy = vy + ay; vz = vz + az; }
    vx = vx + ax; vy = vy + ay; vz = vz + az;
    if (p.langevin) {
        // electron-ion coupling (Eqs. 13-14): exact Ornstein-Uhlenbeck
        // update with Philox stream 1 of (seed, atom, step)
        const double2 cs = p.lgv[(size_t)r * kMaxSpecies + s];
        const unsigned long long sd = p.seed[r];
        const uint4 w4 = philox4x32_10(make_uint4((unsigned)p.local_id[i], (unsigned)step, 1u, 0u),
                                       make_uint2((unsigned)sd, (unsigned)(sd >> 32)));
        double gx, gy, gz;
        gauss3(w4, p.precision == 0, gx, gy, gz);
        vx = cs.x * vx + cs.y * gx;
        vy = cs.x * vy + cs.y * gy;
        vz = cs.x * vz + cs.y * gz;
    }
    // x + dt v with one rounding (GB300 issues FP64 at 2 lanes per SM per clock)
    x = __fma_rn(p.dt, vx, x);
    y = __fma_rn(p.dt, vy, y);
    z = __fma_rn(p.dt, vz, z);
    if (g.periodic) {
        // wrap only atoms that left the box (FP64 division is slow); the
        // tests run on the bit patterns
        const double L0 = g.box[0], L1 = g.box[1], L2 = g.box[2];
        if (below_zero(x) || at_or_above(x, L0)) { x -= L0 * floor(x / L0); if (x >= L0) x -= L0; }
        if (below_zero(y) || at_or_above(y, L1)) { y -= L1 * floor(y / L1); if (y >= L1) y -= L1; }
        if (below_zero(z) || at_or_above(z, L2)) { z -= L2 * floor(z / L2); if (z >= L2) z -= L2; }
    }
    // finite check on the exponent bits (integer ops; FP64 compares are slow here)
    if (((__double2hiint(x) & 0x7ff00000) == 0x7ff00000) || ((__double2hiint(y) & 0x7ff00000) == 0x7ff00000) ||
        ((__double2hiint(z) & 0x7ff00000) == 0x7ff00000) || ((__double2hiint(vx) & 0x7ff00000) == 0x7ff00000) ||
        ((__double2hiint(vy) & 0x7ff00000) == 0x7ff00000) || ((__double2hiint(vz) & 0x7ff00000) == 0x7ff00000))
        atomicOr(p.err, ERR_NONFINITE);
}

// Squared displacement since the last list build (minimum image) as the bits of
// an FP32 number: it only decides the rebuild, against half the skin.
// Non-negative floats order like their bit patterns (NaN sorts high).
__device__ __forceinline__ unsigned moved2(const Params& p, const Grid& g, int i, double x, double y, double z)
{
    double d[3] = {x - p.xr[i], y - p.yr[i], z - p.zr[i]};
    if (g.periodic)
        for (int k = 0; k < 3; ++k) {
            const int o = beyond_half(d[k], g.box[k]);
            if (o > 0) d[k] -= g.box[k];
            else if (o < 0) d[k] += g.box[k];
        }
    const float e0 = (float)d[0], e1 = (float)d[1], e2 = (float)d[2];
    return __float_as_uint(e0 * e0 + e1 * e1 + e2 * e2);
}

// Rates of one atom in type state ts (species s of nuclear charge Z, charge q)
// with K-hole flag h: the running sums of the four channels (Sec. II.A).
struct Rates {
    double a_pi, a_a, a_ci, a_rec, c1, c2, lam;
};
__device__ __forceinline__ Rates cr_rates(const Params& p, const RepState& st, double dF, int ts, int s, int Z, int q, int h)
{
    Rates x;
    x.a_pi = __dmul_rn(p.sigma_pi[2 * ts + h], dF);
    x.a_a = h ? p.auger_dt[s] : 0.0;
    x.a_ci = 0.0;
    x.a_rec = 0.0;
    if (q < Z) x.a_ci = __dmul_rn(st.ne_dt, interp(p.k_ci + (long long)ts * p.n_te, st.it0, st.wt));
    if (q > 0 && h == 0) x.a_rec = __dmul_rn(st.ne_dt, interp(p.k_rec + (long long)ts * p.n_te, st.it0, st.wt));
    x.c1 = __dadd_rn(x.a_pi, x.a_a);
    x.c2 = __dadd_rn(x.c1, x.a_ci);
    x.lam = __dadd_rn(x.c2, x.a_rec);
    return x;
}

// An FP32 number above the double whose high word is hi (infinity for what FP32
// cannot hold, infinities and NaN; its smallest normal number for what is smaller).
__device__ __forceinline__ float above_f(int hi)
{
    const int mag = hi & 0x7fffffff;
    if (mag >= 0x47e00000) return __int_as_float(0x7f800000);
    return hi < 0x38100000 ? 1.17549435e-38f : __uint_as_float((unsigned)hi * 8u + 0x40000008u);
}
__device__ __forceinline__ int hi_word(const double* a) { return reinterpret_cast<const int*>(a)[1]; }

// Whether u0 = u53(a, .) is certainly below 1 - e^{-lam} >= lam - lam^2 / 2 (lam > 0),
// which spares the exponential's forty FP64 operations but for the few atoms that
// draw a number between the two.
__device__ __forceinline__ bool sure_event(unsigned a, double lam)
{
    const int hi = __double2hiint(lam);
    const float lo_f = hi < 0x38100000 || hi >= 0x47e00000 ? 0.0f : __uint_as_float((unsigned)hi * 8u + 0x40000000u);
    const float t = __fmul_rn(lo_f, __fmul_rn(__fsub_rn(1.0f, __fmul_rn(0.5f, above_f(hi))), 0.999998f));
    return __fmul_rn(__uint2float_ru((a >> 5) + 1u), 7.4505806e-9f) < t;
}

// An upper bound of cr_rates' total rate in FP32: the interpolated coefficients
// are at most the larger of their two table values.  GB300's FP64 pipe takes 16
// cycles of the SM per warp instruction, and the bound rules an event out for
// all but the few atoms that draw a number near or below their rate.
__device__ __forceinline__ float cr_bound(const Params& p, const RepState& st, double dF, int ts, int s, int Z, int q, int h)
{
    float b = __fmul_rn(above_f(hi_word(p.sigma_pi + 2 * ts + h)), above_f(__double2hiint(dF)));
    if (h) b = __fadd_rn(b, above_f(hi_word(p.auger_dt + s)));
    float k = 0.0f;
    if (q < Z) {
        const double* K = p.k_ci + (long long)ts * p.n_te + st.it0;
        k = above_f(max(hi_word(K), hi_word(K + 1)));
    }
    if (q > 0 && h == 0) {
        const double* K = p.k_rec + (long long)ts * p.n_te + st.it0;
        k = __fadd_rn(k, above_f(max(hi_word(K), hi_word(K + 1))));
    }
    return __fmul_rn(__fadd_rn(b, __fmul_rn(k, above_f(__double2hiint(st.ne_dt)))), 1.000001f);
}

// a < b for non-negative doubles, in the integer pipe: their order is that of
// their bit patterns.
__device__ __forceinline__ bool below(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }

// The channel that t, uniform in [0, lam), falls into: 0 PI, 1 Auger, 2 CI, 3 REC.
__device__ __forceinline__ int cr_channel(const Rates& x, double t)
{
    if (below(t, x.a_pi)) return 0;
    if (below(t, x.c1)) return 1;
    if (below(t, x.c2)) return 2;
    if (below(t, x.lam)) return 3;
    return x.a_rec > 0.0 ? 3 : (x.a_ci > 0.0 ? 2 : (x.a_a > 0.0 ? 1 : 0));
}

// Applies an event of channel ch to (q, h) of type state ts; returns the energy
// given to the electron gas (meV).
__device__ __forceinline__ long long cr_event(const Params& p, int ch, int ts, int s, int Z, int& q, int& h)
{
    long long de;
    if (ch == 0) {
        de = p.e_pi_mev[2 * ts + h];
        q += 1;
        if (q == Z) h = 0;
        else if (Z >= 3 && h == 0 && Z - q >= 2) h = 1;
    } else if (ch == 1) {
        q += 1;
        h = 0;
        de = p.e_auger_mev[s];
    } else if (ch == 2) {
        q += 1;
        if (q == Z) h = 0;
        de = -p.ip_mev[ts];
    } else {
        q -= 1;
        de = p.ip_mev[ts - 1];
    }
    return de;
}

// The running sums of the rates of every (replica, type state, K-hole flag) at the
// step about to be taken, for the step kernel of large systems: an atom then tests
// its uniform against one table entry (the same expressions, so the same values).
__global__ void __launch_bounds__(128) k_rates(Params p)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= p.n_rep * p.n_ts * 2) return;
    const int r = k / (2 * p.n_ts), h = k & 1, ts = (k >> 1) % p.n_ts;
    int s = 0;
    while (s + 1 < p.n_species && ts >= p.ts_off[s + 1]) ++s;
    const long long step = *p.step;
    const double dF = step < p.max_steps ? p.dF[(long long)r * p.max_steps + step] : 0.0;
    const Rates x = cr_rates(p, p.rs[r], dF, ts, s, p.zs[s], ts - p.ts_off[s], h);
    double* t = p.rate_tab + 4ll * k;
    t[0] = x.a_pi; t[1] = x.c1; t[2] = x.c2; t[3] = x.lam;
}

// Bounding box of the vacuum replicas' atoms into the block's window of replicas
// from r0 (whole warps; one atom per lane; vac: the lane's atom counts).  ONE: no
// other warp of the block writes the window.  A replica at a time, reduced in the
// warp: 64-bit minima and maxima in shared memory are compare-and-swap loops, and
// 28 lanes of a last block contending for six of them took 3 us.
template <bool ONE>
__device__ __forceinline__ void box_update(const Params& p, int r, int r0, bool vac, const double pos[3],
                                           unsigned long long (*s_bmin)[3], unsigned long long (*s_bmax)[3])
{
    constexpr unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(kFull, vac);
    while (todo) {
        const int r1 = __shfl_sync(kFull, r, __ffs(todo) - 1);
        const bool in = vac && r == r1;
        todo &= ~__ballot_sync(kFull, in);
        unsigned long long v = 0ull;   // lane d: lower end of dimension d, lane 3 + d: upper end
        for (int d = 0; d < 3; ++d) {
            const unsigned long long key = ordered_bits(pos[d]);
            const unsigned long long mn = warp_extreme<false>(in ? key : ~0ull), mx = warp_extreme<true>(in ? key : 0ull);
            if (lane == d) v = mn;
            if (lane == 3 + d) v = mx;
        }
        if (lane < 6) {
            const int w = r1 - r0, d = lane < 3 ? lane : lane - 3;
            RepAccum* a = p.acc + (size_t)r1 * kAccCopies + (blockIdx.x & (kAccCopies - 1));
            const bool win = w < kRepWindow;
            unsigned long long* dst = lane < 3 ? (win ? &s_bmin[w][d] : &a->bmin[d]) : (win ? &s_bmax[w][d] : &a->bmax[d]);
            if (ONE && win) *dst = v;
            else if (lane < 3) atomicMin(dst, v);
            else atomicMax(dst, v);
        }
    }
}

// The block's sums and boxes of replicas r0 .. r0 + nw - 1 into the accumulators,
// by threads t of n_t.
__device__ __forceinline__ void flush_block(const Params& p, int r0, int nw, long long (*s_acc)[6],
                                            unsigned long long (*s_bmin)[3], unsigned long long (*s_bmax)[3], int t, int n_t)
{
    for (int k = t; k < nw * 12; k += n_t) {
        const int w = k / 12, f = k % 12;
        RepAccum* a = p.acc + (size_t)(r0 + w) * kAccCopies + (blockIdx.x & (kAccCopies - 1));
        if (f < 6) {
            const long long v = s_acc[w][f];
            if (v != 0) {
                unsigned long long* dst = f == 0 ? (unsigned long long*)&a->dNe
                                        : f == 1 ? (unsigned long long*)&a->dE
                                                 : (unsigned long long*)&a->counts[f - 2];
                atomicAdd(dst, (unsigned long long)v);
            }
        } else if (f < 9) {
            if (s_bmin[w][f - 6] != ~0ull) atomicMin(&a->bmin[f - 6], s_bmin[w][f - 6]);
        } else {
            if (s_bmax[w][f - 9] != 0ull) atomicMax(&a->bmax[f - 9], s_bmax[w][f - 9]);
        }
    }
}

// The full step of large systems with rates: a thread does an atom's kick, drift,
// charge update (against the table of total rates) and re-pack, with all of its
// loads issued before the first use and no barrier in between; k_step_fin
// reduces the replicas.  Two threads per atom (k_step_a) shorten the chain of a
// system that leaves the chip idle, but with many blocks per SM the instructions
// count: FP64 runs at 2 lanes per SM and clock here, and evaluating the rates and
// 1 - e^{-lam} was most of the charge role's work, for an event in one atom of some
// tens.  2 M-atom droplet: 302.6 us -> 126 + 4.0 (k_rates) + 6.7 us (k_step_fin),
// 3.8 TB/s of state (203 us before sure_event); 1,024 x 1,500 methane: 188.1 + 16.3
// -> 90.5 + 4.1 + 8.1 us; 199,773 atoms 46.6 -> 24.6 + 2.7 + 5.7.  Blocks of 64
// atoms took 1 % less than 128.
constexpr int kWideAtoms = 64;
__global__ void __launch_bounds__(kWideAtoms, 16) k_step_wide(Params p)
{
    __shared__ long long s_acc[kRepWindow][6];
    __shared__ unsigned long long s_bmin[kRepWindow][3], s_bmax[kRepWindow][3];
    const int tid = threadIdx.x, lane = tid & 31;
    const int first = blockIdx.x * kWideAtoms;
    const int last = min(first + kWideAtoms, p.n_atoms) - 1;
    const int i = min(first + tid, last);
    const bool live = first + tid <= last;
    const unsigned err = *p.err;
    const long long step = *p.step;
    const int kick_full = *p.kick_full;
    const int r0 = p.rep[first], r_last = p.rep[last], r = p.rep[i];
    const int s = p.species[i], slot = p.slot_of[i], qi = p.q[i], hi = p.h[i], fr = p.frag[i], loc = p.local_id[i];
    double x = p.x[i], y = p.y[i], z = p.z[i];
    double vx = p.vx[i], vy = p.vy[i], vz = p.vz[i];
    const bool repack = p.xr != nullptr;
    double4_32a cen = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    if (repack) cen = p.cl_cen[slot / kClusterSize];
    double ax, ay, az;
    half_kick(p, s, slot, ax, ay, az);
    const int Z = p.zs[s], ts = p.ts_off[s] + qi;
    const unsigned long long sd = p.seed[r];
    const double* tab = p.rate_tab + (((long long)r * p.n_ts + ts) * 2 + hi) * 4;
    const double lam = tab[3];
    const Grid& g = p.grid[r];
    const int nw = min(r_last - r0 + 1, kRepWindow);
    for (int k = tid; k < nw * 6; k += kWideAtoms) (&s_acc[0][0])[k] = 0;
    for (int k = tid; k < nw * 3; k += kWideAtoms) {
        (&s_bmin[0][0])[k] = ~0ull;
        (&s_bmax[0][0])[k] = 0ull;
    }
    // a cluster-pair list overflow freezes the state (see k_step_a)
    if (err & ERR_LIST) return;
    __syncthreads();
    unsigned d2_bits = 0u;
    double pos[3] = {0.0, 0.0, 0.0};
    if (live) {
        kick_drift(p, g, r, s, i, step, kick_full, ax, ay, az, vx, vy, vz, x, y, z);
        if (repack) d2_bits = moved2(p, g, i, x, y, z);
        p.vx[i] = vx; p.vy[i] = vy; p.vz[i] = vz;
        p.x[i] = x; p.y[i] = y; p.z[i] = z;
        pos[0] = x; pos[1] = y; pos[2] = z;
        int qn = qi;
        if (step >= p.max_steps) atomicOr(p.err, ERR_TABLE_END);
        // the tests of k_step_a, on the table's total rate
        if (below(0.0, lam)) {
            const uint4 w4 = philox4x32_10(make_uint4((unsigned)loc, (unsigned)step, 0u, 0u),
                                           make_uint2((unsigned)sd, (unsigned)(sd >> 32)));
            const double u0 = u53(w4.x, w4.y);
            if (below(u0, lam) &&
                (sure_event(w4.x, lam) || u0 < one_minus_exp_neg(lam, p.etab, p.inv12))) {
                const double t = __dmul_rn(u53(w4.z, w4.w), lam);
                int ch = below(t, tab[0]) ? 0 : (below(t, tab[1]) ? 1 : (below(t, tab[2]) ? 2 : 3));
                if (!below(t, lam)) {   // t rounded up to lam
                    const double dF = step < p.max_steps ? p.dF[(long long)r * p.max_steps + step] : 0.0;
                    ch = cr_channel(cr_rates(p, p.rs[r], dF, ts, s, Z, qi, hi), t);
                }
                int hn = hi;
                const long long de = cr_event(p, ch, ts, s, Z, qn, hn);
                p.q[i] = (uint8_t)qn;
                p.h[i] = (uint8_t)hn;
                const int w = r - r0;
                unsigned long long* acc[3];
                if (w < kRepWindow) {
                    acc[0] = (unsigned long long*)&s_acc[w][0];
                    acc[1] = (unsigned long long*)&s_acc[w][1];
                    acc[2] = (unsigned long long*)&s_acc[w][2 + ch];
                } else {
                    RepAccum* a = p.acc + (size_t)r * kAccCopies + (blockIdx.x & (kAccCopies - 1));
                    acc[0] = (unsigned long long*)&a->dNe;
                    acc[1] = (unsigned long long*)&a->dE;
                    acc[2] = (unsigned long long*)&a->counts[ch];
                }
                atomicAdd(acc[0], (unsigned long long)(ch == 3 ? -1ll : 1ll));
                atomicAdd(acc[1], (unsigned long long)de);
                atomicAdd(acc[2], 1ull);
            }
        }
        if (repack) {
            const Grid& gb = p.grid_b[r];
            const double c[3] = {cen.x, cen.y, cen.z};
            pack_record(p, slot, pos, c, gb.periodic, gb.box, s, qn, fr);
        }
    }
    if (repack) {
        const unsigned m = __reduce_max_sync(0xffffffffu, d2_bits);
        if (lane == 0 && m) atomicMax(p.maxd2, m);
    }
    box_update<false>(p, r, r0, live && !g.periodic, pos, s_bmin, s_bmax);
    __syncthreads();
    flush_block(p, r0, nw, s_acc, s_bmin, s_bmax, tid, kWideAtoms);
}

// SETCOND: the Verlet-buffered variant that decides the rebuild and sets the
// graph condition (ncu does not profile kernels that can set one, so the
// every-step variant is a separate instantiation).  MINB: resident blocks per
// SM the registers are sized for; 16 (64 registers) for grids of many blocks
// per SM, where the FP64 pipe binds and more resident warps pay (2 M-atom
// droplet: 3.80 -> 3.71 ms per step); 10 (96 registers) for small grids, which
// are latency-bound (water box: 108.4 against 110.9 us per step with 16)
template <bool SETCOND, int MINB, bool FIN>
__global__ void __launch_bounds__(kStepThreads, MINB) k_step_a(Params p, int mode)
{
    __shared__ long long s_acc[kRepWindow][6];
    __shared__ unsigned long long s_bmin[kRepWindow][3], s_bmax[kRepWindow][3];
    __shared__ int s_last;
    __shared__ unsigned s_maxd2;
    __shared__ uint8_t s_q[kStepAtoms];   // charges after this step's update (charge-update warp)
    // a cluster-pair list overflow freezes the state at the step whose forces
    // are missing; the host grows the list, recomputes them and resumes
    if (*p.err & ERR_LIST) return;
    const int tid = threadIdx.x;
    const long long step = *p.step;
    const int kick_full = *p.kick_full;
    // the first kStepAtoms threads kick, drift and re-pack atoms first ..
    // first + kStepAtoms - 1; the others run the charge update of the same
    // atoms (independent until the re-pack)
    const bool cr_role = tid >= kStepAtoms;
    const int first = blockIdx.x * kStepAtoms;
    const int r0 = p.rep[first], r_last = p.rep[min(first + kStepAtoms, p.n_atoms) - 1];
    const int i = first + (tid & (kStepAtoms - 1));
    const bool live = i < p.n_atoms;
    const int lane = tid & 31;
    int r = live ? p.rep[i] : -1;
    double pos[3] = {0.0, 0.0, 0.0};
    bool vac = false;
    unsigned d2_bits = 0u;   // squared displacement since the last build
    // inputs of this atom's re-pack (Verlet-buffered list), loaded before the
    // charge update is waited for
    const bool repack = live && !cr_role && p.xr && (mode & STEP_KICK_DRIFT);
    int pk_slot = 0, pk_sp = 0, pk_fr = 0, pk_q = 0, pk_per = 0;
    double pk_cen[3] = {0.0, 0.0, 0.0}, pk_box[3] = {0.0, 0.0, 0.0};

    if (live && !cr_role) {
        const int s = p.species[i];
        double x = p.x[i], y = p.y[i], z = p.z[i];
        if (repack) {
            pk_slot = p.slot_of[i];
            const double4_32a c = p.cl_cen[pk_slot / kClusterSize];
            pk_cen[0] = c.x; pk_cen[1] = c.y; pk_cen[2] = c.z;
            const Grid& gb = p.grid_b[r];
            pk_per = gb.periodic;
            pk_box[0] = gb.box[0]; pk_box[1] = gb.box[1]; pk_box[2] = gb.box[2];
            pk_sp = s;
            pk_fr = p.frag[i];
            pk_q = p.q[i];
        }
        if (mode & STEP_KICK_DRIFT) {
            double ax, ay, az;
            half_kick(p, s, p.slot_of[i], ax, ay, az);
            double vx = p.vx[i], vy = p.vy[i], vz = p.vz[i];
            const Grid& g = p.grid[r];
            kick_drift(p, g, r, s, i, step, kick_full, ax, ay, az, vx, vy, vz, x, y, z);
            p.vx[i] = vx; p.vy[i] = vy; p.vz[i] = vz;
            p.x[i] = x; p.y[i] = y; p.z[i] = z;
            if (p.xr) {
                d2_bits = moved2(p, g, i, x, y, z);
            }
        }
        pos[0] = x; pos[1] = y; pos[2] = z;
        vac = !p.grid[r].periodic;
    }

    // ---- bounding box of vacuum replicas; each warp clears the sums it writes ----
    if (!cr_role) {
        unsigned m = 0u;
        if (p.xr && (mode & STEP_KICK_DRIFT)) m = __reduce_max_sync(0xffffffffu, d2_bits);
        if (lane == 0) s_maxd2 = m;
        for (int k = lane; k < kRepWindow * 3; k += 32) {
            (&s_bmin[0][0])[k] = ~0ull;
            (&s_bmax[0][0])[k] = 0ull;
        }
        __syncwarp();
        box_update<true>(p, r, r0, vac, pos, s_bmin, s_bmax);
    } else {
        for (int k = lane; k < kRepWindow * 6; k += 32) (&s_acc[0][0])[k] = 0;
        __syncwarp();
    }

    // ---- collisional-radiative update (reading of Sec. II.A) ----
    if (live && cr_role && (mode & STEP_CR) && p.charge_mode == kChargeTable) {
        // charges from the CR charge-state fractions (reading of Sec. II.A): the
        // atom's fixed quantile u (Philox stream 2) against the running sums of
        // its species at the end of this step (table row step + 1)
        const int s = p.species[i];
        const int Z = p.zs[s];
        const int qi = p.q[i];
        int qn = qi;
        if (step < p.max_steps) {
            const double* cum = p.qcum + ((size_t)r * (p.max_steps + 1) + (size_t)(step + 1)) * p.n_ts + p.ts_off[s];
            const unsigned long long sd = p.seed[r];
            const uint4 w4 = philox4x32_10(make_uint4((unsigned)p.local_id[i], 0u, 2u, 0u),
                                           make_uint2((unsigned)sd, (unsigned)(sd >> 32)));
            const double u = u53(w4.x, w4.y);
            qn = Z;
            for (int k = 0; k <= Z; ++k)
                if (u < cum[k]) { qn = k; break; }
        } else {
            atomicOr(p.err, ERR_TABLE_END);
        }
        s_q[i - first] = (uint8_t)qn;
        if (qn != qi || p.h[i]) {
            p.q[i] = (uint8_t)qn;
            p.h[i] = 0;
        }
        const int dq = qn - qi;
        if (dq != 0) {
            const int w = r - r0;
            const unsigned long long up = (unsigned long long)(dq > 0 ? dq : -dq);
            if (w < kRepWindow) {
                atomicAdd((unsigned long long*)&s_acc[w][0], (unsigned long long)(long long)dq);
                atomicAdd((unsigned long long*)&s_acc[w][dq > 0 ? 2 : 5], up);
            } else {
                RepAccum* a = p.acc + (size_t)r * kAccCopies + (blockIdx.x & (kAccCopies - 1));
                atomicAdd((unsigned long long*)&a->dNe, (unsigned long long)(long long)dq);
                atomicAdd((unsigned long long*)&a->counts[dq > 0 ? 0 : 3], up);
            }
        }
    }
    if (live && cr_role && (mode & STEP_CR) && p.charge_mode != kChargeTable) {
        const int s = p.species[i];
        const int Z = p.zs[s];
        const int qi = p.q[i], hi = p.h[i];
        s_q[i - first] = (uint8_t)qi;   // replaced below if an event changes it
        const int ts = p.ts_off[s] + qi;
        if (step >= p.max_steps) atomicOr(p.err, ERR_TABLE_END);
        const double dF = step < p.max_steps ? p.dF[(long long)r * p.max_steps + step] : 0.0;
        const RepState& rs = p.rs[r];
        int ch = -1;
        const unsigned long long sd = p.seed[r];
        const uint4 w4 = philox4x32_10(make_uint4((unsigned)p.local_id[i], (unsigned)step, 0u, 0u),
                                       make_uint2((unsigned)sd, (unsigned)(sd >> 32)));
        // u0 = u53(w4.x, w4.y) has w4.x >> 5 as its leading 27 bits; 1 - e^{-lam} <=
        // lam, so u0 >= lam, and u0 above a bound of lam, decide "no event" exactly
        if (!(__fmul_rn(__uint2float_rz(w4.x >> 5), 7.4505806e-9f) > cr_bound(p, rs, dF, ts, s, Z, qi, hi))) {
            const Rates x = cr_rates(p, rs, dF, ts, s, Z, qi, hi);
            const double u0 = u53(w4.x, w4.y);
            if (below(0.0, x.lam) && below(u0, x.lam) &&
                (sure_event(w4.x, x.lam) || u0 < one_minus_exp_neg(x.lam, p.etab, p.inv12))) {
                ch = cr_channel(x, __dmul_rn(u53(w4.z, w4.w), x.lam));
            }
        }
        if (ch >= 0) {
            int qn = qi, hn = hi;
            const long long de = cr_event(p, ch, ts, s, Z, qn, hn);
            p.q[i] = (uint8_t)qn;
            p.h[i] = (uint8_t)hn;
            s_q[i - first] = (uint8_t)qn;
            const int w = r - r0;
            if (w < kRepWindow) {
                atomicAdd((unsigned long long*)&s_acc[w][0], (unsigned long long)(ch == 3 ? -1ll : 1ll));
                atomicAdd((unsigned long long*)&s_acc[w][1], (unsigned long long)de);
                atomicAdd((unsigned long long*)&s_acc[w][2 + ch], 1ull);
            } else {
                RepAccum* a = p.acc + (size_t)r * kAccCopies + (blockIdx.x & (kAccCopies - 1));
                atomicAdd((unsigned long long*)&a->dNe, (unsigned long long)(ch == 3 ? -1ll : 1ll));
                atomicAdd((unsigned long long*)&a->dE, (unsigned long long)de);
                atomicAdd((unsigned long long*)&a->counts[ch], 1ull);
            }
        }
    }
    // ---- Verlet-buffered list: the packed record of this atom for the forces
    // of this step, in the slot of the last build (a build, if one follows,
    // rewrites all records); the force sums are cleared after the kick read them
    __syncthreads();   // the charges of this step, the boxes and the sums are written
    if (repack) {
        const int qi = (mode & STEP_CR) ? (int)s_q[i - first] : pk_q;
        pack_record(p, pk_slot, pos, pk_cen, pk_per, pk_box, pk_sp, qi, pk_fr);
    }

    // ---- flush block partials: by the charge-update warp, whose fence then waits
    // for no record on its way to memory ----
    if (cr_role) {
        flush_block(p, r0, min(r_last - r0 + 1, kRepWindow), s_acc, s_bmin, s_bmax, lane, 32);
        if (lane == 0 && s_maxd2) atomicMax(p.maxd2, s_maxd2);
    }

    // ---- per-replica reduction (Eq. 3) and next grid: by this kernel's last
    // block for a few replicas, by k_step_fin for more ----
    if constexpr (FIN) return;
    if (cr_role) {
        __threadfence();
        __syncwarp();
        if (lane == 0) s_last = (atomicAdd(&p.counters[3], 1) == (int)gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const long long next = (mode & STEP_ADVANCE) ? step + 1 : step;
    if (cr_role) {
        finalize_plasma(p, 0, p.n_rep, lane, next);
    } else {
        const unsigned m2 = SETCOND ? __ldcg(p.maxd2) : 0u;
        finalize_grid(p, 0, p.n_rep, lane, next_rlist<SETCOND>(p, m2));
        __syncwarp();
        if (lane == 0) finalize_step<SETCOND>(p, mode, next, m2);
    }
}

// Per-replica reduction when there are many replicas: two warps each, then the
// last block finishes the step.
template <bool SETCOND>
__global__ void __launch_bounds__(256) k_step_fin(Params p, int mode)
{
    __shared__ int s_last;
    if (*p.err & ERR_LIST) return;
    const int tid = threadIdx.x, lane = tid & 31;
    const long long step = *p.step;
    const long long next = (mode & STEP_ADVANCE) ? step + 1 : step;
    const int gw = (blockIdx.x * blockDim.x + tid) >> 5, rr = gw >> 1;
    if (rr < p.n_rep) {
        // every block reads maxd2 and the list state before the last one records the decision
        if (gw & 1) finalize_grid(p, rr, 1, lane, next_rlist<SETCOND>(p, SETCOND ? __ldcg(p.maxd2) : 0u));
        else finalize_plasma(p, rr, 1, lane, next);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&p.counters[3], 1) == (int)gridDim.x - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) finalize_step<SETCOND>(p, mode, next, SETCOND ? __ldcg(p.maxd2) : 0u);
}

static int sm_count()
{
    int d = 0, n = 0;
    if (cudaGetDevice(&d) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, d) != cudaSuccess)
        return 1;
    return n > 0 ? n : 1;
}

void launch_step_a(const Params& p, int mode, cudaStream_t s, int grid_atoms)
{
    (void)grid_atoms;
    static const int n_sm = sm_count();
    constexpr int kWide = kWideBlocks;   // MINB of the variant for grids of many blocks per SM
    const int blocks = (p.n_atoms + kStepAtoms - 1) / kStepAtoms;
    const int fin_blocks = (p.n_rep * 64 + 255) / 256;
    const bool wide = step_is_wide(p.n_atoms, n_sm);
    const bool full = wide && (mode & STEP_KICK_DRIFT) && (mode & STEP_CR) && p.charge_mode != kChargeTable && p.rate_tab;
    const bool fin = wide || p.n_rep > kInlineReps;
    const bool cond = (mode & STEP_SETCOND) != 0;
    if (full) {
        k_rates<<<(p.n_rep * p.n_ts * 2 + 127) / 128, 128, 0, s>>>(p);
        k_step_wide<<<(p.n_atoms + kWideAtoms - 1) / kWideAtoms, kWideAtoms, 0, s>>>(p);
    } else if (wide) {
        k_step_a<false, kWide, true><<<blocks, kStepThreads, 0, s>>>(p, mode);
    } else if (fin) {
        k_step_a<false, 10, true><<<blocks, kStepThreads, 0, s>>>(p, mode);
    } else if (cond) {
        k_step_a<true, 10, false><<<blocks, kStepThreads, 0, s>>>(p, mode);
    } else {
        k_step_a<false, 10, false><<<blocks, kStepThreads, 0, s>>>(p, mode);
    }
    if (fin) {
        if (cond) k_step_fin<true><<<fin_blocks, 256, 0, s>>>(p, mode);
        else k_step_fin<false><<<fin_blocks, 256, 0, s>>>(p, mode);
    }
}

// ---------------------------------------------------------------------------
// Velocities at the integer step (state stores v_{n+1/2} once stepping has
// started), forces in kJ/mol/nm, kinetic energy, Philox diagnostic.
// ---------------------------------------------------------------------------
__global__ void k_velocity_out(Params p, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.n_atoms) return;
    const int full = *p.kick_full;
    double vx = p.vx[i], vy = p.vy[i], vz = p.vz[i];
    if (full) {
        double ax, ay, az;
        half_kick(p, p.species[i], p.slot_of[i], ax, ay, az);
        vx = vx + ax; vy = vy + ay; vz = vz + az;
    }
    out[3 * i + 0] = vx;
    out[3 * i + 1] = vy;
    out[3 * i + 2] = vz;
}

__global__ void k_force_out(Params p, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.n_atoms) return;
    const int slot = p.slot_of[i];
    out[3 * i + 0] = (double)p.fx[slot] * kFixInv;
    out[3 * i + 1] = (double)p.fy[slot] * kFixInv;
    out[3 * i + 2] = (double)p.fz[slot] * kFixInv;
}

// ---------------------------------------------------------------------------
// State exchange: the caller's arrays of structures (x y z per atom) are copied
// as they are and split or joined here, next to their check.  Bound by memory;
// doing the same on the host cost 25 ms to restore and 13 ms to read a state of
// 2 M atoms, these take 0.03 ms per field.  The copies take 0.25 ms a field from and
// into host memory that is pinned or already mapped; a read into arrays fresh from the
// allocator adds the host's page faults, 3.9 ms for positions and velocities (0.57 ->
// 4.45 ms).
// A check that fails sets its bit in *bad; the kernels that would write the
// state afterwards then do nothing.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

__global__ void __launch_bounds__(256) k_check_vectors(const double* __restrict__ a, int n, unsigned* bad, unsigned bit)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (!finite_bits(a[3 * (size_t)i]) || !finite_bits(a[3 * (size_t)i + 1]) || !finite_bits(a[3 * (size_t)i + 2]))
        atomicOr(bad, bit);
}

__global__ void __launch_bounds__(256) k_split_vectors(const double* __restrict__ a, int n, double* x, double* y, double* z,
                                                       const unsigned* bad, int* flag)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || *bad) return;
    if (flag && i == 0) *flag = 0;
    x[i] = a[3 * (size_t)i];
    y[i] = a[3 * (size_t)i + 1];
    z[i] = a[3 * (size_t)i + 2];
}

__global__ void __launch_bounds__(256) k_join_vectors(const double* __restrict__ x, const double* __restrict__ y,
                                                      const double* __restrict__ z, int n, double* a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    a[3 * (size_t)i] = x[i];
    a[3 * (size_t)i + 1] = y[i];
    a[3 * (size_t)i + 2] = z[i];
}

// charges up to Z (zs given) or K-hole flags up to 1 (zs null)
__global__ void __launch_bounds__(256) k_check_bytes(const uint8_t* __restrict__ a, int n, const uint8_t* species, const int* zs,
                                                     unsigned* bad, unsigned bit)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if ((int)a[i] > (zs ? zs[species[i]] : 1)) atomicOr(bad, bit);
}

__global__ void __launch_bounds__(256) k_store_bytes(const uint8_t* __restrict__ a, int n, uint8_t* dst, const unsigned* bad)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && !*bad) dst[i] = a[i];
}

void launch_store_vectors(const double* a, int n, double* const dst[3], unsigned* bad, unsigned bit, cudaStream_t s,
                          int* flag)
{
    const int blocks = (n + 255) / 256;
    if (bit) k_check_vectors<<<blocks, 256, 0, s>>>(a, n, bad, bit);
    k_split_vectors<<<blocks, 256, 0, s>>>(a, n, dst[0], dst[1], dst[2], bad, flag);
}
void launch_join_vectors(const double* const src[3], int n, double* a, cudaStream_t s)
{
    k_join_vectors<<<(n + 255) / 256, 256, 0, s>>>(src[0], src[1], src[2], n, a);
}
void launch_store_bytes(const uint8_t* a, int n, uint8_t* dst, const uint8_t* species, const int* zs, unsigned* bad, unsigned bit,
                        cudaStream_t s)
{
    const int blocks = (n + 255) / 256;
    k_check_bytes<<<blocks, 256, 0, s>>>(a, n, species, zs, bad, bit);
    k_store_bytes<<<blocks, 256, 0, s>>>(a, n, dst, bad);
}

// Kinetic and potential energy, in two passes whose grouping depends only on a
// replica's own size (deterministic sums, a replica alone equals its slot in a
// batch): blocks of kEnergyAtoms atoms, then a block per replica over their
// sums.  Bound by memory (about 60 bytes per atom, the slot gathers through
// L2); one block per replica left all but one SM idle: 3,950 us for a million
// atoms in one replica, 26 us in blocks of 1,024 atoms.  A replica of one block has
// its energies from the first pass, and where all are such the second is not
// launched.
__global__ void __launch_bounds__(256) k_energy_parts(Params p, const int4* part, double* ekin_part, long long* epot_part,
                                                      double* ekin, long long* epot)
{
    __shared__ double s_k[256];
    __shared__ long long s_u[256];
    const int4 me = part[blockIdx.x];   // (first atom, one past the last, replica, the replica's only block)
    const int a0 = me.x, a1 = me.y, r = me.z;
    const int full = *p.kick_full;
    double k = 0.0;
    long long u = 0;
    for (int i = a0 + threadIdx.x; i < a1; i += blockDim.x) {
        const int slot = p.slot_of[i];
        const int s = p.species[i];
        double vx = p.vx[i], vy = p.vy[i], vz = p.vz[i];
        if (full) {
            double ax, ay, az;
            half_kick(p, s, slot, ax, ay, az);
            vx = vx + ax; vy = vy + ay; vz = vz + az;
        }
        k += 0.5 * p.mass[s] * (vx * vx + vy * vy + vz * vz);
        u += p.epot[slot];
    }
    s_k[threadIdx.x] = k;
    s_u[threadIdx.x] = u;
    __syncthreads();
    for (int o = blockDim.x / 2; o; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s_k[threadIdx.x] += s_k[threadIdx.x + o];
            s_u[threadIdx.x] += s_u[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const bool whole = me.w != 0;
        *(whole ? ekin + r : ekin_part + blockIdx.x) = s_k[0];
        *(whole ? epot + r : epot_part + blockIdx.x) = s_u[0];
    }
}

__global__ void __launch_bounds__(256) k_energy_sum(const int* part_off, const double* ekin_part, const long long* epot_part,
                                                    double* ekin, long long* epot)
{
    __shared__ double s_k[256];
    __shared__ long long s_u[256];
    const int r = blockIdx.x;
    if (part_off[r + 1] - part_off[r] == 1) return;
    double k = 0.0;
    long long u = 0;
    for (int b = part_off[r] + threadIdx.x; b < part_off[r + 1]; b += blockDim.x) {
        k += ekin_part[b];
        u += epot_part[b];
    }
    s_k[threadIdx.x] = k;
    s_u[threadIdx.x] = u;
    __syncthreads();
    for (int o = blockDim.x / 2; o; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s_k[threadIdx.x] += s_k[threadIdx.x + o];
            s_u[threadIdx.x] += s_u[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        ekin[r] = s_k[0];
        epot[r] = s_u[0];
    }
}

__global__ void k_philox(unsigned long long seed, const uint4* ctr, long long n, uint4* out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = philox4x32_10(ctr[i], make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
}

void launch_velocity_out(const Params& p, double* d_v_out, cudaStream_t s)
{
    k_velocity_out<<<(p.n_atoms + 255) / 256, 256, 0, s>>>(p, d_v_out);
}
void launch_force_out(const Params& p, double* d_f_out, cudaStream_t s)
{
    k_force_out<<<(p.n_atoms + 255) / 256, 256, 0, s>>>(p, d_f_out);
}
void launch_energy(const Params& p, int n_parts, const int4* part, const int* part_off, double* ekin_part,
                   long long* epot_part, double* d_ekin, long long* d_epot, cudaStream_t s)
{
    k_energy_parts<<<n_parts, 256, 0, s>>>(p, part, ekin_part, epot_part, d_ekin, d_epot);
    if (n_parts > p.n_rep) k_energy_sum<<<p.n_rep, 256, 0, s>>>(part_off, ekin_part, epot_part, d_ekin, d_epot);
}
void launch_philox(unsigned long long seed, const uint32_t* ctr, long long n, uint32_t* out,
                   cudaStream_t s)
{
    if (n <= 0) return;
    const long long blocks = (n + 255) / 256;
    k_philox<<<(unsigned)blocks, 256, 0, s>>>(seed, (const uint4*)ctr, n, (uint4*)out);
}

}  // namespace mdg
