// Residual / FD-JVP stencil of the FMA build with the face fluxes on 64-bit fixed
// point (fixed.cuh), included by stencil_impl.cuh inside its namespace.
//
// The binary64 form of this kernel is bound by FP64 issue: 271 FP64
// instructions a cell, 86 % of the pipe.  Here the reconstruction and Roe's flux
// of every face run on the integer pipe.  FP64 keeps what needs a floating
// range: the state y + sum c_t add_t, the primitives, the viscous terms, the cell
// balance and the epilogue (about 100 instructions a cell with viscous terms),
// which overlap with it.  Measured (us), binary64 form -> this: residual 148 -> 75 at
// 512^2 (Navier-Stokes), 26.6 -> 7.7 at 64^2 (Euler), 132 -> 58 on the 256 x 512
// O-grid (Sutherland's law); FD-JVP 563 -> 293 at 1024^2.  At 512^2 the FP64 pipe is busy
// 60 % of the time and the integer ALU 35 %; the rest is latency of the dependent
// chains at 24 warps an SM.
//
// Units.  Every face is scaled by powers of two that its own cells set, so that
// its result depends neither on the tile it is computed in nor on the rest of
// the grid: R for densities (the largest of the four cells in [1/4, 1/2) R), U
// for sound speeds (the largest pressure in [2^-7, 2^-5) R U^2, and all
// velocities below U / 2), and for the normal and the tangential velocity each a
// unit U 2^-kn, U 2^-kt in which the largest of the four cells is in
// [1/8, 1/4) (k at least 0).  Mass and energy flux and the normal
// velocity's part of the dissipation are linear in the normal velocity and in
// dp / c; they are formed in U 2^-kf, kf = kn reduced until dp / c fits; the
// tangential momentum flux, linear in the tangential velocity too, in
// U^2 2^-(kf + kt).  So every flux component has about 55 bits below its own
// largest term (the normal momentum flux: below the pressure), as the binary64
// form has 53, however small the velocities are and whatever state the other
// cells are in.  (One scale for the whole grid, taken from a cell of it, spares the
// conversions a face and the FP64 primitives, 55 us at 512^2, but leaves zones of low
// pressure and small velocities fewer bits than binary64 and sends flows with
// contrasts to the binary64 faces.)
//
// A face's result is used when its reconstructed densities are in (1/16, 1) R,
// pressures in (2^-11, 1/8) R U^2, c~ above U / 16, and no product of the list in
// fixed_roe reaches its bound: jumps by more than a factor of about 6 across its
// four cells, Mach numbers above 4 to 8, velocities below 2^-252 U that are not
// zero, near-vacuum and non-finite states do not pass.  Such faces are collected
// and computed by slow_faces in binary64 with the formulas of roe2_nt from the
// same primitives; the choice is made face by face.

// primitives in shared memory, halo included
template <bool VISC, bool SUTH, class SH>
struct FixedTile {
    double r[SH::EH][SH::EW], u[SH::EH][SH::EW], v[SH::EH][SH::EW], p[SH::EH][SH::EW];
    double T[VISC ? SH::EH : 1][VISC ? SH::EW : 1], mu[SUTH ? SH::EH : 1][SUTH ? SH::EW : 1];
};

// faces left to slow_faces
template <class SH>
struct SlowList {
    static constexpr int NF = (SH::TX + 1) * SH::TY + SH::TX * (SH::TY + 1);
    unsigned short f[NF];
    int n;
};

// dynamic shared memory: the tile, then the faces
template <bool VISC, bool SUTH, class SH>
struct FixedSmem {
    static constexpr size_t bytes = sizeof(FixedTile<VISC, SUTH, SH>) + sizeof(Faces<double, SH>);
};

// CTAs per SM the kernels' registers are held to: 3 (72 to 80 registers, some spilled)
// against 2, because the dependent integer chains need the warps (512^2: 73 against 79 us,
// Euler 58 against 63; 1024^2: 254 against 283 us)
constexpr int kFixedMinB = 3;

// Threads of a tile: the 17 (16 x 16) and 18 (32 x 8) face batches of 32 make
// two rounds on nine warps, three on eight (512^2: 73 against 78 us).
template <class SH>
using FixedShape = Shape<SH::TX, SH::TY, SH::TX == 64 ? 320 : 288>;
using FixedShapeL = Shape<32, 15, 256>;   // large grids: 32 batches, four rounds on eight warps
using FixedShapeS = Shape<16, 7, 256>;    // small grids: 8 batches, one round

// v 2^e (|e| < 900), rounded to nearest (ties away), on the integer pipe: the conversion
// instruction runs at the FP64 rate
__device__ __forceinline__ double scaled(long long v, int e)
{
    const long long m = v >> 63;
    const unsigned long long a = (unsigned long long)((v ^ m) - m);
    const int z = __clzll((long long)a);
    const unsigned long long n = ((a << (z & 63)) >> 10) + 1;   // 54 bits, the lowest for the rounding
    // the top bit adds one to the exponent field; rounding up to 2^54 adds another
    const unsigned long long b = (n >> 1) + ((unsigned long long)(unsigned)(1023 + 62 - z + e) << 52);
    return __hiloint2double(v != 0 ? (int)(b >> 32) | (int)((unsigned)(m >> 32) & 0x80000000u) : 0, v != 0 ? (int)b : 0);
}

// x as a fixed-point number: the bit 2^-62 2^S 2^e of x is the integer's lowest
// for base = 1022 + S + e (low bits are dropped towards zero).  |x| < 2^(S + e).
__device__ __forceinline__ long long fixed_of(double x, int base)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned n = (unsigned)(base - ((hi >> 20) & 0x7ff));
    const unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)lo) << 9;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(n));   // 64 and more (zero, subnormals): zero
    const long long s = (long long)(hi >> 31);
    return ((long long)r ^ s) - s;
}
// the same for x > 0
__device__ __forceinline__ long long fixed_of_positive(double x, int base)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned n = (unsigned)(base - (hi >> 20));
    const unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)lo) << 9;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(n));
    return (long long)r;
}

// grid constants of one instance (StencilConsts holds the shared ones)
struct GridRef {
    int nx, ny;
    double hrdx, hrdy, mu;
};

// Sutherland's law mu(T) = mu_ref g with g in fixed point for t = T / t_ref in
// (1/4, 4) (error below 2^-56; a square root and two divisions in binary64 are some
// sixty FP64 instructions a cell), in binary64 elsewhere
__device__ __noinline__ double sutherland_wide(double t, double s) { return (t * sqrt(t)) * ((1.0 + s) / (t + s)); }
__device__ __forceinline__ double fixed_sutherland(const StencilConsts &C, double mu, double T)
{
    using namespace fx;
    const FixedConsts &F = C.fx;
    const double t = T * C.inv_tref;
    if ((unsigned)__double2hiint(t) - 0x3fd00001u >= 0x00400000u - 1u) return mu * sutherland_wide(t, C.suth_s);
    const Fx<0> t4 = {fixed_of_positive(t, 1024)};               // t / 4 in (1/16, 1)
    Fx<3> z;
    Fx<0> sq;                                                    // sqrt(t) / 2
    rsqrt_sqrt<6>(t4, z, sq);
    const Fx<5> di = rcp_below1<5>(Fx<0>{(t4.v >> 1) + F.suth_s});   // 8 / (t + s), (t + s) / 8 in (1/32, 5/8)
    const Fx<1> n = mul<1>(mul<0>(t4, sq), Fx<1>{F.suth_1s});    // (t^(3/2) / 8) (1 + s), below 2
    const Fx<2> g = mul<2>(n, di);                               // t^(3/2) (1 + s) / (t + s), below 16/5
    return (mu * 0x1p-60) * (double)g.v;
}

// Primitives of one cell, the pressure rounded as the strict build's (the difference E - k
// first): where the kinetic energy is below the last bit of E, the pressure has none.
template <bool VISC, bool SUTH, class SH>
__device__ __forceinline__ void fixed_store_prim(FixedTile<VISC, SUTH, SH> &t, int ly, int lx, double rho, double mx,
                                                 double my, double E, bool mirror, const StencilConsts &C, double mu)
{
    const double rinv = rcp(rho), u = mx * rinv, v = my * rinv;
    const double p = C.gm1 * (E - half(mx * u + my * v));
    t.r[ly][lx] = rho;
    t.u[ly][lx] = mirror ? -u : u;
    t.v[ly][lx] = mirror ? -v : v;
    t.p[ly][lx] = p;
    if (VISC) {
        double T = p * rinv;
        T = fma(fma(-T, rho, p), rinv, T);   // p / rho rounded once: its noise is divided by the cell width twice
        t.T[ly][lx] = T;
        if (SUTH) t.mu[ly][lx] = fixed_sutherland(C, mu, T);
    }
}

// high words of four numbers
struct Four {
    double m2, m1, p1, p2;
    __device__ __forceinline__ Four(const double *a, int i, int s) : m2(a[i - 2 * s]), m1(a[i - s]), p1(a[i]), p2(a[i + s]) {}
    __device__ __forceinline__ int top() const
    {
        return max(max(__double2hiint(m2), __double2hiint(m1)), max(__double2hiint(p1), __double2hiint(p2)));
    }
    __device__ __forceinline__ int bottom() const
    {
        return min(min(__double2hiint(m2), __double2hiint(m1)), min(__double2hiint(p1), __double2hiint(p2)));
    }
    __device__ __forceinline__ int magnitude() const
    {
        return max(max(__double2hiint(m2) & 0x7fffffff, __double2hiint(m1) & 0x7fffffff),
                   max(__double2hiint(p1) & 0x7fffffff, __double2hiint(p2) & 0x7fffffff));
    }
};

// MUSCL states on both sides of a face
__device__ __forceinline__ void fixed_muscl(long long m2, long long m1, long long p1, long long p2,
                                            const FixedConsts &F, long long &L, long long &R)
{
    const long long dc = fx::mul62(F.c_hi, p1 - m1);
    L = m1 + fx::mul62(F.c_lo, m1 - m2) + dc;
    R = p1 - fx::mul62(F.c_lo, p2 - p1) - dc;
}
__device__ __forceinline__ void fixed_muscl(const Four &q, int base, const FixedConsts &F, long long &L, long long &R)
{
    fixed_muscl(fixed_of(q.m2, base), fixed_of(q.m1, base), fixed_of(q.p1, base), fixed_of(q.p2, base), F, L, R);
}
__device__ __forceinline__ void fixed_muscl_positive(const Four &q, int base, const FixedConsts &F, long long &L,
                                                     long long &R)
{
    fixed_muscl(fixed_of_positive(q.m2, base), fixed_of_positive(q.m1, base), fixed_of_positive(q.p1, base),
                fixed_of_positive(q.p2, base), F, L, R);
}
// The pressure, and with ROUND its two roundings of the binary64 form (see fixed_roe)
template <bool ROUND>
__device__ __forceinline__ void fixed_muscl_pressure(const Four &q, int base, const FixedConsts &F, fx::Fx<-3> &L,
                                                     fx::Fx<-3> &R)
{
    using namespace fx;
    if (!ROUND) {
        fixed_muscl_positive(q, base, F, L.v, R.v);
        return;
    }
    const long long m2 = fixed_of_positive(q.m2, base), m1 = fixed_of_positive(q.m1, base);
    const long long p1 = fixed_of_positive(q.p1, base), p2 = fixed_of_positive(q.p2, base);
    const long long dc = mul62(F.c_hi, p1 - m1);
    L = round53(Fx<-3>{round53(Fx<-3>{m1 + mul62(F.c_lo, m1 - m2)}).v + dc});
    R = round53(Fx<-3>{round53(Fx<-3>{p1 - mul62(F.c_lo, p2 - p1)}).v - dc});
}

// velocities down to 2^-252 U have a unit; the exponents of all products stay in range
constexpr int kMaxVelocityShift = 250;

// A face's units: exponents of R and U; bad where the cells leave no such units
// (a density or pressure that is not a positive normal number, extreme exponents)
struct FaceUnits {
    int eR, eU;
    __device__ __forceinline__ FaceUnits(const Four &r, const Four &p, int vmag, bool &bad)
    {
        eR = (r.top() >> 20) - 1021;
        const int x = (p.top() >> 20) - 1023 - eR;   // p / R in [2^x, 2^(x+1))
        eU = max((x + 7) >> 1, (vmag >> 20) - 1021);
        if (min(r.bottom(), p.bottom()) < 0x00100000 || (unsigned)(eR + 100) > 200u || (unsigned)(eU + 100) > 200u)
            bad = true;
    }
    // k of a velocity component of magnitude mag: in [2^-g, 2^(1-g)) of the unit U 2^-k
    template <int g>
    __device__ __forceinline__ int velocity(int mag, bool &bad) const
    {
        const int k = eU - ((mag >> 20) - 1023) - g;
        if (k > kMaxVelocityShift && mag != 0) bad = true;
        return min(max(k, 0), kMaxVelocityShift);
    }
};

// reconstructed states: velocities in the units U 2^-kn, U 2^-kt
struct FixedState {
    fx::Fx<0> r, n, t;
    fx::Fx<-3> p;
};
// doubled Roe flux: g0, g3 in R U 2^-kf, R U^3 2^-kf; gn in R U^2; gt in R U^2 2^-(kf + kt)
struct FixedFlux {
    fx::Fx<0> g0, gn;
    fx::Fx<-2> gt, g3;
    int kf;
};

// Doubled Roe flux, as roe2_nt (the same averages and wave grouping, written with
// the Mach number M = u~ / c~ and the half speeds m1,3 = |M -+ 1| / 2 in units of c~:
// A1 = m1 (dp/c - rho~ dn), A3 = m3 (dp/c + rho~ dn)).  Most products are plain
// mul62 (a product that keeps K more bits costs three to five instructions more);
// a number below its scale by 2^-K is multiplied with those bits where the result is
// a leading term.  The comments give the bounds that keep the values in their formats
// (Fx<S> holds numbers below 2^S; sums may reach 2^(S + 1)).
//
// ROUND (uniform grids): the pressure is rounded to 53 bits where the binary64 form
// rounds it, in the reconstruction and in the momentum sum.  At low Mach numbers
// these roundings are most of the noise of f, a finite-difference quotient divides
// the noise by eps, and the Krylov space built from it then follows the one of a
// plain binary64 evaluation: leading columns of H on a Mach 0.1 Taylor-Green vortex
// (64^2) within 3e-7 of it, against 2.4e-5 without (a residual rounded once from 64
// bits: 3.8e-5).  The price is half a binary64 rounding of the pressure and about 50
// instructions a face.  Curvilinear faces round the reconstruction only.
template <bool ROUND>
__device__ __forceinline__ void fixed_roe(FixedState L, FixedState R, int kn, int kt, const FixedConsts &F, FixedFlux &G,
                                          bool &bad)
{
    using namespace fx;
    if (!in_window<4>(L.r) || !in_window<4>(R.r) || !in_window<8>(L.p) || !in_window<8>(R.p)) bad = true;
    if (outside<1>(L.n) || outside<1>(R.n) || outside<1>(L.t) || outside<1>(R.t)) bad = true;
    // the unit of everything linear in the normal velocity: dp 2^kf below 2^-8
    const Fx<-3> dp = R.p - L.p;
    const int z7 = __clzll(dp.v ^ (dp.v >> 63)) - 7;
    const int kf = dp.v == 0 ? kn : min(kn, max(z7, 0));
    // shifts from those units to U (a shift by 63 leaves the sign)
    const int kd = min(kn - kf, 63), f1 = min(kf, 63), f2 = min(2 * kf, 63), t2 = min(2 * kt, 63);
    L.n.v >>= kd;
    R.n.v >>= kd;
    // rho H = gg p + rho k, k = (n^2 + t^2) / 2
    const Fx<-1> kL = {(mul<0>(L.n, L.n).v >> f2) + (mul<0>(L.t, L.t).v >> t2)};
    const Fx<-1> kR = {(mul<0>(R.n, R.n).v >> f2) + (mul<0>(R.t, R.t).v >> t2)};
    const Fx<0> eL = mul<0>(Fx<3>{F.gg}, L.p) + to<0>(mul<-1>(L.r, kL));
    const Fx<0> eR = mul<0>(Fx<3>{F.gg}, R.p) + to<0>(mul<-1>(R.r, kR));
    if (outside<1>(eL) || outside<1>(eR)) bad = true;
    // Roe averages: z = 1/sqrt(rho_L rho_R), rho~ = sqrt(rho_L rho_R), a = rho_R z in [1/4, 4], tested below 2
    const Fx<0> prr = mul<0>(L.r, R.r);   // in (2^-8, 1)
    Fx<4> z;
    Fx<0> rt;
    rsqrt_sqrt<8>(prr, z, rt);
    const Fx<4> a = mul<4>(R.r, z);
    if (outside<3>(a)) bad = true;
    const Fx<0> wl = rcp_above1(Fx<4>{a.v + (1ll << 58)});
    const Fx<0> drho = R.r - L.r, dn = R.n - L.n, dt = R.t - L.t;   // below 1
    const Fx<0> nt = R.n - mul<0>(wl, dn), tt = R.t - mul<0>(wl, dt);   // below 1/2
    const Fx<1> q = mul<1>(eL, to<1>(a)) + to<1>(eR);                   // below 3/2
    const Fx<5> H5 = mul<5>(mul<4>(wl, z), q);                          // e / rho: below 8
    const Fx<-1> k = {(mul<0>(nt, nt).v >> f2) + (mul<0>(tt, tt).v >> t2)};
    const Fx<5> hk = H5 - to<5>(k);
    if ((unsigned)hi_word(hk.v) >= (1u << 25)) bad = true;   // tested in [0, 1): H below 3/2
    const Fx<0> ct2 = mul<0>(Fx<0>{F.gm1}, to<0>(hk));
    if (!in_window<8>(ct2)) bad = true;
    Fx<4> rc;   // 1 / c~
    Fx<0> ct;
    rsqrt_sqrt<8>(ct2, rc, ct);
    // the acoustic speeds in units of c~: ms = ||M| - 1| (with Harten's fix) and mb = |M| + 1,
    // whose fix is always idle (efix < 1)
    const Fx<4> M = {mul<4>(nt, rc).v >> f1};   // below 8
    constexpr long long one4 = 1ll << 58;
    const Fx<4> aM = abs_of(M), mb = {aM.v + one4};
    Fx<4> ms = abs_of(Fx<4>{aM.v - one4});
    const int mh = hi_word(aM.v);
    if (mh >= F.m_lo && mh <= F.m_hi) {   // the fix may act: (ms^2 / delta + delta) / 2 below delta = efix (|M| + 1)
        const Fx<4> d = mul<4>(Fx<0>{F.efix}, mb);
        // below 1 where ms < d, as |M| < 2 there for efix up to 1/3 (fix_ok); h is unused elsewhere
        const Fx<0> m0 = to<0>(ms);
        const Fx<3> h = {mul<3>(mul<0>(m0, m0), mul<3>(Fx<3>{F.hfix}, rcp_above1(mb))).v + d.v};   // d / 2 as Fx<3>
        if (ms.v < d.v) ms = to<4>(h);
        if (!F.fix_ok) bad = true;
    }
    const Fx<1> dpc1 = mul<1>(Fx<-3>{(long long)((unsigned long long)dp.v << f1)}, rc);
    const Fx<0> rdn = mul<0>(rt, dn);
    if (outside<4>(dpc1) || outside<2>(rdn)) bad = true;   // below 1/8 and 1/4
    const Fx<0> dpc = to<0>(dpc1);
    const bool up = M.v < 0;   // the bits of Fx<4> read as Fx<3> are the half
    const Fx<3> m1 = {up ? mb.v : ms.v}, m3 = {up ? ms.v : mb.v};
    const Fx<0> A1 = mul<0>(m1, dpc - rdn), A3 = mul<0>(m3, dpc + rdn);   // below 9/2 3/8
    const Fx<0> l2 = abs_of(nt);
    const Fx<0> A2 = mul<0>(l2, to<4>(drho) - Fx<4>{mul<4>(dpc, rc).v >> f1});   // below 3/2
    if (outside<2>(A1) || outside<2>(A3) || outside<2>(A2)) bad = true;   // below 1/4
    const Fx<0> sA = A1 + A3, dA = A3 - A1;   // below 1/2
    const Fx<0> D0 = sA + A2;                 // below 3/4
    const Fx<0> Asdt = mul<0>(mul<0>(l2, rt), dt);
    const Fx<0> cdA = mul<0>(ct, dA);
    const Fx<0> Dn = {(mul<0>(nt, D0).v >> f2) + (cdA.v >> f1)};
    const Fx<0> Dt = mul<0>(tt, D0) + Asdt;
    const Fx<0> D3 = mul<0>(H5, sA) + (to<0>(mul<-1>(k, A2)) + Fx<0>{mul<0>(nt, cdA).v >> f1}) +
                     Fx<0>{mul<0>(tt, Asdt).v >> t2};
    const Fx<0> mL = mul<0>(L.r, L.n), mR = mul<0>(R.r, R.n);   // below 1/2
    const Fx<-2> tL = mul<-2>(mL, L.t), tR = mul<-2>(mR, R.t);  // below 1/4
    const Fx<-2> hL = mul<-2>(L.n, eL), hR = mul<-2>(R.n, eR);  // below 1/4
    if (outside<1>(Dn) || outside<3>(Dt) || outside<3>(D3)) bad = true;
    if (outside<1>(tL) || outside<1>(tR) || outside<1>(hL) || outside<1>(hR)) bad = true;   // below 1/8
    G.g0 = (mL + mR) - D0;
    const Fx<0> nL = {mul<0>(mL, L.n).v >> f2}, nR = {mul<0>(mR, R.n).v >> f2};
    if (ROUND) G.gn = nL + round53(nR + round53(to<0>(round53(L.p + R.p)) - Dn));
    else G.gn = nL + (nR + (to<0>(L.p + R.p) - Dn));
    G.gt = tL + (tR - to<-2>(Dt));
    G.g3 = hL + (hR - to<-2>(D3));
    G.kf = kf;
}

// appends the faces f of a warp's lanes with `left' set to the list
template <class SH>
__device__ __forceinline__ void append_slow(SlowList<SH> &sl, int f, bool left)
{
    const unsigned m = __ballot_sync(0xffffffffu, left);
    if (m == 0) return;
    int at = 0;
    if ((threadIdx.x & 31) == 0) at = atomicAdd(&sl.n, __popc(m));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
    if (left) sl.f[at] = (unsigned short)f;
}

// The faces that the fixed-point path left out, in binary64 from the tile's
// primitives: full warps of them, in any order (each is computed by itself).
template <bool VISC, bool SUTH, class SH>
__device__ __noinline__ void slow_faces(const StencilConsts &C, const double (*vk)[5],
                                        const FixedTile<VISC, SUTH, SH> &tl, Faces<double, SH> &fc,
                                        const SlowList<SH> &sl)
{
    constexpr int TX = SH::TX, TY = SH::TY, EW = SH::EW, NFX = (TX + 1) * TY;
    for (int s = threadIdx.x; s < sl.n; s += SH::NT) {
        const int f = sl.f[s];
        const bool yd = f >= NFX;
        const int g = yd ? f - NFX : f;
        const int fx = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int ip = (fy + 2) * EW + fx + 2, sn = yd ? EW : 1, st = yd ? 1 : EW, im = ip - sn;
        const double *pn = yd ? &tl.v[0][0] : &tl.u[0][0], *pt = yd ? &tl.u[0][0] : &tl.v[0][0];
        const double *w[4] = {&tl.r[0][0], pn, pt, &tl.p[0][0]};
        double WL[4], WR[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            muscl(w[k][im - sn], w[k][im], w[k][ip], w[k][ip + sn], C.c_lo, C.c_hi, WL[k], WR[k]);
        double vn = 0.0, vt = 0.0, ve = 0.0;
        if (VISC) {
            const double *pT = &tl.T[0][0], *pm = &tl.mu[0][0];
            auto along = [&](const double *a) { return (a[im + st] + a[ip + st]) - (a[im - st] + a[ip - st]); };
            visc2_terms<SUTH>(pn[ip] - pn[im], pt[ip] - pt[im], pT[ip] - pT[im], along(pn), along(pt), pn[im] + pn[ip],
                              pt[im] + pt[ip], SUTH ? pm[SUTH ? im : 0] + pm[SUTH ? ip : 0] : 0.0, vk[yd ? 1 : 0], vn, vt, ve);
        }
        double g0, gn, gt, g3;
        roe2_nt<VISC>(WL[0], WL[1], WL[2], WL[3], WR[0], WR[1], WR[2], WR[3], C, g0, gn, gt, g3, vn, vt, ve);
        double *out = yd ? &fc.fy[0][fy][fx] : &fc.fx[0][fy][fx];
        const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
        out[0] = g0;
        out[ks] = yd ? gt : gn;
        out[2 * ks] = yd ? gn : gt;
        out[3 * ks] = g3;
    }
}

// One TX x TY tile as cart_tile, the faces in fixed point.
template <bool VISC, bool SUTH, class SH>
__device__ __forceinline__ void fixed_cart_tile(const StencilConsts &C, const GridRef Gr, const double (*vkd)[5],
                                                const StencilIO &io, int i0, int j0, unsigned char *smem_raw,
                                                size_t off = 0, size_t sb = 0)
{
    using namespace fx;
    constexpr int TX = SH::TX, TY = SH::TY, NT = SH::NT, EW = SH::EW, EH = SH::EH;
    constexpr int NFX_ = (TX + 1) * TY, NF = NFX_ + TX * (TY + 1);
    if (io.active && *at_bytes(io.active, sb) == 0) return;
    __shared__ SlowList<SH> sl;
    __shared__ double vks[2][5];
    typedef FixedTile<VISC, SUTH, SH> FT;
    FT &tl = *reinterpret_cast<FT *>(smem_raw);
    Faces<double, SH> &fc = *reinterpret_cast<Faces<double, SH> *>(smem_raw + sizeof(FT));
    const FixedConsts &F = C.fx;
    const int nx = Gr.nx, ny = Gr.ny;
    const size_t nc = (size_t)nx * ny;
    const int tid = threadIdx.x;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2, sb);
    if (tid == 0) sl.n = 0;
    if (VISC && tid < 10) vks[tid / 5][tid % 5] = vkd[tid / 5][tid % 5];
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        const int gi = wrapi(i0 + lx - 2, nx), gj = wrapi(j0 + ly - 2, ny);
        const size_t c = off + (size_t)gj * nx + gi;
        const double q0 = load_value(io, cf, cff, c), q1 = load_value(io, cf, cff, nc + c);
        const double q2 = load_value(io, cf, cff, 2 * nc + c), q3 = load_value(io, cf, cff, 3 * nc + c);
        fixed_store_prim(tl, ly, lx, q0, q1, q2, q3, false, C, Gr.mu);
    }
    __syncthreads();

    // one face per thread in full warp batches, the orientation a per-lane value
    // (as in cart_tile): it selects the cells and the order of u and v
    for (int bt = tid >> 5; bt < (NF + 31) / 32; bt += NT / 32) {
        const int f = bt * 32 + (tid & 31);
        const bool valid = f < NF;
        const bool yd = f >= NFX_;
        const int g = valid ? (yd ? f - NFX_ : f) : 0;
        const int fx_ = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int sn = yd ? EW : 1, st = yd ? 1 : EW;   // steps along the normal and along the face
        const int ip = (fy + 2) * EW + fx_ + 2, im = ip - sn;
        const double *pn = yd ? &tl.v[0][0] : &tl.u[0][0], *pt = yd ? &tl.u[0][0] : &tl.v[0][0];
        const Four r(&tl.r[0][0], ip, sn), p(&tl.p[0][0], ip, sn), n(pn, ip, sn), t(pt, ip, sn);
        bool bad = !valid;
        const int hn = n.magnitude(), ht = t.magnitude();
        const FaceUnits un(r, p, max(hn, ht), bad);
        const int kn = un.velocity<3>(hn, bad), kt = un.velocity<3>(ht, bad);
        if (__any_sync(0xffffffffu, !bad)) {
            FixedState L, R;
            fixed_muscl_positive(r, 1022 + un.eR, F, L.r.v, R.r.v);
            fixed_muscl_pressure<true>(p, 1022 - 3 + un.eR + 2 * un.eU, F, L.p, R.p);
            fixed_muscl(n, 1022 + un.eU - kn, F, L.n.v, R.n.v);
            fixed_muscl(t, 1022 + un.eU - kt, F, L.t.v, R.t.v);
            FixedFlux G;
            fixed_roe<true>(L, R, kn, kt, F, G, bad);
            if (!bad) {
                // the units' exponents; viscous terms join in binary64
                const int e0 = un.eR + un.eU - 62 - G.kf, e1 = un.eR + 2 * un.eU - 62;
                const int et = e1 - 2 - G.kf - kt, e3 = e0 + 2 * un.eU - 2;
                double gn, gt, g3;
                if (VISC) {
                    const double *pT = &tl.T[0][0], *pm = &tl.mu[0][0];
                    auto along = [&](const double *a) { return (a[im + st] + a[ip + st]) - (a[im - st] + a[ip - st]); };
                    double vn, vt, ve;
                    visc2_terms<SUTH>(n.p1 - n.m1, t.p1 - t.m1, pT[ip] - pT[im], along(pn), along(pt), n.m1 + n.p1,
                                      t.m1 + t.p1, SUTH ? pm[SUTH ? im : 0] + pm[SUTH ? ip : 0] : 0.0, vks[yd ? 1 : 0], vn, vt,
                                      ve);
                    gn = scaled(G.gn.v, e1) - vn;
                    gt = scaled(G.gt.v, et) - vt;
                    g3 = scaled(G.g3.v, e3) - ve;
                } else {
                    gn = scaled(G.gn.v, e1);
                    gt = scaled(G.gt.v, et);
                    g3 = scaled(G.g3.v, e3);
                }
                double *out = yd ? &fc.fy[0][fy][fx_] : &fc.fx[0][fy][fx_];
                const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
                out[0] = scaled(G.g0.v, e0);
                out[ks] = yd ? gt : gn;
                out[2 * ks] = yd ? gn : gt;
                out[3 * ks] = g3;
            }
        }
        append_slow(sl, f, bad && valid);
    }
    __syncthreads();
    if (sl.n) {
        slow_faces<VISC, SUTH, SH>(C, vks, tl, fc, sl);
        __syncthreads();
    }

#pragma unroll
    for (int cell = tid; cell < TX * TY; cell += NT) {
        const int tx = cell % TX, ty = cell / TX;
        const int gi = i0 + tx, gj = j0 + ty;
        if (gi < nx && gj < ny) {
            const size_t c = off + (size_t)gj * nx + gi;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double dX = fc.fx[k][ty][tx + 1] - fc.fx[k][ty][tx];
                const double dY = fc.fy[k][ty + 1][tx] - fc.fy[k][ty][tx];
                const size_t e = k * nc + c;
                // r - sub = -(dX bx + (dY by + sub)): two FMAs
                const double t = io.sub ? -(dX * Gr.hrdx + (dY * Gr.hrdy + io.sub[e])) : -(dX * Gr.hrdx + dY * Gr.hrdy);
                epilogue_finish(io, s2, e, t * s1, sb);
            }
        }
    }
}

template <bool VISC, bool SUTH, class SH, int MINB>
__global__ void __launch_bounds__(SH::NT, MINB)
    fixed_cart_kernel(const __grid_constant__ StencilConsts C, const __grid_constant__ StencilIO io)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fixed_cart_tile<VISC, SUTH, SH>(C, GridRef{C.nx, C.ny, C.hrdx, C.hrdy, C.mu}, C.vk, io, blockIdx.x * SH::TX,
                                    blockIdx.y * SH::TY, smem_raw);
}

// many grids in one launch, as cart_batch_kernel
template <bool VISC, bool SUTH, class SH, int MINB>
__global__ void __launch_bounds__(SH::NT, MINB)
    fixed_batch_kernel(const __grid_constant__ StencilConsts C, const __grid_constant__ StencilIO io, const BatchTiles bt)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = blockIdx.x;
    const int k = bt.tile_inst[b];
    const BatchInst &I = bt.inst[k];
    const int t = b - bt.tile_first[k];
    const int ntx = (I.nx + SH::TX - 1) / SH::TX;
    fixed_cart_tile<VISC, SUTH, SH>(C, GridRef{I.nx, I.ny, I.hrdx, I.hrdy, I.mu}, I.vk, io, (t % ntx) * SH::TX,
                                    (t / ntx) * SH::TY, smem_raw, I.off, (size_t)k * bt.stride_bytes);
}

// ============================== curvilinear grid ===============================
// The same for curv_kernel's grids.  A face's reconstructed velocities are
// rotated into its (normal, tangential) frame, fixed_roe runs there (the flux is
// invariant under rotation) and the momentum fluxes are rotated back in binary64.
// u and v share one unit, except on faces along a grid line (a normal with one
// component zero), which mix nothing.

// a component of a unit normal (|x| <= 1) as Fx<0>, 1 just below
__device__ __forceinline__ fx::Fx<0> fixed_normal(double x)
{
    const int ex = __double2hiint(x) >> 20 & 0x7ff;
    const long long one = (1ll << 62) - 1;
    return {ex >= 1023 ? (__double2hiint(x) < 0 ? -one : one) : fixed_of(x, 1022)};
}

// Viscous coefficients of a curvilinear face.  The doubled stress and heat flux of
// visc_n2_terms are linear in the differences across (dC) and along (dV, four
// cells) the face; with the metric terms, the normal and the viscosity multiplied
// out they are 10 products of a face instead of 28 operations:
//   t1 = a0 dCu + a1 dVu + a2 dCv + a3 dVv, t2 = a4 dCu + .. + a7 dVv, q = a8 dCT + a9 dVT.
__global__ void __launch_bounds__(256)
    visc_coefs_kernel(const __grid_constant__ StencilConsts C, const double *__restrict__ nx,
                      const double *__restrict__ ny, const double *__restrict__ c0, const double *__restrict__ c1,
                      const double *__restrict__ c2, const double *__restrict__ c3, size_t n, double *__restrict__ out)
{
    const size_t f = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (f >= n) return;
    const double x = nx[f], y = ny[f];
    const double k0 = C.vc[0], k1 = C.vc[1], k2 = C.vc[2], k3 = C.vc[3];
    const double cx[2] = {c0[f], 0.25 * c1[f]}, cy[2] = {c2[f], 0.25 * c3[f]};   // across, along
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        out[d * n + f] = k0 * x * cx[d] + k2 * y * cy[d];         // t1: u
        out[(2 + d) * n + f] = k1 * x * cy[d] + k2 * y * cx[d];   // t1: v
        out[(4 + d) * n + f] = k2 * x * cy[d] + k1 * y * cx[d];   // t2: u
        out[(6 + d) * n + f] = k2 * x * cx[d] + k0 * y * cy[d];   // t2: v
        out[(8 + d) * n + f] = k3 * (x * cx[d] + y * cy[d]);
    }
}

// Viscous terms of one face (v1, v2 the momentum, v3 the energy) from the tile's
// primitives; nf the faces of its direction, st the step along the face (+1 row
// on i-faces, -1 column on j-faces)
template <bool VISC, bool SUTH, class SH>
__device__ __forceinline__ void curv_visc(const double *__restrict__ a, size_t nf, const FixedTile<VISC, SUTH, SH> &tl,
                                          int im, int ip, int st, double &v1, double &v2, double &v3)
{
    const double *pu = &tl.u[0][0], *pv = &tl.v[0][0], *pT = &tl.T[0][0], *pm = &tl.mu[0][0];
    auto across = [&](const double *w) { return w[ip] - w[im]; };
    auto along = [&](const double *w) { return (w[im + st] + w[ip + st]) - (w[im - st] + w[ip - st]); };
    const double Cu = across(pu), Vu = along(pu), Cv = across(pv), Vv = along(pv);
    double t1 = (a[0] * Cu + a[nf] * Vu) + (a[2 * nf] * Cv + a[3 * nf] * Vv);
    double t2 = (a[4 * nf] * Cu + a[5 * nf] * Vu) + (a[6 * nf] * Cv + a[7 * nf] * Vv);
    double q = a[8 * nf] * across(pT) + a[9 * nf] * along(pT);
    if (SUTH) {
        const double mus = pm[SUTH ? im : 0] + pm[SUTH ? ip : 0];
        t1 = t1 * mus;
        t2 = t2 * mus;
        q = q * mus;
    }
    v1 = t1;
    v2 = t2;
    v3 = half(pu[im] + pu[ip]) * t1 + (half(pv[im] + pv[ip]) * t2 + q);
}

// the faces left out by the fixed-point path, in binary64 (as slow_faces)
template <bool VISC, bool SUTH, class SH>
__device__ __noinline__ void slow_curv_faces(const StencilConsts &C, const CurvGeom &G,
                                             const FixedTile<VISC, SUTH, SH> &tl, int i0, int j0,
                                             Faces<double, SH> &fc, const SlowList<SH> &sl)
{
    constexpr int TX = SH::TX, TY = SH::TY, EW = SH::EW, NFX = (TX + 1) * TY;
    const int nx = C.nx;
    const size_t nfi = (size_t)(nx + 1) * C.ny, nfj = (size_t)nx * (C.ny + 1);
    for (int s = threadIdx.x; s < sl.n; s += SH::NT) {
        const int f = sl.f[s];
        const bool yd = f >= NFX;
        const int g = yd ? f - NFX : f;
        const int fx = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int gi = i0 + fx, gj = j0 + fy;
        const size_t fi = yd ? (size_t)gj * nx + gi : (size_t)gj * (nx + 1) + gi;
        const int ip = (fy + 2) * EW + fx + 2, sn = yd ? EW : 1, im = ip - sn;
        const double *w[4] = {&tl.r[0][0], &tl.u[0][0], &tl.v[0][0], &tl.p[0][0]};
        double WL[4], WR[4], Fl[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            muscl(w[k][im - sn], w[k][im], w[k][ip], w[k][ip + sn], C.c_lo, C.c_hi, WL[k], WR[k]);
        const double nxf = yd ? G.jn_x[fi] : G.in_x[fi], nyf = yd ? G.jn_y[fi] : G.in_y[fi];
        double v1 = 0.0, v2 = 0.0, v3 = 0.0;
        if (VISC) curv_visc((yd ? G.jv : G.iv) + fi, yd ? nfj : nfi, tl, im, ip, yd ? -1 : EW, v1, v2, v3);
        roe_n2<VISC>(WL, WR, nxf, nyf, C, Fl, v1, v2, v3);
        const double len = half(yd ? G.jl[fi] : G.il[fi]);
        double *out = yd ? &fc.fy[0][fy][fx] : &fc.fx[0][fy][fx];
        const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k * ks] = Fl[k] * len;
    }
}

template <bool VISC, bool SUTH, class SH, int MINB>
__global__ void __launch_bounds__(SH::NT, MINB)
    fixed_curv_kernel(const __grid_constant__ StencilConsts C, const __grid_constant__ CurvGeom G,
                      const __grid_constant__ StencilIO io)
{
    using namespace fx;
    constexpr int TX = SH::TX, TY = SH::TY, NT = SH::NT, EW = SH::EW, EH = SH::EH;
    constexpr int NFX_ = (TX + 1) * TY, NF = NFX_ + TX * (TY + 1);
    if (io.active && *io.active == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ SlowList<SH> sl;
    typedef FixedTile<VISC, SUTH, SH> FT;
    FT &tl = *reinterpret_cast<FT *>(smem_raw);
    Faces<double, SH> &fc = *reinterpret_cast<Faces<double, SH> *>(smem_raw + sizeof(FT));
    const FixedConsts &F = C.fx;
    const int nx = C.nx, ny = C.ny;
    const size_t nc = (size_t)nx * ny, nfi = (size_t)(nx + 1) * ny, nfj = (size_t)nx * (ny + 1);
    const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
    const int tid = threadIdx.x;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2);
    if (tid == 0) sl.n = 0;
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        int gi = i0 + lx - 2, gj = j0 + ly - 2;
        bool mirror, inf;
        curv_source(C, gi, gj, mirror, inf);
        if (inf) {
            tl.r[ly][lx] = C.prim_inf[0];
            tl.u[ly][lx] = mirror ? -C.prim_inf[1] : C.prim_inf[1];
            tl.v[ly][lx] = mirror ? -C.prim_inf[2] : C.prim_inf[2];
            tl.p[ly][lx] = C.prim_inf[3];
            if (VISC) tl.T[ly][lx] = C.prim_inf[4];
            if (SUTH) tl.mu[ly][lx] = C.prim_inf[5];
        } else {
            const size_t c = (size_t)gj * nx + gi;
            const double q0 = load_value(io, cf, cff, c), q1 = load_value(io, cf, cff, nc + c);
            const double q2 = load_value(io, cf, cff, 2 * nc + c), q3 = load_value(io, cf, cff, 3 * nc + c);
            fixed_store_prim(tl, ly, lx, q0, q1, q2, q3, mirror, C, C.mu);
        }
    }
    __syncthreads();

    for (int bt = tid >> 5; bt < (NF + 31) / 32; bt += NT / 32) {
        const int f = bt * 32 + (tid & 31);
        const bool yd = f >= NFX_;
        const int g = f < NF ? (yd ? f - NFX_ : f) : 0;
        const int fx_ = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int gi = i0 + fx_, gj = j0 + fy;
        const bool valid = f < NF && (yd ? (gi < nx && gj <= ny) : (gi <= nx && gj < ny));
        bool bad = !valid;
        const size_t fi = valid ? (yd ? (size_t)gj * nx + gi : (size_t)gj * (nx + 1) + gi) : 0;
        const double nxd = yd ? G.jn_x[fi] : G.in_x[fi], nyd = yd ? G.jn_y[fi] : G.in_y[fi];
        const double len = half(yd ? G.jl[fi] : G.il[fi]);
        const int ip = (fy + 2) * EW + fx_ + 2;
        const int sn = yd ? EW : 1, im = ip - sn;
        const Four r(&tl.r[0][0], ip, sn), p(&tl.p[0][0], ip, sn), u(&tl.u[0][0], ip, sn), v(&tl.v[0][0], ip, sn);
        const int hu = u.magnitude(), hv = v.magnitude(), h = max(hu, hv);
        const FaceUnits un(r, p, h, bad);
        const bool ax = nyd == 0.0, ay = nxd == 0.0;   // along x, along y
        const bool own = ax || ay;
        const int ku = un.velocity<4>(own ? hu : h, bad), kv = un.velocity<4>(own ? hv : h, bad);
        const int kn = ay ? kv : ku, kt = ay ? ku : kv;
        if (!__any_sync(0xffffffffu, !bad)) {
            append_slow(sl, f, valid);
            continue;
        }
        FixedState L, R;
        Fx<0> uL, uR, vL, vR;
        fixed_muscl_positive(r, 1022 + un.eR, F, L.r.v, R.r.v);
        fixed_muscl_pressure<true>(p, 1022 - 3 + un.eR + 2 * un.eU, F, L.p, R.p);
        fixed_muscl(u, 1022 + un.eU - ku, F, uL.v, uR.v);
        fixed_muscl(v, 1022 + un.eU - kv, F, vL.v, vR.v);
        const Fx<0> mnx = fixed_normal(nxd), mny = fixed_normal(nyd);
        L.n = mul<0>(uL, mnx) + mul<0>(vL, mny);
        R.n = mul<0>(uR, mnx) + mul<0>(vR, mny);
        L.t = mul<0>(vL, mnx) - mul<0>(uL, mny);
        R.t = mul<0>(vR, mnx) - mul<0>(uR, mny);
        FixedFlux H;
        fixed_roe<false>(L, R, kn, kt, F, H, bad);
        if (!bad) {
            const int e0 = un.eR + un.eU - 62 - H.kf, e1 = un.eR + 2 * un.eU - 62;
            const int et = e1 - 2 - H.kf - kt, e3 = e0 + 2 * un.eU - 2;
            const double gn = scaled(H.gn.v, e1), gt = scaled(H.gt.v, et);
            double m1, m2, g3 = scaled(H.g3.v, e3);
            if (VISC) {
                double v1, v2, v3;
                curv_visc((yd ? G.jv : G.iv) + fi, yd ? nfj : nfi, tl, im, ip, yd ? -1 : EW, v1, v2, v3);
                m1 = gn * nxd - (gt * nyd + v1);
                m2 = gn * nyd + (gt * nxd - v2);
                g3 = g3 - v3;
            } else {
                m1 = gn * nxd - gt * nyd;
                m2 = gn * nyd + gt * nxd;
            }
            double *out = yd ? &fc.fy[0][fy][fx_] : &fc.fx[0][fy][fx_];
            const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
            out[0] = scaled(H.g0.v, e0) * len;
            out[ks] = m1 * len;
            out[2 * ks] = m2 * len;
            out[3 * ks] = g3 * len;
        }
        append_slow(sl, f, bad && valid);
    }
    __syncthreads();
    if (sl.n) {
        slow_curv_faces<VISC, SUTH, SH>(C, G, tl, i0, j0, fc, sl);
        __syncthreads();
    }

    for (int cell = tid; cell < TX * TY; cell += NT) {
        const int tx = cell % TX, ty = cell / TX;
        const int gi = i0 + tx, gj = j0 + ty;
        if (gi < nx && gj < ny) {
            const size_t c = (size_t)gj * nx + gi;
            const double iv = G.inv_vol[c];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double dX = fc.fx[k][ty][tx + 1] - fc.fx[k][ty][tx];
                const double dY = fc.fy[k][ty + 1][tx] - fc.fy[k][ty][tx];
                epilogue_store(io, s1, s2, k * nc + c, -((dX + dY) * iv));
            }
        }
    }
}
