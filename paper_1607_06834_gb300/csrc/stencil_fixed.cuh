// Uniform-grid residual / FD-JVP stencil of the FMA build on 64-bit fixed point
// (fixed.cuh), included by stencil_impl.cuh inside its namespace.
//
// The binary64 form of this kernel is bound by FP64 issue: 271 FP64
// instructions a cell, 86 % of the pipe.  Here the primitives and the face
// fluxes (MUSCL, Roe, viscous terms) run on the integer pipe, and FP64 keeps
// what needs a floating range: the state y + sum c_t add_t, the cell balance
// and the epilogue (about 30 instructions a cell), which overlaps.  Measured
// (us): residual 147.6 -> 55.3 at 512^2 (Navier-Stokes), 26.6 -> 8.2 at 64^2
// (Euler); FD-JVP 607 -> 210 at 1024^2.  What bounds it now: the integer ALU is
// busy half of the time and FP64 a third, the rest is latency of the dependent
// chains at 24 to 27 warps an SM.
//
// Units.  Every instance is scaled by powers of two, R for densities and U for
// velocities (momenta R U, energies R U^2, pressures R U^2), taken from its
// cell 0, so that a face's result does not depend on the tile it is computed
// in.  With rho of cell 0 in [1/4, 1/2) R and E / rho in (1/32, 1/4) U^2, the
// sound speed there is 0.13 to 0.38 U.  A cell is `good' when rho in [1/16, 1) R,
// |u|, |v| < U / 2 (Mach 1.3 to 3.8), p in [2^-11, 1/8) R U^2 and T < U^2 / 2;
// a face when its reconstructed states are in the same ranges, the jumps of
// pressure and velocity across it are below the sound-speed scale (dp / c and
// rho~ du below R U / 8) and the Roe-averaged state is in range.  Inside these ranges no intermediate wraps, and the
// results carry an error of a few 2^-60 R U^k, below the binary64 rounding of
// the primitives.  All other faces (near-vacuum, strong shocks, non-finite states, a cell 0 far from the rest) are
// computed by slow_faces in binary64 with the formulas of roe2_nt; the choice
// is made face by face from the face's own cells.

// shared-memory tile of fixed-point primitives, halo included; the lowest bit
// of u is set for a cell that is not good.  With Sutherland's law g is
// mu / mu_ref.
template <bool SUTH, class SH>
struct FixedTile {
    long long r[SH::EH][SH::EW], u[SH::EH][SH::EW], v[SH::EH][SH::EW], p[SH::EH][SH::EW], T[SH::EH][SH::EW];
    long long g[SUTH ? SH::EH : 1][SUTH ? SH::EW : 1];
};

// per-CTA constants: the scales' exponents, the balance factors and the viscous
// coefficients as mantissas (common exponent)
struct FixedShared {
    long long vk[2][5];
    double bx[4], by[4];   // 0.5/dx, 0.5/dy times the unit of each flux component (raw integers in fc)
    double up[4];          // the inverse unit (slow faces)
    int eR, eU;
    int vshift;            // viscous terms: right shift (negative: all faces slow)
    int any_slow;
};

// dynamic shared memory: the tile (the slow faces reuse it in binary64), then the faces
template <bool SUTH, class SH>
struct FixedSmem {
    static constexpr size_t fixed = sizeof(FixedTile<SUTH, SH>), dbl = (SUTH ? 6 : 5) * sizeof(double) * SH::EH * SH::EW;
    static constexpr size_t faces = fixed > dbl ? fixed : dbl;
    static constexpr size_t bytes = faces + sizeof(Faces<double, SH>);
};

// CTAs per SM the kernels' registers are held to: 3 (72 to 80 registers, a few
// words of local memory) against 2 (126) is 16 % faster at 512^2 and 27 % at
// 1024^2; the dependent integer chains need the warps.
constexpr int kFixedMinB = 3;

// Threads of a tile: the 17 (16 x 16) and 18 (32 x 8) face batches of 32 make
// two rounds on nine warps, three on eight (1024^2: 224 against 235 us).
template <class SH>
using FixedShape = Shape<SH::TX, SH::TY, SH::TX == 64 ? 320 : 288>;
using FixedShapeL = Shape<32, 15, 256>;   // large grids: 32 batches, four rounds on eight warps
using FixedShapeS = Shape<16, 7, 256>;    // small grids: 8 batches, one round

// 2^e as binary64 (|e| < 1000)
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Scale exponents of an instance from its cell 0 (rho, E): rho 2^-eR in
// [1/4, 1/2), (E / rho) 2^-2eU in (1/32, 1/4).  A non-positive or
// extreme cell 0 gives 0 (the windows then decide cell by cell).
__device__ __forceinline__ void fixed_scales(double rho, double E, int &eR, int &eU)
{
    const int hr = __double2hiint(rho), he = __double2hiint(E);
    const int xr = (hr >> 20) - 1023, xe = (he >> 20) - 1023;
    eR = xr + 2;
    const int x = xe - xr;   // E / rho in (2^(x-1), 2^(x+1))
    eU = (x + 4) >> 1;       // 2 eU in {x + 3, x + 4}
    if (hr <= 0 || he <= 0 || abs(eR) > 100 || abs(eU) > 100) eR = eU = 0;
}

// grid constants of one instance (StencilConsts holds the shared ones)
struct GridRef {
    int nx, ny;
    double hrdx, hrdy, mu;
};

// primitives of one cell in fixed point, the lowest bit of u set outside the windows
template <bool VISC, bool SUTH>
__device__ __forceinline__ void fixed_prim(double q0, double q1, double q2, double q3, int eR, int eU,
                                           const FixedConsts &F, long long (&w)[6])
{
    using namespace fx;
    bool bad = false;
    const Fx<0> r = from_double<0>(q0, eR, bad);
    const Fx<0> mx = from_double<0>(q1, eR + eU, bad), my = from_double<0>(q2, eR + eU, bad);
    const Fx<0> E = from_double<0>(q3, eR + 2 * eU, bad);
    if (!in_window<4>(r)) bad = true;
    const Fx<4> ri = rcp_below1<4>(r);
    const Fx<0> u = mul_below<0, 1>(mx, ri, bad), v = mul_below<0, 1>(my, ri, bad);
    const Fx<0> ke = half_of(mul<0>(mx, u) + mul<0>(my, v));
    const Fx<-3> p = round53(mul_below<-3, 0>(Fx<0>{F.gm1}, round53(E - ke), bad));
    if (!in_window<8>(p)) bad = true;
    w[0] = r.v;
    w[2] = v.v;
    w[3] = p.v;
    if (VISC) {
        const Fx<0> T = mul_below<0, 1>(p, ri, bad);
        w[4] = T.v;
        if (SUTH) {
            // g(T) = t^(3/2) (1 + s) / (t + s), t = T / t_ref in [1/4, 4):
            // t / 4 as Fx<0>, t / 4 by the power of two left of U^2 / t_ref
            const int sl = F.itref_e + 2 * eU - 2;
            const Fx<0> tm = mul<0>(T, Fx<0>{F.itref});
            const int s0 = sl < 0 ? 0 : (sl > 31 ? 31 : sl);
            if (sl < 0 || sl > 31 || tm.v < 0 || (tm.v >> (62 - s0)) != 0) bad = true;
            const Fx<0> t4 = {tm.v << s0};
            if (!in_window<4>(t4)) bad = true;
            Fx<3> z;
            Fx<0> sq;                                                // sqrt(t) / 2
            rsqrt_sqrt<6>(t4, z, sq);
            const Fx<0> d = {t4.v + F.suth_s};                       // (t + s) / 4
            if (!in_window<3>(d)) bad = true;
            const Fx<3> di = rcp_below1<3>(d);
            // g = t sqrt(t) (1 + s) / (t + s) = 2 (t/4) (2 sqrt(t)/2 (1 + s)) / d / ... : 2 t4 sq (1 + s) / d
            const Fx<1> n = mul<1>(mul<0>(t4, sq), Fx<1>{F.suth_1s});   // (t^(3/2) / 8) (1 + s)
            const Fx<2> g = mul_below<2, 1>(n, Fx<4>{di.v}, bad);      // times 2 / d: t^(3/2) (1 + s) / (t + s)
            w[5] = g.v;
        }
    }
    w[1] = (u.v & ~1ll) | (bad ? 1 : 0);
}

// MUSCL states on both sides of a face from the four cells along its normal
__device__ __forceinline__ void fixed_muscl(long long m2, long long m1, long long p1, long long p2,
                                            const FixedConsts &F, long long &L, long long &R)
{
    const long long dc = fx::mul62(F.c_hi, p1 - m1);
    L = m1 + fx::mul62(F.c_lo, m1 - m2) + dc;
    R = p1 - fx::mul62(F.c_lo, p2 - p1) - dc;
}

// the same for the pressure, with the two roundings of the binary64 form
__device__ __forceinline__ void fixed_muscl_p(long long m2, long long m1, long long p1, long long p2,
                                              const FixedConsts &F, fx::Fx<-3> &L, fx::Fx<-3> &R)
{
    using namespace fx;
    const long long dc = mul62(F.c_hi, p1 - m1);
    L = round53(Fx<-3>{round53(Fx<-3>{m1 + mul62(F.c_lo, m1 - m2)}).v + dc});
    R = round53(Fx<-3>{round53(Fx<-3>{p1 - mul62(F.c_lo, p2 - p1)}).v - dc});
}

struct FixedState {
    fx::Fx<0> r, n, t;
    fx::Fx<-3> p;
};

// Doubled Roe flux minus the doubled viscous terms, as roe2_nt (the same
// averages and wave grouping, written with the Mach number M = u~ / c~ and the
// half speeds m1,3 = |M -+ 1| / 2 in units of c~: A1 = m1 (dp/c - rho~ dn),
// A3 = m3 (dp/c + rho~ dn)).  The scales are chosen so that every product is
// a plain mul62 and results are realigned by shifts (a product that keeps more
// bits costs five instructions more); the comments give the bounds that keep
// the values in their formats.
// ROUND: the uniform grids' roundings of the pressure sums.
template <bool ROUND>
__device__ __forceinline__ void fixed_roe(const FixedState &L, const FixedState &R, const FixedConsts &F, fx::Fx<0> vn,
                                          fx::Fx<0> vt, fx::Fx<0> ve, fx::Fx<0> (&G)[4], bool &bad)
{
    using namespace fx;
    if (!in_window<4>(L.r) || !in_window<4>(R.r) || !in_window<8>(L.p) || !in_window<8>(R.p)) bad = true;
    if (outside<1>(L.n) || outside<1>(R.n) || outside<1>(L.t) || outside<1>(R.t)) bad = true;
    // rho H = gg p + rho k, k = (n^2 + t^2) / 2
    const Fx<-1> kL = {mul<0>(L.n, L.n).v + mul<0>(L.t, L.t).v}, kR = {mul<0>(R.n, R.n).v + mul<0>(R.t, R.t).v};
    const Fx<0> eL = mul<0>(Fx<3>{F.gg}, L.p) + to<0>(mul<-1>(L.r, kL));
    const Fx<0> eR = mul<0>(Fx<3>{F.gg}, R.p) + to<0>(mul<-1>(R.r, kR));
    if (outside<1>(eL) || outside<1>(eR)) bad = true;
    // Roe averages: z = 1/sqrt(rho_L rho_R), rho~ = sqrt(rho_L rho_R), a = rho_R z in [1/4, 4], tested below 2
    const Fx<0> prr = mul<0>(L.r, R.r);   // in [2^-8, 1)
    Fx<4> z;
    Fx<0> rt;
    rsqrt_sqrt<8>(prr, z, rt);
    const Fx<4> a = mul<4>(R.r, z);
    if (outside<3>(a)) bad = true;
    const Fx<0> wl = rcp_above1(Fx<4>{a.v + (1ll << 58)});
    const Fx<0> drho = R.r - L.r, dn = R.n - L.n, dt = R.t - L.t;   // below 1
    const Fx<-3> dp = R.p - L.p;
    const Fx<0> nt = R.n - mul<0>(wl, dn), tt = R.t - mul<0>(wl, dt);   // below 1/2
    const Fx<1> q = mul<1>(eL, to<1>(a)) + to<1>(eR);                   // below 3/2
    const Fx<5> H5 = mul<5>(mul<4>(wl, z), q);                          // e / rho: below 8
    const Fx<-1> kt = {mul<0>(nt, nt).v + mul<0>(tt, tt).v};
    const Fx<5> hk = H5 - to<5>(kt);
    if ((unsigned)hi_word(hk.v) >= (1u << 25)) bad = true;   // tested in [0, 1)
    const Fx<0> ct2 = mul<0>(Fx<0>{F.gm1}, to<0>(hk));
    if (!in_window<8>(ct2)) bad = true;
    Fx<4> rc;   // 1 / c~
    Fx<0> ct;
    rsqrt_sqrt<8>(ct2, rc, ct);
    // the acoustic speeds in units of c~: ms = ||M| - 1| (with Harten's fix) and mb = |M| + 1,
    // whose fix is always idle (efix < 1)
    const Fx<4> M = mul<4>(nt, rc);   // below 8
    constexpr long long one4 = 1ll << 58;
    const Fx<4> aM = abs_of(M), mb = {aM.v + one4};
    Fx<4> ms = abs_of(Fx<4>{aM.v - one4});
    const int mh = hi_word(aM.v);
    if (mh >= F.m_lo && mh <= F.m_hi) {   // the fix may act: (ms^2 / delta + delta) / 2 below delta = efix (|M| + 1)
        const Fx<4> d = mul<4>(Fx<0>{F.efix}, mb);
        const Fx<0> m0 = to<0>(ms);       // below 1/2 here
        const Fx<3> h = {mul<3>(mul<0>(m0, m0), mul<3>(Fx<3>{F.hfix}, rcp_above1(mb))).v + d.v};   // d / 2 as Fx<3>
        if (ms.v < d.v) ms = to<4>(h);
        if (!F.fix_ok) bad = true;
    }
    const Fx<1> dpc1 = mul<1>(dp, rc);
    const Fx<0> rdn = mul<0>(rt, dn);
    if (outside<4>(dpc1) || outside<3>(rdn)) bad = true;   // both below 1/8
    const Fx<0> dpc = to<0>(dpc1);
    const bool up = M.v < 0;   // the bits of Fx<4> read as Fx<3> are the half
    const Fx<3> m1 = {up ? mb.v : ms.v}, m3 = {up ? ms.v : mb.v};
    const Fx<3> A1 = mul<3>(m1, dpc - rdn), A3 = mul<3>(m3, dpc + rdn);   // below 9/8
    const Fx<3> sA3 = A1 + A3, dA3 = A3 - A1;
    const Fx<0> l2 = abs_of(nt);
    const Fx<4> A24 = mul<4>(l2, to<4>(drho) - mul<4>(dpc, rc));          // below 3/2
    if (outside<5>(sA3) || outside<5>(dA3) || outside<6>(A24)) bad = true;   // below 1/4
    const Fx<0> sA = to<0>(sA3), dA = to<0>(dA3), A2 = to<0>(A24);
    const Fx<0> D0 = sA + A2;
    const Fx<0> Asdt = mul<0>(mul<0>(l2, rt), dt);
    const Fx<0> cdA = mul<0>(ct, dA);
    const Fx<0> Dn = mul<0>(nt, D0) + (cdA + vn);
    const Fx<0> Dt = mul<0>(tt, D0) + (Asdt + vt);
    const Fx<0> D3 = to<0>(mul<1>(to<1>(H5), sA)) + (to<0>(mul<-1>(kt, A2)) + mul<0>(nt, cdA) + (mul<0>(tt, Asdt) + ve));
    if (outside<1>(Dn) || outside<1>(Dt) || outside<1>(D3)) bad = true;
    const Fx<0> mL = mul<0>(L.r, L.n), mR = mul<0>(R.r, R.n);   // below 1/2
    G[0] = (mL + mR) - D0;
    if (ROUND) G[1] = mul<0>(mL, L.n) + round53(mul<0>(mR, R.n) + round53(to<0>(round53(L.p + R.p)) - Dn));
    else G[1] = mul<0>(mL, L.n) + (mul<0>(mR, R.n) + (to<0>(L.p + R.p) - Dn));
    G[2] = mul<0>(mL, L.t) + (mul<0>(mR, R.t) - Dt);
    G[3] = mul<0>(L.n, eL) + (mul<0>(R.n, eR) - D3);
}

// The faces that the fixed-point path left out (bit f % 32 of slow[f / 32]), in
// binary64: the CTA's primitives once more, now in binary64 over the tile's
// shared memory, then one face per thread.  Rarely called; a CTA whose faces
// all come here costs its binary64 time plus the integer pass.
template <bool VISC, bool SUTH, class SH>
__device__ __noinline__ void slow_faces(const StencilConsts &C, const GridRef Gr, const StencilIO &io, int i0,
                                        int j0, size_t off, size_t sb, unsigned char *smem_raw, Faces<double, SH> &fc,
                                        const FixedShared &fs, const unsigned *slow, const double (*vk)[5])
{
    constexpr int TX = SH::TX, TY = SH::TY, NT = SH::NT, EW = SH::EW, EH = SH::EH;
    typedef double Arr[EH][EW];
    Arr *w = reinterpret_cast<Arr *>(smem_raw);   // rho, u, v, p, T, mu
    const int nx = Gr.nx, ny = Gr.ny, tid = threadIdx.x;
    const size_t nc = (size_t)nx * ny;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2, sb);
    __syncthreads();
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        const size_t c = off + (size_t)wrapi(j0 + ly - 2, ny) * nx + wrapi(i0 + lx - 2, nx);
        const double rho = load_value(io, cf, cff, c), mx = load_value(io, cf, cff, nc + c);
        const double my = load_value(io, cf, cff, 2 * nc + c), E = load_value(io, cf, cff, 3 * nc + c);
        const double rinv = rcp(rho), u = mx * rinv, v = my * rinv;
        const double p = C.gm1 * E - C.gm1h * (mx * u + my * v), T = p * rinv;
        w[0][ly][lx] = rho;
        w[1][ly][lx] = u;
        w[2][ly][lx] = v;
        w[3][ly][lx] = p;
        w[4][ly][lx] = T;
        if (SUTH) {
            const double tt = T * C.inv_tref;
            w[5][ly][lx] = Gr.mu * (tt * sqrt(tt)) * ((1.0 + C.suth_s) / (tt + C.suth_s));
        }
    }
    __syncthreads();
    constexpr int NFX_ = (TX + 1) * TY, NF = NFX_ + TX * (TY + 1);
    for (int f = tid; f < NF; f += NT) {
        if (!(slow[f >> 5] >> (f & 31) & 1)) continue;
        const bool yd = f >= NFX_;
        const int g = yd ? f - NFX_ : f;
        const int fx = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int ym = yd ? fy + 1 : fy + 2, xm = yd ? fx + 2 : fx + 1, yp = fy + 2, xp = fx + 2;
        const int sy = yp - ym, sx = xp - xm;   // unit step along the normal
        double WL[4], WR[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            muscl(w[k][ym - sy][xm - sx], w[k][ym][xm], w[k][yp][xp], w[k][yp + sy][xp + sx], C.c_lo, C.c_hi, WL[k],
                  WR[k]);
        double vn = 0.0, vt = 0.0, ve = 0.0;
        const int N = yd ? 2 : 1, T = yd ? 1 : 2;
        if (VISC) {
            auto along = [&](const Arr &a) {   // four-cell difference along the face
                return (a[ym + sx][xm + sy] + a[yp + sx][xp + sy]) - (a[ym - sx][xm - sy] + a[yp - sx][xp - sy]);
            };
            visc2_terms<SUTH>(w[N][yp][xp] - w[N][ym][xm], w[T][yp][xp] - w[T][ym][xm], w[4][yp][xp] - w[4][ym][xm],
                              along(w[N]), along(w[T]), w[N][ym][xm] + w[N][yp][xp], w[T][ym][xm] + w[T][yp][xp],
                              SUTH ? w[SUTH ? 5 : 0][ym][xm] + w[SUTH ? 5 : 0][yp][xp] : 0.0, vk[yd ? 1 : 0], vn, vt, ve);
        }
        double g0, gn, gt, g3;
        roe2_nt<VISC>(WL[0], WL[N], WL[T], WL[3], WR[0], WR[N], WR[T], WR[3], C, g0, gn, gt, g3, vn, vt, ve);
        double *out = yd ? &fc.fy[0][fy][fx] : &fc.fx[0][fy][fx];
        const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
        out[0] = g0 * fs.up[0];
        out[ks] = (yd ? gt : gn) * fs.up[1];
        out[2 * ks] = (yd ? gn : gt) * fs.up[2];
        out[3 * ks] = g3 * fs.up[3];
    }
}

// One TX x TY tile as cart_tile, the primitives and faces in fixed point.
template <bool VISC, bool SUTH, class SH>
__device__ __forceinline__ void fixed_cart_tile(const StencilConsts &C, const GridRef Gr, const FixedVisc &V,
                                                const double (*vkd)[5], const StencilIO &io, int i0, int j0, unsigned char *smem_raw,
                                                size_t off = 0, size_t sb = 0)
{
    using namespace fx;
    constexpr int TX = SH::TX, TY = SH::TY, NT = SH::NT, EW = SH::EW, EH = SH::EH;
    constexpr int NFX_ = (TX + 1) * TY, NF = NFX_ + TX * (TY + 1);
    if (io.active && *at_bytes(io.active, sb) == 0) return;
    __shared__ FixedShared fs;
    __shared__ unsigned slow[(NF + 31) / 32];
    typedef FixedTile<SUTH, SH> FT;
    FT &tl = *reinterpret_cast<FT *>(smem_raw);
    Faces<double, SH> &fc = *reinterpret_cast<Faces<double, SH> *>(smem_raw + FixedSmem<SUTH, SH>::faces);
    const FixedConsts &F = C.fx;
    const int nx = Gr.nx, ny = Gr.ny;
    const size_t nc = (size_t)nx * ny;
    const int tid = threadIdx.x;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2, sb);
    int eR, eU;
    fixed_scales(io.base[off], io.base[off + 3 * nc], eR, eU);
    if (tid < 4) {
        // flux component k has the unit R U^(1, 2, 2, 3)
        const int e = eR + eU * (tid == 0 ? 1 : (tid == 3 ? 3 : 2)) - 62;
        fs.bx[tid] = Gr.hrdx * pow2(e);
        fs.by[tid] = Gr.hrdy * pow2(e);
        fs.up[tid] = pow2(-e);
    }
    if (tid == 0) {
        fs.vshift = eR + eU - V.e;
        fs.any_slow = 0;
    }
    if (VISC && tid < 10) fs.vk[tid / 5][tid % 5] = V.k[tid / 5][tid % 5];
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        const int gi = wrapi(i0 + lx - 2, nx), gj = wrapi(j0 + ly - 2, ny);
        const size_t c = off + (size_t)gj * nx + gi;
        const double q0 = load_value(io, cf, cff, c), q1 = load_value(io, cf, cff, nc + c);
        const double q2 = load_value(io, cf, cff, 2 * nc + c), q3 = load_value(io, cf, cff, 3 * nc + c);
        long long w[6];
        fixed_prim<VISC, SUTH>(q0, q1, q2, q3, eR, eU, F, w);
        tl.r[ly][lx] = w[0];
        tl.u[ly][lx] = w[1];
        tl.v[ly][lx] = w[2];
        tl.p[ly][lx] = w[3];
        if (VISC) tl.T[ly][lx] = w[4];
        if (SUTH) tl.g[ly][lx] = w[5];
    }
    __syncthreads();

    // one face per thread in full warp batches, the orientation a per-lane value
    // (as in cart_tile): it selects the cells and the order of u and v
    for (int bt = tid >> 5; bt < (NF + 31) / 32; bt += NT / 32) {
        const int f = bt * 32 + (tid & 31);
        bool bad = false;
        if (f < NF) {
            const bool yd = f >= NFX_;
            const int g = yd ? f - NFX_ : f;
            const int fx_ = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
            const int yp = fy + 2, xp = fx_ + 2;
            const int sn = yd ? EW : 1, st = yd ? 1 : EW;   // steps along the normal and along the face
            const int ip = yp * EW + xp, im = ip - sn;
            const long long *pr = &tl.r[0][0], *pp = &tl.p[0][0];
            const long long *pn = yd ? &tl.v[0][0] : &tl.u[0][0], *pt = yd ? &tl.u[0][0] : &tl.v[0][0];
            FixedState L, R;
            fixed_muscl(pr[im - sn], pr[im], pr[ip], pr[ip + sn], F, L.r.v, R.r.v);
            fixed_muscl_p(pp[im - sn], pp[im], pp[ip], pp[ip + sn], F, L.p, R.p);
            const long long nm = pn[im], np = pn[ip], tm = pt[im], tp = pt[ip];
            const long long nm2 = pn[im - sn], np2 = pn[ip + sn], tm2 = pt[im - sn], tp2 = pt[ip + sn];
            fixed_muscl(nm2, nm, np, np2, F, L.n.v, R.n.v);
            fixed_muscl(tm2, tm, tp, tp2, F, L.t.v, R.t.v);
            // the good flags are the lowest bits of u
            unsigned flag = yd ? (unsigned)(tm | tp | tm2 | tp2) : (unsigned)(nm | np | nm2 | np2);
            Fx<0> vn{0}, vt{0}, ve{0};
            if (VISC) {
                const long long *vk = fs.vk[yd ? 1 : 0];
                const long long *pT = &tl.T[0][0];
                const long long nu0 = pn[im + st], nu1 = pn[ip + st], nd0 = pn[im - st], nd1 = pn[ip - st];
                const long long tu0 = pt[im + st], tu1 = pt[ip + st], td0 = pt[im - st], td1 = pt[ip - st];
                flag |= yd ? (unsigned)(tu0 | tu1 | td0 | td1) : (unsigned)(nu0 | nu1 | nd0 | nd1);
                const Fx<0> dnt = {(nu0 + nu1) - (nd0 + nd1)}, dtt = {(tu0 + tu1) - (td0 + td1)};
                if (outside<1>(dnt) || outside<1>(dtt)) bad = true;
                // coefficients below 1/2: the sums stay below 1
                Fx<0> tnn = {mul62(np - nm, vk[0]) + mul62(dtt.v, vk[1])};
                Fx<0> tnt = {mul62(dnt.v, vk[2]) + mul62(tp - tm, vk[3])};
                Fx<0> q = {mul62(pT[ip] - pT[im], vk[4])};
                if (SUTH) {
                    const long long *pg = &tl.g[0][0];
                    const Fx<2> mus = {pg[im] + pg[ip]};   // below 4
                    Fx<2> a = mul<2>(tnn, mus), b = mul<2>(tnt, mus), c = mul<2>(q, mus);
                    if (outside<3>(a) || outside<3>(b) || outside<3>(c)) bad = true;
                    tnn = to<0>(a);
                    tnt = to<0>(b);
                    q = to<0>(c);
                }
                const Fx<0> s2 = half_of(Fx<0>{mul62(nm + np, tnn.v) + mul62(tm + tp, tnt.v)});
                const int sh = fs.vshift;
                const int shc = sh < 63 ? (sh < 0 ? 0 : sh) : 63;
                if (sh < 0) bad = true;
                vn = {tnn.v >> shc};
                vt = {tnt.v >> shc};
                ve = {(s2.v + q.v) >> shc};
            }
            if (flag & 1) bad = true;
            Fx<0> G[4];
            fixed_roe<true>(L, R, F, vn, vt, ve, G, bad);
            if (!bad) {
                double *out = yd ? &fc.fy[0][fy][fx_] : &fc.fx[0][fy][fx_];
                const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
                out[0] = (double)G[0].v;
                out[ks] = (double)(yd ? G[2].v : G[1].v);
                out[2 * ks] = (double)(yd ? G[1].v : G[2].v);
                out[3 * ks] = (double)G[3].v;
            }
        }
        const unsigned left = __ballot_sync(0xffffffffu, bad);
        if ((tid & 31) == 0) {
            slow[bt] = left;
            if (left) fs.any_slow = 1;
        }
    }
    __syncthreads();
    if (fs.any_slow) {
        slow_faces<VISC, SUTH, SH>(C, Gr, io, i0, j0, off, sb, smem_raw, fc, fs, slow, vkd);
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
                const double t = io.sub ? -(dX * fs.bx[k] + (dY * fs.by[k] + io.sub[e])) : -(dX * fs.bx[k] + dY * fs.by[k]);
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
    fixed_cart_tile<VISC, SUTH, SH>(C, GridRef{C.nx, C.ny, C.hrdx, C.hrdy, C.mu}, C.fxv, C.vk, io,
                                    blockIdx.x * SH::TX, blockIdx.y * SH::TY, smem_raw);
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
    fixed_cart_tile<VISC, SUTH, SH>(C, GridRef{I.nx, I.ny, I.hrdx, I.hrdy, I.mu}, I.fxv, I.vk, io, (t % ntx) * SH::TX,
                                    (t / ntx) * SH::TY, smem_raw, I.off, (size_t)k * bt.stride_bytes);
}

// ============================== curvilinear grid ===============================
// The same for curv_kernel's grids.  A face's reconstructed velocities are
// rotated into its (normal, tangential) frame, fixed_roe runs there (the flux is
// invariant under rotation) and the momentum fluxes are rotated back: twelve
// products more than the uniform faces.  The normals are 62-bit fractions; the
// diamond coefficients of a face are mantissas with one exponent per face
// (they span the inverse cell widths, 1e-2 to 1e4 on a stretched grid), which
// the viscous terms are shifted by.  Residual on the 256 x 512 O-grid with
// Sutherland's law: 134 -> 45 us.

__device__ __forceinline__ FixedMetric fixed_metric(double nx, double ny, double len, double c0, double c1, double c2,
                                                    double c3)
{
    const auto unit = [](double x) {   // |x| <= 1 in 62 bits, 1 just below
        const long long one = 1ll << 62, v = (long long)(x * 4611686018427387904.0);
        return v >= one ? one - 1 : (v <= -one ? 1 - one : v);
    };
    FixedMetric m{unit(nx), unit(ny), 0, 0, 0, 0, 0.5 * len, 1 << 20};
    const double c[4] = {c0, 0.25 * c1, c2, 0.25 * c3};
    double big = 0.0;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        big = fmax(big, fabs(c[k]));
        ok = ok && isfinite(c[k]);
    }
    const int x = (__double2hiint(big) >> 20) - 1022;   // big in [2^(x-1), 2^x)
    if (!ok || x < -900 || x > 900) return m;             // an exponent no state's units reach
    m.e = x + 1;
    const double up = pow2(62 - x - 1);
    m.c0 = (long long)(c[0] * up);
    m.c1 = (long long)(c[1] * up);
    m.c2 = (long long)(c[2] * up);
    m.c3 = (long long)(c[3] * up);
    return m;
}

// x 2^l for l in [0, 30]; bad where it would reach 1/2
__device__ __forceinline__ fx::Fx<0> scale_up(fx::Fx<0> x, int l, bool &bad)
{
    const int top = (int)(x.v >> 31) >> (30 - l);   // 0 or -1 where 2^l x stays below 1/2
    if (top != 0 && top != -1) bad = true;
    return {(long long)((unsigned long long)x.v << l)};
}

// ghost rules of one tile cell (global indices gi, gj): the source cell, whether
// its velocity is mirrored, whether it is the free stream
__device__ __forceinline__ void curv_source(const StencilConsts &C, int &gi, int &gj, bool &mirror, bool &inf)
{
    const int nx = C.nx, ny = C.ny;
    mirror = inf = false;
    if (gi < 0 || gi >= nx) {
        const int b = gi < 0 ? C.bc[0] : C.bc[1];
        if (b == ROK_BC_PERIODIC) gi = wrapi(gi, nx);
        else if (b == ROK_BC_WALL) { gi = gi < 0 ? -gi - 1 : 2 * nx - 1 - gi; mirror = !mirror; }
        else inf = true;
    }
    if (!inf && (gj < 0 || gj >= ny)) {
        const int b = gj < 0 ? C.bc[2] : C.bc[3];
        if (b == ROK_BC_PERIODIC) gj = wrapi(gj, ny);
        else if (b == ROK_BC_WALL) { gj = gj < 0 ? -gj - 1 : 2 * ny - 1 - gj; mirror = !mirror; }
        else inf = true;
    }
    // a tile cell past the last valid index of a partial tile may still be out of
    // range after the rules above; clamp it (its faces are never used)
    gi = min(max(gi, 0), nx - 1);
    gj = min(max(gj, 0), ny - 1);
}

// the faces left out by the fixed-point path, in binary64 (as slow_faces)
template <bool VISC, bool SUTH, class SH>
__device__ __noinline__ void slow_curv_faces(const StencilConsts &C, const CurvGeom &G, const StencilIO &io, int i0,
                                             int j0, unsigned char *smem_raw, Faces<double, SH> &fc,
                                             const FixedShared &fs, const unsigned *slow)
{
    constexpr int TX = SH::TX, TY = SH::TY, NT = SH::NT, EW = SH::EW, EH = SH::EH;
    typedef double Arr[EH][EW];
    Arr *w = reinterpret_cast<Arr *>(smem_raw);   // rho, u, v, p, T, mu
    const int nx = C.nx, tid = threadIdx.x;
    const size_t nc = (size_t)nx * C.ny;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2);
    __syncthreads();
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        int gi = i0 + lx - 2, gj = j0 + ly - 2;
        bool mirror, inf;
        curv_source(C, gi, gj, mirror, inf);
        double q[6];
        if (inf) {
#pragma unroll
            for (int k = 0; k < 6; ++k) q[k] = C.prim_inf[k];
        } else {
            const size_t c = (size_t)gj * nx + gi;
            const double rho = load_value(io, cf, cff, c), mx = load_value(io, cf, cff, nc + c);
            const double my = load_value(io, cf, cff, 2 * nc + c), E = load_value(io, cf, cff, 3 * nc + c);
            const double rinv = rcp(rho);
            q[0] = rho;
            q[1] = mx * rinv;
            q[2] = my * rinv;
            q[3] = C.gm1 * E - C.gm1h * (mx * q[1] + my * q[2]);
            q[4] = q[3] * rinv;
            if (SUTH) {
                const double tt = q[4] * C.inv_tref;
                q[5] = C.mu * (tt * sqrt(tt)) * ((1.0 + C.suth_s) / (tt + C.suth_s));
            }
        }
        w[0][ly][lx] = q[0];
        w[1][ly][lx] = mirror ? -q[1] : q[1];
        w[2][ly][lx] = mirror ? -q[2] : q[2];
        w[3][ly][lx] = q[3];
        w[4][ly][lx] = q[4];
        if (SUTH) w[SUTH ? 5 : 0][ly][lx] = q[5];
    }
    __syncthreads();
    constexpr int NFX_ = (TX + 1) * TY, NF = NFX_ + TX * (TY + 1);
    for (int f = tid; f < NF; f += NT) {
        if (!(slow[f >> 5] >> (f & 31) & 1)) continue;
        const bool yd = f >= NFX_;
        const int g = yd ? f - NFX_ : f;
        const int fx = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int gi = i0 + fx, gj = j0 + fy;
        const size_t fi = yd ? (size_t)gj * nx + gi : (size_t)gj * (nx + 1) + gi;
        const int ym = yd ? fy + 1 : fy + 2, xm = yd ? fx + 2 : fx + 1, yp = fy + 2, xp = fx + 2;
        const int sy = yp - ym, sx = xp - xm;            // unit step along the normal
        const int ty = yd ? 0 : 1, txo = yd ? -1 : 0;    // tangential step
        double WL[4], WR[4], Fl[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            muscl(w[k][ym - sy][xm - sx], w[k][ym][xm], w[k][yp][xp], w[k][yp + sy][xp + sx], C.c_lo, C.c_hi, WL[k],
                  WR[k]);
        const double nxf = yd ? G.jn_x[fi] : G.in_x[fi], nyf = yd ? G.jn_y[fi] : G.in_y[fi];
        double v1 = 0.0, v2 = 0.0, v3 = 0.0;
        if (VISC) {
            auto across = [&](const Arr &a) { return a[yp][xp] - a[ym][xm]; };
            auto along = [&](const Arr &a) {
                return (a[ym + ty][xm + txo] + a[yp + ty][xp + txo]) - (a[ym - ty][xm - txo] + a[yp - ty][xp - txo]);
            };
            visc_n2_terms<SUTH>(nxf, nyf, yd ? G.jc0[fi] : G.ic0[fi], quarter(yd ? G.jc1[fi] : G.ic1[fi]),
                                yd ? G.jc2[fi] : G.ic2[fi], quarter(yd ? G.jc3[fi] : G.ic3[fi]), across(w[1]),
                                across(w[2]), across(w[4]), along(w[1]), along(w[2]), along(w[4]),
                                w[1][ym][xm] + w[1][yp][xp], w[2][ym][xm] + w[2][yp][xp],
                                SUTH ? w[SUTH ? 5 : 0][ym][xm] + w[SUTH ? 5 : 0][yp][xp] : 0.0, C, v1, v2, v3);
        }
        roe_n2<VISC>(WL, WR, nxf, nyf, C, Fl, v1, v2, v3);
        const double len = half(yd ? G.jl[fi] : G.il[fi]);
        double *out = yd ? &fc.fy[0][fy][fx] : &fc.fx[0][fy][fx];
        const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k * ks] = (Fl[k] * len) * fs.up[k];
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
    __shared__ FixedShared fs;
    __shared__ unsigned slow[(NF + 31) / 32];
    __shared__ long long winf[6];
    typedef FixedTile<SUTH, SH> FT;
    FT &tl = *reinterpret_cast<FT *>(smem_raw);
    Faces<double, SH> &fc = *reinterpret_cast<Faces<double, SH> *>(smem_raw + FixedSmem<SUTH, SH>::faces);
    const FixedConsts &F = C.fx;
    const int nx = C.nx, ny = C.ny;
    const size_t nc = (size_t)nx * ny;
    const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
    const int tid = threadIdx.x;
    double cf[kMaxAdd], cff, s1, s2;
    coefs(io, cf, cff, s1, s2);
    int eR, eU;
    fixed_scales(io.base[0], io.base[3 * nc], eR, eU);
    if (tid < 4) {
        const int e = eR + eU * (tid == 0 ? 1 : (tid == 3 ? 3 : 2)) - 62;
        fs.bx[tid] = pow2(e);
        fs.up[tid] = pow2(-e);
    }
    if (tid == 32) {   // the free stream (far-field ghosts)
        fs.any_slow = 0;
        bool bad = false;
        const Fx<0> r = from_double<0>(C.prim_inf[0], eR, bad), u = from_double<0>(C.prim_inf[1], eU, bad);
        const Fx<0> v = from_double<0>(C.prim_inf[2], eU, bad), T = from_double<0>(C.prim_inf[4], 2 * eU, bad);
        const Fx<-3> p = from_double<-3>(C.prim_inf[3], eR + 2 * eU, bad);
        if (!in_window<4>(r) || !in_window<8>(p) || outside<1>(u) || outside<1>(v) || outside<1>(T)) bad = true;
        if (SUTH && F.g_inf < 0) bad = true;
        winf[0] = r.v;
        winf[1] = (u.v & ~1ll) | (bad ? 1 : 0);
        winf[2] = v.v;
        winf[3] = p.v;
        winf[4] = T.v;
        winf[5] = F.g_inf;
    }
    __syncthreads();
    for (int idx = tid; idx < EW * EH; idx += NT) {
        const int lx = idx % EW, ly = idx / EW;
        int gi = i0 + lx - 2, gj = j0 + ly - 2;
        bool mirror, inf;
        curv_source(C, gi, gj, mirror, inf);
        long long w[6];
        if (inf) {
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = winf[k];
        } else {
            const size_t c = (size_t)gj * nx + gi;
            const double q0 = load_value(io, cf, cff, c), q1 = load_value(io, cf, cff, nc + c);
            const double q2 = load_value(io, cf, cff, 2 * nc + c), q3 = load_value(io, cf, cff, 3 * nc + c);
            fixed_prim<VISC, SUTH>(q0, q1, q2, q3, eR, eU, F, w);
        }
        if (mirror) {
            w[1] = -(w[1] & ~1ll) | (w[1] & 1);
            w[2] = -w[2];
        }
        tl.r[ly][lx] = w[0];
        tl.u[ly][lx] = w[1];
        tl.v[ly][lx] = w[2];
        tl.p[ly][lx] = w[3];
        if (VISC) tl.T[ly][lx] = w[4];
        if (SUTH) tl.g[ly][lx] = w[5];
    }
    __syncthreads();

    for (int bt = tid >> 5; bt < (NF + 31) / 32; bt += NT / 32) {
        const int f = bt * 32 + (tid & 31);
        const bool yd = f >= NFX_;
        const int g = yd ? f - NFX_ : f;
        const int fx_ = yd ? g % TX : g % (TX + 1), fy = yd ? g / TX : g / (TX + 1);
        const int gi = i0 + fx_, gj = j0 + fy;
        bool bad = false;
        if (f < NF && (yd ? (gi < nx && gj <= ny) : (gi <= nx && gj < ny))) {
            const longlong2 *mp = reinterpret_cast<const longlong2 *>(yd ? G.fj + ((size_t)gj * nx + gi)
                                                                         : G.fi + ((size_t)gj * (nx + 1) + gi));
            const longlong2 mn = __ldg(mp), ml = __ldg(mp + 3);   // normal; half length, exponent
            const Fx<0> mnx = {mn.x}, mny = {mn.y};
            const int ip = (fy + 2) * EW + fx_ + 2;
            const int sn = yd ? EW : 1, im = ip - sn;
            const int st = yd ? -1 : EW;   // step along the face: +1 row on i-faces, -1 column on j-faces
            const long long *pr = &tl.r[0][0], *pu = &tl.u[0][0], *pv = &tl.v[0][0], *pp = &tl.p[0][0];
            FixedState L, R;
            Fx<0> uL, uR, vL, vR;
            fixed_muscl(pr[im - sn], pr[im], pr[ip], pr[ip + sn], F, L.r.v, R.r.v);
            fixed_muscl_p(pp[im - sn], pp[im], pp[ip], pp[ip + sn], F, L.p, R.p);
            const long long um = pu[im], up = pu[ip], um2 = pu[im - sn], up2 = pu[ip + sn];
            const long long vm = pv[im], vp = pv[ip];
            fixed_muscl(um2, um, up, up2, F, uL.v, uR.v);
            fixed_muscl(pv[im - sn], vm, vp, pv[ip + sn], F, vL.v, vR.v);
            unsigned flag = (unsigned)(um | up | um2 | up2);
            if (outside<1>(uL) || outside<1>(uR) || outside<1>(vL) || outside<1>(vR)) bad = true;
            L.n = mul<0>(uL, mnx) + mul<0>(vL, mny);
            R.n = mul<0>(uR, mnx) + mul<0>(vR, mny);
            L.t = mul<0>(vL, mnx) - mul<0>(uL, mny);
            R.t = mul<0>(vR, mnx) - mul<0>(uR, mny);
            Fx<0> v1{0}, v2{0}, ve{0};
            if (VISC) {
                const long long *pT = &tl.T[0][0];
                const longlong2 ca = __ldg(mp + 1), cb = __ldg(mp + 2);
                const Fx<0> c0 = {ca.x}, c1 = {ca.y}, c2 = {cb.x}, c3 = {cb.y};
                const long long a0 = pu[im + st], a1 = pu[ip + st], b0 = pu[im - st], b1 = pu[ip - st];
                flag |= (unsigned)(a0 | a1 | b0 | b1);
                Fx<0> dVu = {(a0 + a1) - (b0 + b1)};
                Fx<0> dVv = {(pv[im + st] + pv[ip + st]) - (pv[im - st] + pv[ip - st])};
                Fx<0> dVT = {(pT[im + st] + pT[ip + st]) - (pT[im - st] + pT[ip - st])};
                Fx<0> dCu = {up - um}, dCv = {vp - vm}, dCT = {pT[ip] - pT[im]};
                if (outside<1>(dVu) || outside<1>(dVv) || outside<1>(dVT)) bad = true;
                // the terms are those of the mantissas times 2^-sh.  On thin cells
                // (sh < 0) the differences are scaled up first, as far as they allow
                // (by l1), the terms by the rest: the products then drop no bits that matter
                const int sh = eR + eU - C.fxv.e - (int)ml.y;
                int l1 = 0, l2 = 0;
                if (sh < 0) {
                    const Fx<0> *d[6] = {&dCu, &dCv, &dCT, &dVu, &dVv, &dVT};
                    int m = 0;
#pragma unroll
                    for (int k = 0; k < 6; ++k) m |= hi_word(d[k]->v) ^ (hi_word(d[k]->v) >> 31);
                    l1 = min(max(__clz(m) - 3, 0), -sh);
                    l2 = min(-sh - l1, 30);
                    if (-sh - l1 > 30) bad = true;
                    dCu.v <<= l1;
                    dCv.v <<= l1;
                    dCT.v <<= l1;
                    dVu.v <<= l1;
                    dVv.v <<= l1;
                    dVT.v <<= l1;
                }
                // coefficients below 1/2, across-differences below 1, along-differences below 1/2: gradients below 3/4
                const Fx<0> ux = mul<0>(dCu, c0) + mul<0>(dVu, c1), uy = mul<0>(dCu, c2) + mul<0>(dVu, c3);
                const Fx<0> vx = mul<0>(dCv, c0) + mul<0>(dVv, c1), vy = mul<0>(dCv, c2) + mul<0>(dVv, c3);
                const Fx<0> Tx = mul<0>(dCT, c0) + mul<0>(dVT, c1), Ty = mul<0>(dCT, c2) + mul<0>(dVT, c3);
                const Fx<0> sxy = half_of(uy + vx);
                const Fx<0> k0 = {C.fxv.k[0][0]}, k1 = {C.fxv.k[0][1]}, k2 = {C.fxv.k[0][2]}, k3 = {C.fxv.k[0][3]};
                Fx<0> txx = mul<0>(ux, k0) + mul<0>(vy, k1), tyy = mul<0>(vy, k0) + mul<0>(ux, k1);
                const Fx<0> txh = mul<0>(sxy, k2);   // half of txy
                Fx<0> txy = txh + txh;
                Fx<0> q = mul<0>(mul<0>(Tx, mnx) + mul<0>(Ty, mny), k3);
                Fx<0> t1 = mul<0>(txx, mnx) + mul<0>(txy, mny), t2 = mul<0>(txy, mnx) + mul<0>(tyy, mny);
                if (outside<1>(t1) || outside<1>(t2) || outside<1>(q)) bad = true;
                if (SUTH) {
                    const long long *pg = &tl.g[0][0];
                    const Fx<2> mus = {pg[im] + pg[ip]};   // below 4
                    const Fx<2> a = mul<2>(t1, mus), b = mul<2>(t2, mus), c = mul<2>(q, mus);
                    if (outside<3>(a) || outside<3>(b) || outside<3>(c)) bad = true;
                    t1 = to<0>(a);
                    t2 = to<0>(b);
                    q = to<0>(c);
                }
                const Fx<0> w = half_of(mul<0>(Fx<0>{um + up}, t1) + mul<0>(Fx<0>{vm + vp}, t2)) + q;
                if (sh < 0) {
                    v1 = scale_up(t1, l2, bad);
                    v2 = scale_up(t2, l2, bad);
                    ve = scale_up(w, l2, bad);
                } else {
                    const int r = min(sh, 63);
                    v1 = {t1.v >> r};
                    v2 = {t2.v >> r};
                    ve = {w.v >> r};
                }
            }
            if (flag & 1) bad = true;
            Fx<0> g4[4];
            fixed_roe<false>(L, R, F, Fx<0>{0}, Fx<0>{0}, ve, g4, bad);
            // rotate halves of the momentum fluxes, tested below 1/2
            const Fx<0> gn = half_of(g4[1]), gt = half_of(g4[2]);
            if (outside<1>(gn) || outside<1>(gt)) bad = true;
            const Fx<0> m1 = mul<0>(gn, mnx) - mul<0>(gt, mny), m2 = mul<0>(gn, mny) + mul<0>(gt, mnx);
            if (!bad) {
                const double len = __longlong_as_double(ml.x);
                double *out = yd ? &fc.fy[0][fy][fx_] : &fc.fx[0][fy][fx_];
                const int ks = yd ? (TY + 1) * TX : TY * (TX + 1);
                out[0] = (double)g4[0].v * len;
                out[ks] = (double)(m1.v + m1.v - v1.v) * len;
                out[2 * ks] = (double)(m2.v + m2.v - v2.v) * len;
                out[3 * ks] = (double)g4[3].v * len;
            }
        }
        const unsigned left = __ballot_sync(0xffffffffu, bad);
        if ((tid & 31) == 0) {
            slow[bt] = left;
            if (left) fs.any_slow = 1;
        }
    }
    __syncthreads();
    if (fs.any_slow) {
        slow_curv_faces<VISC, SUTH, SH>(C, G, io, i0, j0, smem_raw, fc, fs, slow);
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
                epilogue_store(io, s1, s2, k * nc + c, -((dX + dY) * (iv * fs.bx[k])));
            }
        }
    }
}
