// dg_stage_f64pt.cuh -- the FP64 stage for small meshes, one lane per Gauss
// point (or mode) of an element.  Included by dg_kernels.cuh.
//
// What bounds it and why this shape.  A GB300 SM executes one FP64 warp
// instruction in about 19 cycles, but one of its four quarters takes 64 cycles
// for each, one after the other, however few lanes are active and however
// independent the operations are.  On a mesh with less than a warp per quarter
// the stage therefore takes (FP64 instructions of a warp) x 64 cycles, and
// lanes are free: with N lanes per element (stage_tile) a warp has some 600 to
// 1000 of them, with N^2 lanes about 300.  A warp here holds 32 / N^2 elements and
// depends on no other warp: it evaluates its elements' four edges itself, from
// its own and the four neighbours' modes (a third more operations in all, so
// the tiles win on meshes that fill the chip; the line is at launch_stage_n).
// Both elements of an edge evaluate its flux with the same operations on the
// same traces, so the flux is single-valued to the bit.
#pragma once

namespace dgk {

template <int N>
struct PtGeo {
    static constexpr int NP = N * N, EL = 3 * NP;
    static constexpr int E = 32 / NP;                // elements of a warp
    // shared memory of one element, in doubles
    static constexpr int U = 0;                      // modes of the element and its W, E, S, N neighbours
    static constexpr int V = U + 5 * EL;             // edge sums of the modes
    static constexpr int T = V + 24 * N;             // traces: own W, E, S, N, then the neighbours' facing ones
    static constexpr int FX = T + 24 * N;            // edge fluxes W, E, S, N
    static constexpr int P = FX + 12 * N;            // per-point values between the passes
    static constexpr int LEN = (P + 8 * NP) | 1;
};

template <int N>
__global__ void __launch_bounds__(32) pt_stage_kernel(const StageArgs<double> A)
{
    using GE = PtGeo<N>;
    constexpr int NP = GE::NP, EL = GE::EL;
    __shared__ double sm[GE::E * GE::LEN];
    const BasisTab<double> &B = c_basis[N - 1];
    const int lane = threadIdx.x;
    const int g = min(lane / NP, GE::E - 1), m = min(lane - g * NP, NP - 1), hi = m / N, lo = m - hi * N;
    const int nel = A.nlon * A.nlat, e0 = blockIdx.x * GE::E + g;
    const bool valid = lane < GE::E * NP && e0 < nel;   // (other lanes repeat a valid lane's work on its element, and store nothing)
    const int e = min(e0, nel - 1), j = e / A.nlon, i = e - j * A.nlon;
    const bool store = lane < GE::E * NP;               // shared memory: each lane its own values
    double *const s = sm + g * GE::LEN;
    const RowTab<double> *const RT = A.rows + j;

    // tables of this lane's row and column, before the previous stage's end
    double LVlo[N], LVhi[N], QT[N], PT[N], WD[N], WV[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        LVlo[q] = B.LV[q][lo];
        LVhi[q] = B.LV[q][hi];
        QT[q] = __ldg(&RT->QT[q][hi]);
        PT[q] = __ldg(&RT->PT[q][hi]);
        WD[q] = B.WLD[lo][q];
        WV[q] = B.WLV[lo][q];
    }
    const double csw = __ldg(&RT->CSW[hi]), cse = __ldg(&RT->CSE[hi]), rho = __ldg(&RT->rho[hi]);
    const double cGc = __ldg(&RT->cGc[hi]), sR = __ldg(&RT->sR[hi]), fc = __ldg(&RT->fc[hi]);
    const double se_lo = B.SE[lo], sw_lo = B.SW[lo];
    const double ce_s = A.cG * __ldg(&RT->ce_s), ce_n = A.cG * __ldg(&RT->ce_n);
    pdl_wait();
    const double ga_l = A.galpha ? A.galpha[0] : 0.0, ga_t = A.galpha ? A.galpha[1] : 0.0;
    unsigned st = 0;

    // ---- S0: stage state of the element and of its neighbours (periodic in
    //      lambda, and in theta where the mesh wraps; none across a pole)
    const bool hasS = j > 0 || A.halo_s, hasN = j < A.nlat - 1 || A.halo_n;
    {
        const int jS = A.wrap && j == 0 ? A.nlat - 1 : j - 1, jN = A.wrap && j == A.nlat - 1 ? 0 : j + 1;
        const int nb_j[5] = {j, j, j, hasS ? jS : j, hasN ? jN : j};
        const int nb_i[5] = {i, i > 0 ? i - 1 : A.nlon - 1, i < A.nlon - 1 ? i + 1 : 0, i, i};
        double v[5][3], d[5][3];
#pragma unroll
        for (int n = 0; n < 5; ++n)
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const long long o = ((long long)nb_j[n] * A.nlon + nb_i[n]) * EL + f * NP + m;
                v[n][f] = __ldg(A.base + o);
                d[n][f] = A.inc ? __ldg(A.inc + o) : 0.0;
            }
#pragma unroll
        for (int n = 0; n < 5; ++n)
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                if (A.inc) v[n][f] += d[n][f];
                if (store) s[GE::U + n * EL + f * NP + m] = v[n][f];
            }
    }
    __syncwarp();

    // ---- S1 lambda sums (lane (b, alpha)), S4 edge sums over the modes
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        double t = 0.0;
#pragma unroll
        for (int a = 0; a < N; ++a) t = fma(LVlo[a], s[GE::U + f * NP + hi * N + a], t);
        if (store) s[GE::P + f * NP + m] = t;
    }
    // trace line l: own W, E, S, N (0..3), the neighbours' facing edges (4..7)
#pragma unroll 2
    for (int it = m; it < 24 * N; it += NP) {
        const int l = it / (3 * N), f = (it - l * 3 * N) / N;   // point / mode index it % N = lo
        const bool lam = (l & 2) == 0, plus = l < 4 ? (l & 1) : !(l & 1);
        const double *src = s + GE::U + (l < 4 ? 0 : l - 3) * EL + f * NP + (lam ? lo * N : lo);
        double v = 0.0;
#pragma unroll
        for (int x = 0; x < N; ++x) v = fma(plus ? B.SE[x] : B.SW[x], src[lam ? x : x * N], v);
        if (store) s[GE::V + it] = v;
    }
    __syncwarp();
    double qn[3];   // values at the Gauss point (alpha = lo, beta = hi)
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        qn[f] = 0.0;
#pragma unroll
        for (int b = 0; b < N; ++b) qn[f] = fma(LVhi[b], s[GE::P + f * NP + b * N + lo], qn[f]);
    }
#pragma unroll 2
    for (int it = m; it < 24 * N; it += NP) {
        double t = 0.0;
#pragma unroll
        for (int x = 0; x < N; ++x) t = fma(LVlo[x], s[GE::V + it - lo + x], t);
        if (store) s[GE::T + it] = t;
    }
    __syncwarp();

    // ---- S5: Rusanov fluxes of the four edges, one point per lane; n / t the
    //      momentum normal / tangential to the edge
#pragma unroll 1
    for (int it = m; it < 4 * N; it += NP) {
        const int side = it / N, k = it - side * N;
        const bool lam = side < 2, flip = side & 1;   // E and N: the element is the lower side
        const double *const own = s + GE::T + side * 3 * N + k, *const oth = own + 12 * N;
        const double *const pl = flip ? own : oth, *const pr = flip ? oth : own;
        const int in = lam ? N : 2 * N, itg = lam ? 2 * N : N;
        const double L[3] = {pl[0], pl[in], pl[itg]}, R[3] = {pr[0], pr[in], pr[itg]};
        const double c = lam ? A.cF : side == 2 ? ce_s : ce_n;
        double o[3];
        unsigned sq = 0;
        rusanov_lam(L, R, A.href, A.g, c, o, sq, lam ? ga_l : ga_t);
        const bool there = lam || (side == 2 ? hasS : hasN);   // pole edge: zero flux
        if (there) st |= sq;
        if (store) {
            double *const fx = s + GE::FX + side * 3 * N + k;
            fx[0] = there ? o[0] : 0.0;
            fx[in] = there ? o[1] : 0.0;
            fx[itg] = there ? o[2] : 0.0;
        }
    }

    // ---- S2: fluxes and sources at the lane's Gauss point
    {
        const double hp = qn[0], hu = qn[1], hv = qn[2], h = A.href + hp;
        check_depth(h, st);
        const double rh = rcp(h), u = hu * rh, v = hv * rh, P = pressure(hp, A.href, A.g);
        const double F0 = A.cF * hu, G0 = cGc * hv, K = fma(u, sR, fc);
        double *const p = s + GE::P + m;
        // (the lambda sums in P were read before the last barrier)
        if (store) {
            p[0 * NP] = F0;
            p[1 * NP] = fma(F0, u, A.cF * P);
            p[2 * NP] = F0 * v;
            p[3 * NP] = G0;
            p[4 * NP] = G0 * u;
            p[5 * NP] = fma(G0, v, cGc * P);
            p[6 * NP] = K * hv;
            p[7 * NP] = fma(-K, hu, -(P * sR));
        }
    }
    __syncwarp();

    // ---- S3 theta sums with the inverse mass matrix folded in, S6 N / S lift
    //      (lane (b, alpha))
    double X1[3], X2[3];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        X1[f] = 0.0;
        X2[f] = fma(csw, s[GE::FX + (2 * 3 + f) * N + lo], -(cse * s[GE::FX + (3 * 3 + f) * N + lo]));
#pragma unroll
        for (int q = 0; q < N; ++q) {
            X1[f] = fma(QT[q], s[GE::P + f * NP + q * N + lo], X1[f]);
            X2[f] = fma(PT[q], s[GE::P + (3 + f) * NP + q * N + lo], X2[f]);
            if (f > 0) X2[f] = fma(QT[q], s[GE::P + (5 + f) * NP + q * N + lo], X2[f]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int f = 0; f < 3; ++f)
        if (store) {
            s[GE::P + f * NP + m] = X1[f];
            s[GE::P + (3 + f) * NP + m] = X2[f];
        }
    __syncwarp();

    // ---- S3 lambda sums and S6 E / W lift (lane (b, a)), S8 combine and store
    const double cdt = A.cc * A.dt, adt = A.ca * A.dt;
    unsigned chb = 0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        double yw = 0.0, ye = 0.0, k = 0.0;
#pragma unroll
        for (int q = 0; q < N; ++q) {
            yw = fma(QT[q], s[GE::FX + f * N + q], yw);
            ye = fma(QT[q], s[GE::FX + (3 + f) * N + q], ye);
            k = fma(WD[q], s[GE::P + f * NP + hi * N + q], fma(WV[q], s[GE::P + (3 + f) * NP + hi * N + q], k));
        }
        k = fma(sw_lo, yw, fma(-se_lo, ye, k));
        if (f == 2 && lo == 0) k = fma(A.P0, rho, k);
        if (valid) {
            const size_t off = (size_t)e * EL + f * NP + m;
            chb = nf_acc_bits(k, chb);
            if (A.out_rhs) A.out_rhs[off] = k;
            const double inc = A.inc ? A.inc[off] : 0.0, acc = A.acc_in ? A.acc_in[off] : 0.0;
            const double ci = A.ci * inc;
            if (A.inc_out) A.inc_out[off] = fma(cdt, k, ci);
            if (A.acc_out) A.acc_out[off] = fma(adt, k, acc);
            if (A.out_base) {   // (FP64 keeps no low part)
                const double hi64 = A.base[off] + fma(cdt, k, A.acc_in ? fma(A.cd, acc, ci) : ci);
                A.out_base[off] = hi64;
                chb = nf_acc_bits(hi64, chb);
            }
        }
    }
    if (nf_bits(chb)) st |= DG_STATUS_NONFINITE;
    if (st && valid) atomicOr(A.status, st);
    pdl_launch_dependents();
}

}  // namespace dgk
