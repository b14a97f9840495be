// d3gb_backward.cu -- hand-written backward of (E, F) for damping refits.
// The handle's precision selects the form of the backward: FP64 throughout, or (mixed form) the forward's mixed arithmetic for the values --
// the double-single Eq. 4 term and chain coefficient, float-float Eq. 3
// exponents, FP32 pair math on split positions -- with FP32 tangents.  GB300
// runs FP64 at 1/64 of the FP32 rate, so the FP64 passes bound the mixed form's
// time otherwise.
//
// For a loss L(E, F) with upstream gradients gE = dL/dE (per structure) and
// gF = dL/dF (per atom):
//   dL/dtheta = sum_s gE_s dE_s/dtheta + sum_i gF_i . dF_i/dtheta
//             = sum_s gE_s dE_s/dtheta - d/dtheta (d/dt E(x + t gF))
//   dL/dx     = -gE F + J^T gF,  J = dF/dx = -Hessian (symmetric), so J^T gF = d/dt F(x + t gF).
// Both second-order terms are directional derivatives along u = gF.  They are
// obtained by running the whole evaluation (Eq. 4 coordination numbers, Eq. 3
// weights, Eq. 2 pair terms with their analytic derivatives in s6, s8, a1, a2,
// and the coordination-number chain rule) once with every quantity's derivative
// along u beside its value.  The coordination numbers are recomputed; the FP64
// form keeps the Eq. 4 coefficient and its tangent per CN-list entry, the mixed
// form stores nothing per pair.
#include "d3gb_pair.cuh"

namespace d3gb {

namespace {

struct Dual {
    double v, t;
};
__device__ __forceinline__ Dual dd(double v, double t = 0.0) { return Dual{v, t}; }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual{a.v - b.v, a.t - b.t}; }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return Dual{a.v * b.v, a.v * b.t + a.t * b.v}; }
__device__ __forceinline__ Dual operator*(double s, Dual a) { return Dual{s * a.v, s * a.t}; }
__device__ __forceinline__ Dual operator+(Dual a, double s) { return Dual{a.v + s, a.t}; }
__device__ __forceinline__ Dual& operator+=(Dual& a, Dual b) {
    a.v += b.v;
    a.t += b.t;
    return a;
}
__device__ __forceinline__ Dual inv(Dual a) {
    const double r = 1.0 / a.v;
    return Dual{r, -a.t * r * r};
}
__device__ __forceinline__ Dual dexp(Dual a) {
    const double e = exp(a.v);
    return Dual{e, a.t * e};
}
// per-atom dual arrays carved from one scratch block
struct BW {
    Dual* n;      // [Nr]
    Dual* W;      // [Nr][R]
    Dual* dW;     // [Nr][R]
    Dual* v;      // [Nr][T][R]
    Dual* dEdn;   // [Nr]
    Dual* F;      // [Nr][3]
    Dual* th;     // [Nr][4] dE_i/d(s6, s8, a1, a2), half pair sums
    dbl4* xd;     // [Nr + ghost_cap] tangent positions (bohr)
    double2* cc;  // FP64 form: per CN-list entry, f'(r)/r and its tangent (0 outside R_cn)
    double* sth;  // [B][8] per-structure dE/dtheta (value, tangent)
    // mixed form of the dispersion pass
    float* vf;    // [Nr][T][2 * RP]: R values of v padded to RP, then R tangents padded to RP
    float4* xdf;  // [Nr + ghost_cap] tangent positions as FP32
    float2* dEdnf;  // [Nr] dE/dn (value, tangent) as FP32 for the chain pass
    int RP;
};

// (s on a 32-byte boundary, as the 32-byte records at its start need)
__host__ __device__ inline BW carve(double* s, int64_t Nr, int64_t Ng, int64_t list_cn, int T, int R, int B) {
    BW b;
    b.xd = reinterpret_cast<dbl4*>(s);
    s += 4 * (Nr + Ng);
    b.cc = reinterpret_cast<double2*>(s);
    s += 2 * list_cn;
    Dual* d = reinterpret_cast<Dual*>(s);
    b.n = d;
    d += Nr;
    b.W = d;
    d += Nr * R;
    b.dW = d;
    d += Nr * R;
    b.v = d;
    d += Nr * T * R;
    b.dEdn = d;
    d += Nr;
    b.F = d;
    d += 3 * Nr;
    b.th = d;
    d += 4 * Nr;
    double* x = reinterpret_cast<double*>(d);
    b.sth = x;
    x += 8 * (int64_t)B;
    b.RP = R <= 4 ? 4 : 8;
    x += (4 - ((reinterpret_cast<uintptr_t>(x) / sizeof(double)) & 3)) & 3;  // 32-byte alignment
    b.vf = reinterpret_cast<float*>(x);
    x += Nr * T * b.RP;
    b.xdf = reinterpret_cast<float4*>(x);
    x += 2 * (Nr + Ng);
    b.dEdnf = reinterpret_cast<float2*>(x);
    return b;
}

struct BConsts {
    double rc_disp2, rc_cn2, k1, k3, s6, s8;
    int T, R;
};

// tangent positions: x(t) = x + t * gF / bohr for real atoms, images follow their source
// (FP32 for the mixed form, else FP64)
__global__ void kb_xdot(Work w, BW b, const double* __restrict__ gF, int64_t nt, bool mixed) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nt || q >= w.Nr + min(*w.ghost_count, w.ghost_cap)) return;
    const int src = rec_tsrc(w, q) >> 4;
    const int i = w.perm[src];
    double t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t[a] = gF[3 * (int64_t)i + a] * (1.0 / kBohrA);
    }
    if (mixed) b.xdf[q] = make_float4((float)t[0], (float)t[1], (float)t[2], 0.0f);
    else b.xd[q] = dbl4_make(t[0], t[1], t[2], 0.0);
}

// FP64 form of the CN, dispersion and chain passes.  The FP64 pipe bounds them (one warp
// instruction takes about 80 issue slots), so the tangents come from closed forms: every
// pair function depends on r^2 alone, its tangent is its derivative times
// d(r^2)/dt = 2 d.u (u the tangent of the pair vector d), and where values and tangents
// only meet in one result they are combined before they are summed (dual-number
// arithmetic took 372 instructions per ordered pair in the dispersion pass, this 102:
// 4.53 ms and 1.34 ms on 6.2 M ordered pairs; CN pass 288 us and 93, chain 415 and 51).
// kLanes lanes share an atom's list, entry k going to lane k mod kLanes, and add up their
// sums in a fixed order: with one thread per atom a batch of some 20,000 atoms leaves
// the chip two thirds idle.
constexpr int kLanes = 8;

__device__ __forceinline__ double lanes_sum(double x) {
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// n and dn/dt = sum_q f'(r)/r (d.u); per entry the coefficient c = f'(r)/r and its tangent
// c (d.u) (-k1 rc (1 - 2 f)/r - 3)/r^2.  (The threads past the last atom repeat it.)
__global__ void __launch_bounds__(128) kb_cn(Work w, BW b, BConsts c, const double* __restrict__ k1rc,
                                            const double* __restrict__ exptab64) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = (int)(id % kLanes);
    const bool live = id / kLanes < w.Nr;
    const int64_t p = live ? id / kLanes : w.Nr - 1;
    const StructGeo& G = w.geo[w.sid[p]];
    const int64_t base = list_row(G.list_base_cn, p - G.atom_base, G.cap_cn);
    const int cnt = w.cnt_cn[p];
    const dbl4 x = w.pos64[p], ux = b.xd[p];
    const double* krow = k1rc + (rec_tsrc(w, p) & 15) * c.T;
    double n = 0.0, nt = 0.0;
    for (int k = lane; k < cnt; k += kLanes) {
        const int q = __ldg(w.nbr_cn + base + list_off(k));
        const dbl4 y = w.pos64[q];
        const double dx = y.x - x.x, dy = y.y - x.y, dz = y.z - x.z;
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        double2 o = make_double2(0.0, 0.0);
        if (r2 < c.rc_cn2) {
            const dbl4 uq = b.xd[q];
            const double du = fma(dx, uq.x - ux.x, fma(dy, uq.y - ux.y, dz * (uq.z - ux.z)));
            const double rinv = __double2hiint(r2) > 0x00100000 ? rsqrt64(r2) : 1.0 / sqrt(r2);
            const double a = krow[rec_tsrc(w, q) & 15];
            const double t = exp64_int(fix53(fma(-a, rinv, c.k1)), exptab64);
            const double f = rcp64(1.0 + t);
            const double ri2 = rinv * rinv, ar = a * rinv;
            o.x = -(ar * ri2) * (t * f * f);
            const double s = o.x * du;
            o.y = s * (ri2 * fma(fma(2.0, f, -1.0), ar, -3.0));
            n += f;
            nt += s;
        }
        if (live) b.cc[base + list_off(k)] = o;
    }
    n = lanes_sum(n);
    nt = lanes_sum(nt);
    if (live && lane == 0) b.n[p] = Dual{n, nt};
}

template <int R>
__global__ void kb_weights(Work w, BW b, BConsts c, const double* __restrict__ cnref, const int* __restrict__ nref,
                           const double* __restrict__ c6) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    const int t = rec_tsrc(w, p) & 15;
    const Dual n = b.n[p];
    const int nr = nref[t];
    Dual z[R], ex[R], L[R];
    double emax = -1e300;
#pragma unroll
    for (int a = 0; a < R; ++a) {
        z[a] = n + (-cnref[t * R + a]);
        ex[a] = -c.k3 * (z[a] * z[a]);
        if (a < nr && ex[a].v > emax) emax = ex[a].v;
    }
    Dual sum = dd(0.0);
#pragma unroll
    for (int a = 0; a < R; ++a) {
        L[a] = a < nr ? dexp(ex[a] + (-emax)) : dd(0.0);
        sum += L[a];
    }
    const Dual is = inv(sum);
    Dual gbar = dd(0.0);
#pragma unroll
    for (int a = 0; a < R; ++a) {
        L[a] = L[a] * is;
        gbar += L[a] * (-2.0 * c.k3 * z[a]);
    }
#pragma unroll
    for (int a = 0; a < R; ++a) {
        b.W[p * R + a] = L[a];
        b.dW[p * R + a] = L[a] * ((-2.0 * c.k3 * z[a]) - gbar);
    }
    for (int u = 0; u < c.T; ++u) {
        const double* cu = c6 + ((size_t)(u * c.T + t) * R) * R;
#pragma unroll
        for (int a = 0; a < R; ++a) {
            Dual s = dd(0.0);
#pragma unroll
            for (int bb = 0; bb < R; ++bb) s += cu[a * R + bb] * L[bb];
            b.v[(p * c.T + u) * R + a] = s;
        }
    }
}

// Dispersion pass.  With i6 = 1/(r^6 + R^6), i8 = 1/(r^8 + R^8) and x = r^2 (derivatives by x):
//   g    = s6 i6 + s8 R0^2 i8                       g'   = -fc0/2
//   fc0  = 6 s6 r^4 i6^2 + 8 s8 R0^2 r^6 i8^2       fc0' = 12 s6 r^2 i6^2 (3 R^6 i6 - 2)
//                                                          + 24 s8 R0^2 r^4 i8^2 ((8 R^8 i8 - 5)/3)
//   i6'  = -3 r^4 i6^2                              i8'  = -4 r^6 i8^2
//   h    = 6 s6 R^5 i6^2 + 8 s8 R0^2 R^7 i8^2       (-dg/dR), h' = 12 s6 R^5 i6 i6' + 16 s8 R0^2 R^7 i8 i8'
// An ordered pair adds -g dC6/dn to dE/dn, fc0 C6 d to the force and C6 (-i6, -R0^2 i8, R0 h, h)
// to dE/d(s6, s8, a1, a2) (halved at the end).  Of the last two only gE times the value minus the
// tangent is needed: the force's negative (F slot of b, its v part) and th's t part.
// pairb[ti*T + tj] = (R0, R, R0^2, 0) in bohr
constexpr int kBTab = 12;
template <int R>
__global__ void __launch_bounds__(128) kb_disp(Work w, BW b, BConsts c, const dbl4* __restrict__ pairb,
                                              const double* __restrict__ gE) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* tab = reinterpret_cast<double*>(smem_raw);
    for (int k = threadIdx.x; k < c.T * c.T; k += blockDim.x) {
        const dbl4 pb = pairb[k];
        const double Rd = pb.y, R2 = Rd * Rd, R4 = R2 * R2, R6 = R4 * R2, R8 = R4 * R4, y = c.s8 * pb.z;
        double* t = tab + kBTab * k;
        t[0] = R6; t[1] = R8; t[2] = c.s6; t[3] = y;
        t[4] = 6.0 * c.s6; t[5] = 8.0 * y;
        t[6] = 6.0 * c.s6 * R4 * Rd; t[7] = 8.0 * y * R6 * Rd;
        t[8] = 3.0 * R6; t[9] = 8.0 / 3.0 * R8;
        t[10] = pb.x; t[11] = pb.z;
    }
    __syncthreads();
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = (int)(id % kLanes);
    const bool live = id / kLanes < w.Nr;
    const int64_t p = live ? id / kLanes : w.Nr - 1;
    const int ti = rec_tsrc(w, p) & 15;
    const int s = w.sid[p];
    const StructGeo& G = w.geo[s];
    const int* row = w.nbr_disp + list_row(G.list_base_disp, p - G.atom_base, G.cap_disp);
    const int cnt = w.cnt_disp[p];
    const dbl4 x = w.pos64[p], ux = b.xd[p];
    const double ge = gE[s];
    Dual Wi[R], dWi[R];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        Wi[a] = b.W[p * R + a];
        dWi[a] = b.dW[p * R + a];
    }
    const double* trow = tab + kBTab * ti * c.T;
    const Dual* vb = b.v + (int64_t)ti * R;
    const int vstride = c.T * R;
    double dn = 0, dnt = 0, Gx = 0, Gy = 0, Gz = 0, t6 = 0, t6t = 0, t8 = 0, tR = 0, ta = 0;
    for (int k = lane; k < cnt; k += kLanes) {
        const int q = __ldg(row + list_off(k));
        const dbl4 y = w.pos64[q];
        const double dx = y.x - x.x, dy = y.y - x.y, dz = y.z - x.z;
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        if (!(r2 < c.rc_disp2)) continue;
        const int tsq = rec_tsrc(w, q);
        const dbl4 uq = b.xd[q];
        const double vx = uq.x - ux.x, vy = uq.y - ux.y, vz = uq.z - ux.z;
        const double du = fma(dx, vx, fma(dy, vy, dz * vz));  // d(r^2)/dt / 2
        const double* t = trow + kBTab * (tsq & 15);
        const Dual* vq = vb + (int64_t)(tsq >> 4) * vstride;
        double C = 0, Ct = 0, D = 0, Dt = 0;
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const Dual v = vq[a];
            C = fma(Wi[a].v, v.v, C);
            Ct = fma(Wi[a].v, v.t, fma(Wi[a].t, v.v, Ct));
            D = fma(dWi[a].v, v.v, D);
            Dt = fma(dWi[a].v, v.t, fma(dWi[a].t, v.v, Dt));
        }
        const double r4 = r2 * r2, r6 = r4 * r2;
        const double d6 = r6 + t[0], d8 = fma(r4, r4, t[1]);
        const double pinv = rcp64(d6 * d8);
        const double i6 = d8 * pinv, i8 = d6 * pinv;
        const double g = fma(t[3], i8, t[2] * i6);
        const double a6 = r2 * i6, A6 = a6 * a6, e8 = i8 * i8, B8 = r6 * e8;  // r^4 i6^2, r^6 i8^2
        const double fc0 = fma(t[5], B8, t[4] * A6);
        const double P6 = i6 * a6 * fma(t[8], i6, -2.0), P8 = r4 * e8 * fma(t[9], i8, -5.0 / 3.0);
        const double fc1 = fma(3.0 * t[5], P8, 2.0 * t[4] * P6);
        const double h = fma(t[7], e8, t[6] * (i6 * i6));
        const double h1 = fma(4.0 * t[7], i8 * B8, 3.0 * t[6] * (i6 * A6));  // -h'/2
        dn = fma(-g, D, dn);
        dnt = fma(-g, Dt, dnt);
        dnt = fma(fc0 * du, D, dnt);
        // gE (value) - (tangent): Cv of C6, Cd of the 2 d.u that multiplies derivatives
        const double Cv = fma(ge, C, -Ct), Cd = 2.0 * du * C;
        const double fc = C * fc0;
        const double A = -fma(Cv, fc0, -Cd * fc1);  // tangent - gE (value) of the force coefficient
        Gx = fma(A, dx, fma(fc, vx, Gx));
        Gy = fma(A, dy, fma(fc, vy, Gy));
        Gz = fma(A, dz, fma(fc, vz, Gz));
        t6 = fma(i6, Cv, t6);
        t6t = fma(A6, Cd, t6t);
        t8 = fma(t[11], fma(i8, Cv, 4.0 * B8 * Cd), t8);
        const double z = fma(h, Cv, 2.0 * h1 * Cd);
        ta = fma(t[10], z, ta);
        tR += z;
    }
    dn = lanes_sum(dn); dnt = lanes_sum(dnt);
    Gx = lanes_sum(Gx); Gy = lanes_sum(Gy); Gz = lanes_sum(Gz);
    t6 = lanes_sum(fma(3.0, t6t, t6)); t8 = lanes_sum(t8); ta = lanes_sum(ta); tR = lanes_sum(tR);
    if (!live || lane != 0) return;
    b.dEdn[p] = Dual{dn, dnt};
    b.F[3 * p].v = Gx;
    b.F[3 * p + 1].v = Gy;
    b.F[3 * p + 2].v = Gz;
    b.th[4 * p].t = 0.5 * t6;
    b.th[4 * p + 1].t = 0.5 * t8;
    b.th[4 * p + 2].t = -0.5 * ta;
    b.th[4 * p + 3].t = -0.5 * tR;
}

// ---- mixed form of the dispersion pass of the backward: the same dual-number
// evaluation with FP32 pair arithmetic on the split positions (hi + lo) and
// FP32 tangents, FP32 partial sums promoted to FP64 every kChunk pairs and a
// compensated value part of dE/dn (it scales the chain-rule forces).
struct DF {
    float v, t;
};
__device__ __forceinline__ DF operator+(DF a, DF b) { return DF{a.v + b.v, a.t + b.t}; }
__device__ __forceinline__ DF operator*(DF a, DF b) { return DF{a.v * b.v, fmaf(a.v, b.t, a.t * b.v)}; }
__device__ __forceinline__ DF operator*(float s, DF a) { return DF{s * a.v, s * a.t}; }
__device__ __forceinline__ DF finv(DF a) {
    const float r = 1.0f / a.v;
    return DF{r, -a.t * r * r};
}
__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
// compensated float-pair running sum (value h + l)
struct FF {
    float h = 0.f, l = 0.f;
    __device__ void add(float x) { acc_add(h, l, x); }
    __device__ double value() const { return (double)h + (double)l; }
};

template <int R>
__global__ void __launch_bounds__(128) kb_disp_mixed(Work w, BW b, BConsts c, const dbl4* __restrict__ pairb) {
    // per element pair: R^6, R^8, s8 R0^2, R0, 6 s6 R^4 R, 8 s8 R0^2 R^6 R, R0^2
    __shared__ float tab[kMaxTypes * kMaxTypes][8];
    for (int k = threadIdx.x; k < c.T * c.T; k += blockDim.x) {
        const dbl4 pb = pairb[k];
        const double Rd = pb.y, R2 = Rd * Rd, R4 = R2 * R2, R6 = R4 * R2, R8 = R4 * R4;
        tab[k][0] = (float)R6;
        tab[k][1] = (float)R8;
        tab[k][2] = (float)(c.s8 * pb.z);
        tab[k][3] = (float)pb.x;
        tab[k][4] = (float)(6.0 * c.s6 * R4 * Rd);
        tab[k][5] = (float)(8.0 * c.s8 * pb.z * R6 * Rd);
        tab[k][6] = (float)pb.z;
        tab[k][7] = 0.0f;
    }
    __syncthreads();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    float4 hp, lp;
    rec_load(w, p, hp, lp);
    const int ti = __float_as_int(hp.w) & 15;
    const float4 tp = b.xdf[p];
    DF Wi[R], dWi[R];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        const Dual x = b.W[p * R + a], y = b.dW[p * R + a];
        Wi[a] = DF{(float)x.v, (float)x.t};
        dWi[a] = DF{(float)y.v, (float)y.t};
    }
    const StructGeo& G = w.geo[w.sid[p]];
    const ListView LV{w.nbr_disp + list_row(G.list_base_disp, p - G.atom_base, G.cap_disp)};
    const int cnt = w.cnt_disp[p];
    const float rc2f = (float)c.rc_disp2, s6 = (float)c.s6;
    constexpr int RP = R <= 4 ? 4 : 8;  // b.RP
    const int stride = c.T * 2 * RP;
    float dnh = 0.0f, dnl = 0.0f;
    // running sums as compensated float pairs (FP64 runs at 1/64 of the FP32 rate)
    FF dnt, Fv[3], Ft[3], thv[4], tht[4];
    for (int k0 = 0; k0 < cnt; k0 += kChunk) {
        const int k1e = min(cnt, k0 + kChunk);
        float dt = 0.0f, fv[3] = {0, 0, 0}, ft[3] = {0, 0, 0}, hv[4] = {0, 0, 0, 0}, ht[4] = {0, 0, 0, 0};
        // an entry's position record and tangent, then its v row for type t_i (R values, then R
        // tangents, each padded to RP: vector loads); two entries' loads are issued before their
        // arithmetic (the pass waits for them: 27% of the issue slots were used with one; 57.4 M
        // ordered pairs 1.61 ms and 1.40; the next two's records ahead as well: slower, 168 registers)
        struct Entry {
            float4 h, l, u;
            float vv[R], vt[R];
            int q;
        };
        auto fetch = [&](int q, Entry& x) {
            x.q = q;
            rec_load(w, q, x.h, x.l);
            x.u = __ldg(b.xdf + q);
        };
        auto fetch_row = [&](Entry& x) {
            const float* vq = b.vf + (int64_t)(__float_as_int(x.h.w) >> 4) * stride + ti * 2 * RP;
            load_vec<R>(vq, x.vv);
            load_vec<R>(vq + RP, x.vt);
        };
        auto add = [&](const Entry& x) {
            const float4 hq = x.h, lq = x.l;
            const int q = x.q;
            const float dx = (hq.x - hp.x) + (lq.x - lp.x), dy = (hq.y - hp.y) + (lq.y - lp.y),
                        dz = (hq.z - hp.z) + (lq.z - lp.z);
            const float r2v = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            bool in;
            if (fabsf(r2v - rc2f) > 4e-6f * rc2f) {
                in = r2v < rc2f;
            } else {  // within the FP32 error band of the cutoff: decide in FP64
                const dbl4 x = w.pos64[p], y = w.pos64[q];
                const double ex = y.x - x.x, ey = y.y - x.y, ez = y.z - x.z;
                in = ex * ex + ey * ey + ez * ez < c.rc_disp2;
            }
            if (!in) return;
            const int tsq = __float_as_int(hq.w);
            const float4 tq = x.u;
            const float ux = tq.x - tp.x, uy = tq.y - tp.y, uz = tq.z - tp.z;
            const DF r2 = DF{r2v, 2.0f * fmaf(dx, ux, fmaf(dy, uy, dz * uz))};
            const float* tb = tab[ti * c.T + (tsq & 15)];
            DF C6 = DF{0.0f, 0.0f}, dC6 = DF{0.0f, 0.0f};
#pragma unroll
            for (int a = 0; a < R; ++a) {
                const DF v = DF{x.vv[a], x.vt[a]};
                C6 = C6 + Wi[a] * v;
                dC6 = dC6 + dWi[a] * v;
            }
            const DF r4 = r2 * r2, r6 = r4 * r2, r8 = r4 * r4;
            const DF i6 = finv(DF{r6.v + tb[0], r6.t}), i8 = finv(DF{r8.v + tb[1], r8.t});
            const DF t6 = s6 * i6, t8 = tb[2] * i8;
            const DF g = t6 + t8;
            const DF gd = g * dC6;
            float s, e;
            two_sum_f(dnh, -gd.v, s, e);
            dnh = s;
            dnl += e;
            dt -= gd.t;
            const DF fc = C6 * (6.0f * (r4 * (t6 * i6)) + 8.0f * (r6 * (t8 * i8)));
            fv[0] = fmaf(fc.v, dx, fv[0]); fv[1] = fmaf(fc.v, dy, fv[1]); fv[2] = fmaf(fc.v, dz, fv[2]);
            ft[0] += fmaf(fc.t, dx, fc.v * ux); ft[1] += fmaf(fc.t, dy, fc.v * uy); ft[2] += fmaf(fc.t, dz, fc.v * uz);
            // derivatives of this ordered instance's energy -C6 g in s6, s8, a1, a2 (halved at the end)
            const DF e6 = C6 * i6, e8 = C6 * i8;
            hv[0] -= e6.v; ht[0] -= e6.t;
            hv[1] = fmaf(-tb[6], e8.v, hv[1]); ht[1] = fmaf(-tb[6], e8.t, ht[1]);
            const DF dR = C6 * (tb[4] * (i6 * i6) + tb[5] * (i8 * i8));
            hv[2] = fmaf(tb[3], dR.v, hv[2]); ht[2] = fmaf(tb[3], dR.t, ht[2]);
            hv[3] += dR.v; ht[3] += dR.t;
        };
        auto add_two = [&](int qa, int qb, bool two) {
            Entry x, y;
            fetch(qa, x);
            fetch(two ? qb : (int)p, y);
            fetch_row(x);
            fetch_row(y);
            add(x);
            if (two) add(y);
        };
        for (int k = k0; k < k1e; k += 4) {
            const int4 q4 = __ldg(reinterpret_cast<const int4*>(LV.p + list_off(k)));
            add_two(q4.x, q4.y, k + 1 < k1e);
            if (k + 2 < k1e) add_two(q4.z, q4.w, k + 3 < k1e);
        }
        dnt.add(dt);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            Fv[a].add(fv[a]);
            Ft[a].add(ft[a]);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            thv[m].add(hv[m]);
            tht[m].add(ht[m]);
        }
    }
    b.dEdn[p] = Dual{(double)dnh + (double)dnl, dnt.value()};
    b.dEdnf[p] = make_float2(dnh + dnl, dnt.h + dnt.l);
#pragma unroll
    for (int a = 0; a < 3; ++a) b.F[3 * p + a] = Dual{Fv[a].value(), Ft[a].value()};
#pragma unroll
    for (int m = 0; m < 4; ++m) b.th[4 * p + m] = Dual{0.5 * thv[m].value(), 0.5 * tht[m].value()};
}

// Chain rule: dLdx = -gE F + dF/dt, both from the stored coefficients and tangents.
__global__ void __launch_bounds__(128) kb_chain(Work w, BW b, BConsts c, const double* __restrict__ gE,
                                               double* __restrict__ dLdx) {
    const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = (int)(id % kLanes);
    const bool live = id / kLanes < w.Nr;
    const int64_t p = live ? id / kLanes : w.Nr - 1;
    const int s = w.sid[p];
    const StructGeo& G = w.geo[s];
    const int64_t base = list_row(G.list_base_cn, p - G.atom_base, G.cap_cn);
    const int cnt = w.cnt_cn[p];
    const dbl4 x = w.pos64[p], ux = b.xd[p];
    const Dual dni = b.dEdn[p];
    const double ge = gE[s];
    double Gx = 0, Gy = 0, Gz = 0;
    for (int k = lane; k < cnt; k += kLanes) {
        const double2 cc = b.cc[base + list_off(k)];
        if (__double_as_longlong(cc.x) == 0) continue;  // outside R_cn
        const int q = __ldg(w.nbr_cn + base + list_off(k));
        const dbl4 y = w.pos64[q], uq = b.xd[q];
        const Dual dq = b.dEdn[rec_tsrc(w, q) >> 4];
        const double S = dni.v + dq.v, cv = S * cc.x;
        const double A = fma(dni.t + dq.t, cc.x, fma(S, cc.y, -ge * cv));
        Gx = fma(A, y.x - x.x, fma(cv, uq.x - ux.x, Gx));
        Gy = fma(A, y.y - x.y, fma(cv, uq.y - ux.y, Gy));
        Gz = fma(A, y.z - x.z, fma(cv, uq.z - ux.z, Gz));
    }
    Gx = lanes_sum(Gx); Gy = lanes_sum(Gy); Gz = lanes_sum(Gz);
    if (!live || lane != 0) return;
    const double u = kHartreeEV / kBohrA;
    double* o = dLdx + 3 * (int64_t)w.perm[p];
    o[0] = (b.F[3 * p].v + Gx) * u;
    o[1] = (b.F[3 * p + 1].v + Gy) * u;
    o[2] = (b.F[3 * p + 2].v + Gz) * u;
}

// ---- mixed form of the CN, weight and chain passes of the backward
// n (value) as in the forward's CN pass: double-single Eq. 4 term, integer
// count plus compensated complements; dn/dt = sum_q f'(r)/r (d . u), FP32
// (compensated), u the tangent of d.
__global__ void __launch_bounds__(128) kb_cn_mixed(Work w, BW b, Consts c, const float4* __restrict__ rcpair,
                                                   const float2* __restrict__ exptab) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    const Site<true> S(w, p);
    const StructGeo& G = w.geo[w.sid[p]];
    const ListView LV{w.nbr_cn + list_row(G.list_base_cn, p - G.atom_base, G.cap_cn)};
    const int cnt = w.cnt_cn[p];
    const float4* rrow = rcpair + (S.tsrc() & 15) * c.T;
    const float k1 = c.k1f, rc2 = c.rc_cn2f;
    const float4 tp = b.xdf[p];
    float nh = 0.f, nl = 0.f, th = 0.f, tl = 0.f;
    int nint = 0;
    auto add = [&](int q, const float4* rec, const float4& uq) {
        float D[3], r2, ah, al, rch;
        int tq;
        if (!cn_pair_precise(S, q, rrow, k1, rc2, c.rc_cn2, D, r2, ah, al, rch, tq, nullptr, nullptr, nullptr, rec))
            return;
        const CnDS z = cn_ds(ah, al, exptab);
        if (z.th < 1.0f) {
            ++nint;
            acc_add(nh, nl, -z.ch);
            nl -= z.cl;
        } else {
            acc_add(nh, nl, z.fh);
            nl += z.fl;
        }
        const float du = fmaf(D[0], uq.x - tp.x, fmaf(D[1], uq.y - tp.y, D[2] * (uq.z - tp.z)));
        const float ri = rsqrt_nr(r2);
        acc_add(th, tl, -k1 * rch * z.fh * z.ch * (ri * ri * ri) * du);
    };
    for (int k = 0; k < cnt; k += 4) {  // four entries' loads before their arithmetic
        const int4 q4 = __ldg(reinterpret_cast<const int4*>(LV.p + list_off(k)));
        const int q[4] = {q4.x, k + 1 < cnt ? q4.y : (int)p, k + 2 < cnt ? q4.z : (int)p, k + 3 < cnt ? q4.w : (int)p};
        float4 rec[4][2], u[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            rec_load(w, q[e], rec[e][0], rec[e][1]);
            u[e] = __ldg(b.xdf + q[e]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (k + e < cnt) add(q[e], rec[e], u[e]);
    }
    b.n[p] = Dual{(double)nint + (double)nh + (double)nl, (double)th + (double)tl};
}

// Weights (Eq. 3) as dual numbers: values with float-float exponents as in the
// forward, tangents in FP32; dW/dn = -2 k3 W_a sum_b W_b (nref_b - nref_a) from
// the table of reference differences (no cancellation against n).  The shift
// by the largest exponent is a constant: it cancels in the normalisation.
template <int R>
__global__ void __launch_bounds__(128) kb_weights_mixed(Work w, BW b, Consts c, const float2* __restrict__ cnref2,
                                                        const float* __restrict__ dcr, const int* __restrict__ nref,
                                                        const float* __restrict__ c6) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    const int t = rec_tsrc(w, p) & 15;
    const Dual nd = b.n[p];
    const float Nh = (float)nd.v, Nl = (float)(nd.v - (double)Nh), nt = (float)nd.t;
    const int nr = nref[t];
    float xh[R], xl[R], xt[R];
    float mh = -3.0e38f, ml = 0.0f;
#pragma unroll
    for (int a = 0; a < R; ++a) {
        const float2 cr = cnref2[t * R + a];
        float zh, ze, zl;
        two_sum(Nh, -cr.x, zh, ze);
        two_sum(zh, ze + (Nl - cr.y), zh, zl);
        const float ph = zh * zh, pl = fmaf(zh, zh, -ph) + 2.0f * zh * zl;
        xh[a] = -c.k3h * ph;
        xl[a] = fmaf(-c.k3h, ph, -xh[a]) - c.k3h * pl - c.k3l * ph;
        xt[a] = -2.0f * c.k3f * zh * nt;
        if (a < nr && (xh[a] > mh || (xh[a] == mh && xl[a] > ml))) {
            mh = xh[a];
            ml = xl[a];
        }
    }
    DF L[R];
    DF sum = DF{0.f, 0.f};
#pragma unroll
    for (int a = 0; a < R; ++a) {
        L[a] = DF{0.f, 0.f};
        if (a < nr) {
            float yh, ye, yl;
            two_sum(xh[a], -mh, yh, ye);
            two_sum(yh, ye + (xl[a] - ml), yh, yl);
            const float e = expf(yh) * (1.0f + yl);
            L[a] = DF{e, e * xt[a]};
        }
        sum = sum + L[a];
    }
    const DF is = finv(sum);
#pragma unroll
    for (int a = 0; a < R; ++a) L[a] = L[a] * is;
#pragma unroll
    for (int a = 0; a < R; ++a) {
        DF sa = DF{0.f, 0.f};
        const float* dr = dcr + (t * R + a) * R;
#pragma unroll
        for (int bb = 0; bb < R; ++bb) sa = sa + dr[bb] * L[bb];
        const DF dW = (-2.0f * c.k3f) * (L[a] * sa);
        b.W[p * R + a] = Dual{(double)L[a].v, (double)L[a].t};
        b.dW[p * R + a] = Dual{(double)dW.v, (double)dW.t};
    }
    // v rows (values then tangents, each padded to RP = 4 or 8) as whole 16-byte stores
    constexpr int RP = R <= 4 ? 4 : 8;
    for (int u = 0; u < c.T; ++u) {
        const float* cu = c6 + ((size_t)(u * c.T + t) * R) * R;  // C6ref[u][t][a][b]
        float vv[RP], vt[RP];
#pragma unroll
        for (int a = 0; a < RP; ++a) {
            DF sv = DF{0.f, 0.f};
            if (a < R) {
#pragma unroll
                for (int bb = 0; bb < R; ++bb) sv = sv + cu[a * R + bb] * L[bb];
            }
            vv[a] = sv.v;
            vt[a] = sv.t;
        }
        float4* dst = reinterpret_cast<float4*>(b.vf + (p * c.T + u) * 2 * RP);
#pragma unroll
        for (int k = 0; k < RP / 4; ++k) {
            dst[k] = make_float4(vv[4 * k], vv[4 * k + 1], vv[4 * k + 2], vv[4 * k + 3]);
            dst[RP / 4 + k] = make_float4(vt[4 * k], vt[4 * k + 1], vt[4 * k + 2], vt[4 * k + 3]);
        }
    }
}

// Chain rule as dual numbers: the value of the coefficient f'(r)/r as in the
// forward's chain pass (double-single, rounded once), its tangent
// d(f'/r)/dt = -k1 rc [(1 - 2f) f' / r^3 - 3 f (1 - f) / r^4] (d . u) / r in FP32.
__global__ void __launch_bounds__(128) kb_chain_mixed(Work w, BW b, Consts c, const float4* __restrict__ rcpair,
                                                      const float2* __restrict__ exptab,
                                                      const double* __restrict__ gE, double* __restrict__ dLdx) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    const Site<true> S(w, p);
    const int s = w.sid[p];
    const StructGeo& G = w.geo[s];
    const ListView LV{w.nbr_cn + list_row(G.list_base_cn, p - G.atom_base, G.cap_cn)};
    const int cnt = w.cnt_cn[p];
    const float4* rrow = rcpair + (S.tsrc() & 15) * c.T;
    const float k1 = c.k1f, rc2 = c.rc_cn2f;
    const float2 dnd = b.dEdnf[p];
    const float dni = dnd.x, dnit = dnd.y;
    const float4 tp = b.xdf[p];
    float fv[3] = {0.f, 0.f, 0.f}, ft[3] = {0.f, 0.f, 0.f};
    auto add = [&](int q, const float4* rec, const float4& uq, const float2& dqd) {
        float D[3], r2, ah, al, rch, rcl, r2l;
        int tq;
        if (!cn_pair_precise(S, q, rrow, k1, rc2, c.rc_cn2, D, r2, ah, al, rch, tq, &rcl, &r2l, nullptr, rec)) return;
        const CnDS z = cn_ds(ah, al, exptab);
        const float g = chain_coef(z, r2, r2l, rch, rcl, k1);
        const float dnq = dqd.x, dnqt = dqd.y;
        const float u[3] = {uq.x - tp.x, uq.y - tp.y, uq.z - tp.z};
        const float du = fmaf(D[0], u[0], fmaf(D[1], u[1], D[2] * u[2]));
        const float ri = rsqrt_nr(r2), ri2 = ri * ri;
        const float f = z.fh, omf = z.ch;  // f and 1 - f
        const float fp = -k1 * rch * f * omf * ri2;  // f'(r)
        const float dgdr = -k1 * rch * ((1.0f - 2.0f * f) * fp * ri2 * ri - 3.0f * f * omf * ri2 * ri2);
        const float gt = dgdr * du * ri;
        const float cv = (dni + dnq) * g;
        const float ct = fmaf(dnit + dnqt, g, (dni + dnq) * gt);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            fv[a] = fmaf(cv, D[a], fv[a]);
            ft[a] = fmaf(ct, D[a], fmaf(cv, u[a], ft[a]));
        }
    };
    for (int k = 0; k < cnt; k += 4) {  // four entries' loads before their arithmetic
        const int4 q4 = __ldg(reinterpret_cast<const int4*>(LV.p + list_off(k)));
        const int q[4] = {q4.x, k + 1 < cnt ? q4.y : (int)p, k + 2 < cnt ? q4.z : (int)p, k + 3 < cnt ? q4.w : (int)p};
        float4 rec[4][2], uu[4];
        float2 dq[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            rec_load(w, q[e], rec[e][0], rec[e][1]);
            uu[e] = __ldg(b.xdf + q[e]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) dq[e] = b.dEdnf[__float_as_int(rec[e][0].w) >> 4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (k + e < cnt) add(q[e], rec[e], uu[e], dq[e]);
    }
    if (dLdx) {
        const double uc = kHartreeEV / kBohrA;
        const double ge = gE[s];
        const int i = w.perm[p];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const Dual Fd = b.F[3 * p + a];
            dLdx[3 * (int64_t)i + a] = (-ge * (Fd.v + (double)fv[a]) + (Fd.t + (double)ft[a])) * uc;
        }
    }
}

// per-structure sums of dE/dtheta (value and tangent; in the FP64 form the values are in the tangents), fixed order
__global__ void __launch_bounds__(256) kb_struct_sum(Work w, BW b, bool values) {
    const int s = blockIdx.x;
    const StructGeo& G = w.geo[s];
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t k = threadIdx.x; k < G.natoms; k += blockDim.x) {
        const int64_t p = G.atom_base + k;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (values) acc[m] += b.th[4 * p + m].v;
            acc[4 + m] += b.th[4 * p + m].t;
        }
    }
    __shared__ double red[8][256];
#pragma unroll
    for (int m = 0; m < 8; ++m) red[m][threadIdx.x] = acc[m];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
#pragma unroll
            for (int m = 0; m < 8; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 8) b.sth[8 * s + threadIdx.x] = red[threadIdx.x][0];
}

// dL/dtheta = sum_s gE_s dE_s/dtheta - d/dtheta(dE/dt), in eV per unit parameter
__global__ void __launch_bounds__(256) kb_param_grad(BW b, int B, const double* __restrict__ gE, double* __restrict__ out) {
    double acc[4] = {0, 0, 0, 0};
    for (int s = threadIdx.x; s < B; s += blockDim.x) {
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] += gE[s] * b.sth[8 * s + m] - b.sth[8 * s + 4 + m];
    }
    __shared__ double red[4][256];
#pragma unroll
    for (int m = 0; m < 4; ++m) red[m][threadIdx.x] = acc[m];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
#pragma unroll
            for (int m = 0; m < 4; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 4) out[threadIdx.x] = red[threadIdx.x][0] * kHartreeEV;
}

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <int R>
cudaError_t backward_impl(const Work& w, const Consts& cc, const double* c6d, const dbl4* pairb, const double* cnref,
                          const int* nref, const Tabs& tbm, const double* gE, const double* gF, double* dLdp,
                          double* dLdx, double* scratch, int64_t list_cn, int B, bool mixed, cudaStream_t st) {
    BW b = carve(scratch, w.Nr, w.ghost_cap, mixed ? 0 : list_cn, w.T, R, B);
    BConsts c{cc.rc_disp2, cc.rc_cn2, cc.k1, cc.k3, cc.s6, cc.s8, cc.T, R};
    const int TB = 128;
    if (w.Nr > 0) {
        // tangent positions for real atoms and every image actually built
        kb_xdot<<<nblk(w.Nr + w.ghost_cap, TB), TB, 0, st>>>(w, b, gF, w.Nr + w.ghost_cap, mixed);
        if (mixed) {
            kb_cn_mixed<<<nblk(w.Nr, TB), TB, 0, st>>>(w, b, cc, tbm.rcpair, tbm.exptab);
            kb_weights_mixed<R><<<nblk(w.Nr, TB), TB, 0, st>>>(w, b, cc, tbm.cnref2, tbm.dcr, tbm.nref,
                                                                (const float*)tbm.c6);
            kb_disp_mixed<R><<<nblk(w.Nr, TB), TB, 0, st>>>(w, b, c, pairb);
            kb_chain_mixed<<<nblk(w.Nr, TB), TB, 0, st>>>(w, b, cc, tbm.rcpair, tbm.exptab, gE, dLdx);
        } else {
            const unsigned nl = nblk(w.Nr * kLanes, TB);
            kb_cn<<<nl, TB, 0, st>>>(w, b, c, tbm.k1rc, tbm.exptab64);
            kb_weights<R><<<nblk(w.Nr, TB), TB, 0, st>>>(w, b, c, cnref, nref, c6d);
            kb_disp<R><<<nl, TB, (size_t)c.T * c.T * kBTab * sizeof(double), st>>>(w, b, c, pairb, gE);
            if (dLdx) kb_chain<<<nl, TB, 0, st>>>(w, b, c, gE, dLdx);
        }
    }
    kb_struct_sum<<<B, 256, 0, st>>>(w, b, mixed);
    if (dLdp) kb_param_grad<<<1, 256, 0, st>>>(b, B, gE, dLdp);
    return cudaGetLastError();
}

}  // namespace

int64_t backward_scratch_doubles(const Work& w, int B, int64_t list_cn, bool mixed) {
    const int64_t Nr = w.Nr, Ng = w.ghost_cap;
    const int64_t duals = Nr * (1 + 2 * (int64_t)w.R + (int64_t)w.T * w.R + 1 + 3 + 4);
    const int64_t rp = w.R <= 4 ? 4 : 8;
    // tangent positions, CN coefficients (FP64 form), duals, per-structure sums, FP32 v rows and tangents (+ alignment)
    return 4 * (Nr + Ng) + (mixed ? 0 : 2 * list_cn) + 2 * duals + 8 * (int64_t)B + Nr * (int64_t)w.T * rp +
           2 * (Nr + Ng) + Nr + 64;
}

cudaError_t launch_backward(const Work& w, const Consts& c, const double* c6d, const dbl4* pairb,
                            const double* cnref, const int* nref, const Tabs& tbm, const double* dLdE,
                            const double* dLdF, double* dLdp, double* dLdx, double* scratch, int64_t list_cn, int B,
                            bool mixed, cudaStream_t st) {
#define D3_BWD(RR) \
    return backward_impl<RR>(w, c, c6d, pairb, cnref, nref, tbm, dLdE, dLdF, dLdp, dLdx, scratch, list_cn, B, mixed, st)
    switch (c.R) {
        case 1: D3_BWD(1);
        case 2: D3_BWD(2);
        case 3: D3_BWD(3);
        case 4: D3_BWD(4);
        case 5: D3_BWD(5);
        case 6: D3_BWD(6);
        default: D3_BWD(7);
    }
#undef D3_BWD
}

}  // namespace d3gb
