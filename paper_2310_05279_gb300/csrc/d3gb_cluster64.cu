// d3gb_cluster64.cu -- dispersion pass of the FP64 form over cluster half lists
// (arXiv 2310.05279, Sec. II A, Eq. 2 with the C6 of Eq. 3).
//
// GB300 runs FP64 at 1/64 of the FP32 rate: one FP64 warp instruction occupies its pipe
// for about 80 issue slots, so the FP64 form is bound by their number and by the lanes
// they leave idle.  The per-atom-list pass (k_disp) takes about 60 of them per ordered
// pair.  This pass
//   * evaluates each unordered pair instance once (the half lists of the mixed form);
//   * keeps the lanes full: lane = i + 8 j keeps one atom i of the warp's cluster and
//     tests its quarter of the list in FP32 (FP64 inside the error band of R_pot);
//     what passes goes into a ring of the lane's own, and the pairs are evaluated when
//     every lane has one;
//   * leaves to the FP64 pipe only the damping function (18 instructions a pair).
//     Pair vectors, r^2, the C6 interpolation and all sums are formed on the integer
//     pipe, with 64-bit mantissas scaled by powers of two: positions (ipos_unit); W, dW and the rows v, dv with one exponent per row (Work::i64,
//     row64); products as the upper half of 64 x 64 bits.  Their relative errors are
//     2^-57 and less (the C6 sums: 2^-61 of the row's largest value), below FP64's 2^-53;
//   * adds everything to per-atom 64-bit fixed-point sums, which associate, so the
//     result does not depend on the order in which warps and splits of a list run.
//
// Units.  Each of an atom's sums (force, dE/dn, energy, virial) has its own unit, a power of
// two that leaves 62 bits to a bound of the sum of its terms' sizes and 56 or 58 to one of its
// largest term (SumBound, formed from the atom's own partners in the CN pass): below what
// FP64 additions round.  A pair adds to i's sums in i's units and to j's in j's, which takes
// nine 64-bit shifts a pair more than units for the whole batch.  (Units for
// the whole batch, from the largest term of any element pair at r = 0, lost all digits at small
// damping radii: at a1 = 0.05, a2 = 0.2 a C-C force at 5 A was off by 5e-5, at a2 = 0.003 by 1.)
// Parameters beyond what the bounds hold in FP32 keep the per-atom-list pass.
//
// Measured on 128 x 1440 atoms (27.9 M pairs): 1.70 ms against 5.62 ms for the per-atom-list
// pass, 16 warps per SM (128 registers; at 142 registers and 12 warps 2.07 ms); 1.61 ms with
// units for the whole batch, 1.78 with 61 bits to every sum and shifts in both directions.
#include "d3gb_pair.cuh"

namespace d3gb {

namespace {

constexpr int kRing = 32;  // ring entries per lane
constexpr int kTest = 8;   // entries tested per lane at a time

// v 2^-s rounded to nearest, |v| < 2^62 (and the result below 2^62)
__device__ __forceinline__ long long shr_rn(long long v, int s) {
    if (s <= 0) return v << min(-s, 63);
    s = min(s, 62);
    return (v + (1LL << (s - 1))) >> s;
}
// the same for s >= 1 and several values
struct Shift {
    int s;
    long long half;
    __device__ __forceinline__ explicit Shift(int s1) : s(min(max(s1, 1), 62)), half(1LL << (s - 1)) {}
    __device__ __forceinline__ long long operator()(long long v) const { return (v + half) >> s; }
};
// a normal double as m 2^(e - 1085), |m| in [2^62, 2^63)
__device__ __forceinline__ long long mantissa(double v, int& e) {
    const long long b = __double_as_longlong(v);
    e = (int)((unsigned long long)b >> 52) & 0x7ff;
    const long long m = ((b & 0xfffffffffffffLL) | 0x10000000000000LL) << 10;
    return b < 0 ? -m : m;
}
__device__ __forceinline__ void red_add64(unsigned long long* a, long long x) {
    atomicAdd(a, (unsigned long long)x);  // result unused: a reduction, no return trip
}

// The units of an atom's sums (Work::ks)
struct Units {
    int kF, kD, kE, kV;
    __device__ __forceinline__ explicit Units(int2 k)
        : kF((int)(short)k.x), kD(k.x >> 16), kE((int)(short)k.y), kV(k.y >> 16) {}
};

// Damping constants of an element pair in shared memory: R^6, R^8, s6, s8 R0^2, 6 s6, 8 s8 R0^2.
constexpr int kDamp = 6;

template <int R, bool SITE>
__global__ void __launch_bounds__(128, 4) k_disp_cl64(Work w, Consts c, const dbl4* __restrict__ pair_tab, int nsplit) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* tab = reinterpret_cast<double*>(smem_raw);
    constexpr int S64 = row64_len(R);
    // the clusters' rows W, dW (loaded again for every pair: they would take 20 registers)
    long long* wsh = reinterpret_cast<long long*>(tab + kDamp * c.T * c.T) + (threadIdx.x >> 5) * (kClusterAtoms * S64);
    int* rings = reinterpret_cast<int*>(reinterpret_cast<long long*>(tab + kDamp * c.T * c.T) + 4 * kClusterAtoms * S64);
    for (int k = threadIdx.x; k < c.T * c.T; k += blockDim.x) {
        const dbl4 t = pair_tab[k];
        double* d = tab + kDamp * k;
        d[0] = t.x; d[1] = t.y; d[2] = t.z; d[3] = t.w; d[4] = 6.0 * t.z; d[5] = 8.0 * t.w;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, il = lane & 7, js = lane >> 3;
    const int64_t I = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (I >= w.ncl) return;  // whole warps
    int* ring = rings + (threadIdx.x >> 5) * (kRing * 32) + lane;  // slot k at ring[32 k]
    const int s = w.clu_sid[I];
    const StructGeo& G = w.geo[s];
    const int64_t p0 = G.atom_base + (I - G.clu_base) * kClusterAtoms;
    const int64_t rem = G.atom_base + G.natoms - p0;
    const int nI = rem < kClusterAtoms ? (int)rem : kClusterAtoms;
    const bool ilive = il < nI;
    const int64_t p = p0 + (ilive ? il : 0);
    const int* row = w.nbr_cl + G.list_base_cl + (I - G.clu_base) * (int64_t)G.cap_cl;
    const int cnt = w.cnt_cl[I];
    const int nblocks = (cnt + 31) >> 5;
    // this warp's share of the blocks of 32 entries (blockIdx.y of nsplit)
    const int bb = (int)((int64_t)nblocks * blockIdx.y / nsplit), be = (int)((int64_t)nblocks * (blockIdx.y + 1) / nsplit);
    if (bb >= be) return;
    const Site<true> S(w, p);
    const int ti = S.tsrc() & 15;
    const int pthr = ilive ? (int)p : 0x7fffffff;  // a pair is used when q > pthr
    const longlong2* xi2 = reinterpret_cast<const longlong2*>(w.ipos + 4 * p);
    const longlong2 xa = xi2[0], xb = xi2[1];
    for (int k = lane; k < nI * S64; k += 32) wsh[k] = w.i64[p0 * S64 + k];
    __syncwarp();
    const long long* wi = wsh + (int)(p - p0) * S64;
    const int eW = (int)wi[2 * R];
    const Units K(w.ks[p]);
    const double* trow = tab + kDamp * ti * c.T;
    const long long* rbase = w.row64 + ti * S64;
    const int rstride = c.T * S64;
    const float rc2 = c.rc_disp2f, band = 4e-6f * c.rc_disp2f;
    long long aF[3] = {0, 0, 0}, aD = 0, aE = 0, aV[6] = {0, 0, 0, 0, 0, 0};
    int head = 0, n = 0;  // the lane's ring: first entry and number of entries
    unsigned npairs = 0;

    auto eval = [&](int q) {
        const longlong2* x2 = reinterpret_cast<const longlong2*>(w.ipos + 4 * (int64_t)q);
        const longlong2 ya = __ldg(x2), yb = __ldg(x2 + 1);
        const int tsq = (int)yb.y;
        const int64_t src = tsq >> 4;
        const longlong2* rp = reinterpret_cast<const longlong2*>(rbase + src * rstride);
        long long rv[2 * R + 2];
#pragma unroll
        for (int a = 0; a < 2 * R + 1; a += 2) {
            const longlong2 t = __ldg(rp + a / 2);
            rv[a] = t.x;
            rv[a + 1] = t.y;
        }
        const int ev = (int)rv[2 * R], ed = (int)(rv[2 * R] >> 32);
        const Units J(__ldg(w.ks + src));
        long long dx = ya.x - xa.x, dy = ya.y - xa.y, dz = yb.x - xb.x;
        unsigned long long mant;
        int sh;
        const double r2 = ipos_r2(dx, dy, dz, (int)wi[2 * R + 1], sh, mant);
        const double* t = trow + kDamp * (tsq & 15);
        // damping: g = -de/dC6 = s6/(r^6 + R^6) + s8 R0^2/(r^8 + R^8), fc0 = (de/dr)/(C6 r)
        const double r4 = r2 * r2, r6 = r4 * r2;
        const double d6 = r6 + t[0], d8 = fma(r4, r4, t[1]);
        const double pinv = rcp64(d6 * d8);
        const double i6 = d8 * pinv, i8 = d6 * pinv;
        const double g = fma(t[3], i8, t[2] * i6);
        const double u6 = r2 * i6;
        const double fc0 = fma(t[5], r6 * (i8 * i8), t[4] * (u6 * u6));
        // C6 and both CN derivatives
        long long C6 = (R + 1) / 2, dCi = 0, dCj = 0;  // (each product is rounded down)
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const long long W = wi[a];
            C6 += __mul64hi(W, rv[a]);            // units 2^(ev - 61)
            dCi += __mul64hi(wi[R + a], rv[a]);   // 2^(eW + ev - 60)
            dCj += __mul64hi(W, rv[R + a]);       // 2^(ed - 61)
        }
        // |C6| is below 2^61 and a rounding error (the weights add up to 1): normalised to [2^61, 2^62)
        const int sc = max(__clzll(C6 ^ (C6 >> 63)) - 2, 0), ec = ev - sc;
        C6 <<= sc;  // units 2^(ec - 61)
        dCj <<= 1;
        int eg, ef;
        const long long mg = mantissa(g, eg), mf = mantissa(fc0, ef);
        // energy and dE/dn
        // (terms of C6 lie in [2^59, 2^62) here, a virial's largest component in [2^57, 2^61): with the
        // bits that the units leave to the bounds, every shift is at least 1)
        const int sE = 1082 - eg - ec + (SITE ? 1 : 0);  // SITE: half of it to each atom
        const long long e = __mul64hi(mg, C6);
        aE += Shift(sE - K.kE)(e);
        aD += shr_rn(__mul64hi(mg, dCi), 1081 - eg - eW - ev - K.kD);
        unsigned long long* aj = w.acc + 16 * src;
        red_add64(aj + 3, shr_rn(__mul64hi(mg, dCj), 1083 - eg - ed - J.kD));
        if (SITE) red_add64(aj + 4, Shift(sE - J.kE)(e));
        // force in units 2^-(sF + u), and i's virial from it in units 2^-(sF + sh - 64 + 2 u), u that of the positions
        const long long fC = __mul64hi(mf, C6) << 2;
        const long long ux = __mul64hi(fC, dx), uy = __mul64hi(fC, dy), uz = __mul64hi(fC, dz);
        const int sF = 1020 + sh - ef - ec;
        const Shift fj(sF - J.kF), fi(sF - K.kF), vi(sF + sh - 64 - K.kV);
        red_add64(aj + 0, -fj(ux));
        red_add64(aj + 1, -fj(uy));
        red_add64(aj + 2, -fj(uz));
        aF[0] += fi(ux); aF[1] += fi(uy); aF[2] += fi(uz);
        aV[0] += vi(__mul64hi(ux, dx));
        aV[1] += vi(__mul64hi(uy, dy));
        aV[2] += vi(__mul64hi(uz, dz));
        aV[3] += vi(__mul64hi(ux, dy));
        aV[4] += vi(__mul64hi(ux, dz));
        aV[5] += vi(__mul64hi(uy, dz));
    };
    auto evaluate = [&]() {  // one pair per lane that has one
        if (n > 0) {
            const int q = ring[32 * head];
            head = (head + 1) & (kRing - 1);
            --n;
            eval(q);
        }
    };

    for (int b = bb; b < be; ++b) {
        const int k = 32 * b + lane;
        const int qa = k < cnt ? __ldg(row + k) : -1;
#pragma unroll
        for (int st = 0; st < kTest; ++st) {
            const int q = __shfl_sync(0xffffffffu, qa, (st << 2) + js);
            float4 h, l;
            rec_load(w, q >= 0 ? q : 0, h, l);
            const float dx = (h.x - S.h.x) + (l.x - S.l.x);
            const float dy = (h.y - S.h.y) + (l.y - S.l.y);
            const float dz = (h.z - S.h.z) + (l.z - S.l.z);
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            bool use = q > pthr && r2 < rc2;
            if (q > pthr && fabsf(r2 - rc2) <= band) use = S.inside(q, r2, rc2, c.rc_disp2);
            if (use) {
                ring[32 * ((head + n) & (kRing - 1))] = q;
                ++n;
            }
            npairs += use ? 1u : 0u;
        }
        while (__all_sync(0xffffffffu, n > 0) || __any_sync(0xffffffffu, n > kRing - kTest)) evaluate();
    }
    while (__any_sync(0xffffffffu, n > 0)) evaluate();

    npairs = __reduce_add_sync(0xffffffffu, npairs);
    if (lane == 0 && w.npairs) atomicAdd(w.npairs, (unsigned long long)npairs);
    if (ilive) {
        unsigned long long* ai = w.acc + 16 * p;
        red_add64(ai + 0, aF[0]);
        red_add64(ai + 1, aF[1]);
        red_add64(ai + 2, aF[2]);
        red_add64(ai + 3, aD);
        red_add64(ai + 4, aE);
#pragma unroll
        for (int m = 0; m < 6; ++m) red_add64(ai + 5 + m, aV[m]);
    }
}

// Per atom: the fixed-point totals into the arrays the chain pass, the per-structure
// sums (and the optional three-body pass) read.
__global__ void __launch_bounds__(256) k_disp_fin64(Work w) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= w.Nr) return;
    Units K(w.ks[p]);
    const int iu = ipos_unit(w, w.sid[p]);
    K.kF += iu;
    K.kV += 2 * iu;
    const long long* a = reinterpret_cast<const long long*>(w.acc) + 16 * p;
    auto value = [](long long v, int k) { return ldexp((double)v, -k); };
    ((dbl4*)w.Fd)[p] = dbl4_make(value(a[0], K.kF), value(a[1], K.kF), value(a[2], K.kF), 0.0);
    ((double*)w.dEdn)[p] = -value(a[3], K.kD);
    w.eat[p] = -value(a[4], K.kE);
    double* wv = w.wv + 6 * p;
#pragma unroll
    for (int m = 0; m < 6; ++m) wv[m] = -value(a[5 + m], K.kV);
}

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

cudaError_t launch_disp_cl64(const Work& w, const Consts& c, const dbl4* pair_tab, bool site, cudaStream_t st) {
    if (w.Nr == 0) return cudaGetLastError();
    if (w.ncl > 0) {
        // 16 warps stay resident per SM; with fewer clusters than that each list goes to several warps
        const int64_t want = 16 * (int64_t)w.num_sms;
        const int nsplit = (int)(w.ncl >= want ? 1 : (want / w.ncl < 16 ? (want + w.ncl - 1) / w.ncl : 16));
        const dim3 grid(nblk(w.ncl, 4), (unsigned)nsplit);
        const size_t sm = (size_t)c.T * c.T * kDamp * sizeof(double) +
                          4 * ((size_t)kClusterAtoms * row64_len(c.R) * sizeof(long long) + kRing * 32 * sizeof(int));
#define D3_CL(RR)                                                                          \
    if (site) k_disp_cl64<RR, true><<<grid, 128, sm, st>>>(w, c, pair_tab, nsplit);       \
    else k_disp_cl64<RR, false><<<grid, 128, sm, st>>>(w, c, pair_tab, nsplit);           \
    break
        switch (c.R) {
            case 1: D3_CL(1);
            case 2: D3_CL(2);
            case 3: D3_CL(3);
            case 4: D3_CL(4);
            case 5: D3_CL(5);
            case 6: D3_CL(6);
            default: D3_CL(7);
        }
#undef D3_CL
    }
    k_disp_fin64<<<nblk(w.Nr, 256), 256, 0, st>>>(w);
    return cudaGetLastError();
}

}  // namespace d3gb
