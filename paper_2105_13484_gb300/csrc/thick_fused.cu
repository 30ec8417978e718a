// thick_fused.cu -- the thickness and tracer stage (Eqs. layerthickness,
// tracer, with the transport velocity of Sec. 3.4) as one patch-tiled kernel
// (sm_103a).
//
// The unfused path writes the per-layer edge mass flux h_e (v + u^A) from the
// transport kernel and gathers it back, six edges per cell-layer, in a
// one-thread-per-column kernel whose every layer waits on several rounds of
// gathers.  Here the transport kernel leaves only 2-D results (u^A and the
// FP64 column flux), and one CTA per patch of consecutive cells walks the
// layers from the top, two at a time: the velocities (at the patch's edges)
// and the thickness and tracers (at its cells and their neighbours) of a pair
// of layers sit side by side in shared memory, copied by cp.async one pair
// ahead of the pair being computed; each owned cell's own stage and old
// levels, and its values in the layer below the pair, are loaded by its
// thread (the owned cells are consecutive, so those loads coalesce).  The flux
// is formed in registers.  One barrier per pair.
#include "sse_internal.cuh"
#include "tiles.h"

namespace sse {

namespace {

template <class R> __device__ __forceinline__ R ldg(const R *p) { return __ldg(p); }

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
template <class T> __device__ __forceinline__ void cp_async(T *dst, const T *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_addr(dst)), "l"(src),
                 "n"(sizeof(T)));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::); }
// layer pairs staged in shared memory: one in use, one in flight
constexpr int NBUF = 2;

template <class R> __device__ __forceinline__ const R *sfr_of(const DMesh &m);
template <> __device__ __forceinline__ const double *sfr_of<double>(const DMesh &m) { return m.sfrac; }
template <> __device__ __forceinline__ const float *sfr_of<float>(const DMesh &m) { return m.sfrac_f; }
// per-column shares (partial bottom cells), [L][Cp]
template <class R> __device__ __forceinline__ const R *sfc_of(const DMesh &m);
template <> __device__ __forceinline__ const double *sfc_of<double>(const DMesh &m) { return m.sfc; }
template <> __device__ __forceinline__ const float *sfc_of<float>(const DMesh &m) { return m.sfc_f; }

// correctly rounded reciprocals
__device__ __forceinline__ float rcp_r(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_r(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_r(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_r(double a, double b) { return __dadd_rn(a, b); }
// num / den from r, the correctly rounded reciprocal of den: one residual
// correction of num r gives the correctly rounded quotient for every den
// whose significand is not all ones (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
// 1990, Theorem 8).  A cell-layer's tracers share one reciprocal.
template <class R> __device__ __forceinline__ R quot(R num, R den, R r) {
    const R q = mul_r(num, r);
    return fma_r(fma_r(-q, den, num), r, q);
}

// elements of T in n rounded up to 16 bytes
template <class T> __host__ __device__ __forceinline__ int pad16(int n) {
    return (int)(((size_t)n * sizeof(T) + 15) / 16 * 16 / sizeof(T));
}
template <class T> __device__ __forceinline__ const T &at(const T *base, unsigned off) {
    return *(const T *)((const char *)base + off);
}
template <class T> __device__ __forceinline__ T *carve(char *&p, int n) {
    T *r = reinterpret_cast<T *>(p);
    p += ((size_t)n * sizeof(T) + 15) / 16 * 16;
    return r;
}

}  // namespace

// ---------------------------------------------------------------------------
// Sec. 3.4 per edge, columns only: F^h = cF sum_k v_k h_e,k + cE (extra
// terms), D = F^zeta - F^h, u^A = cA D / sum_k h_e,k; the column flux
// F_col = sum_k v h_e + u^A sum_k h_e (FP64) and u^A in the tendency
// precision.  Sums as in k_transport (a float pair in the mixed form); none
// where k_colflux has left the sum (S_in).  PB (partial bottom cells): the
// edge's own layers, and their thickness summed instead of (zeta + H)_e.
// ---------------------------------------------------------------------------
template <class R, bool PB>
__device__ __forceinline__ void transport_cols_edge(const DMesh &m, const TransportArgs<R> &a,
                                                    R *uA_out, const int e) {
    if (e >= m.E) return;
    const int Ep = m.Ep, Cp = m.Cp, L = PB ? m.ke[e] : m.L;
    const int2 cc = m.coe[e];
    const R ubA = a.ubA[e];
    const R ubB = a.ubB ? a.ubB[e] : R(0);
    const R wA = (R)a.wA, wB = (R)a.wB;
    const bool twoB = a.utB != nullptr;
    PairSum<R> Sacc, hacc;
    // layers in chunks of KC, every load of a chunk issued before its sums
    // (which still run over k in order)
    constexpr int KC = 4;
    for (int k0 = 0; k0 < (a.S_in ? 0 : L); k0 += KC) {
        R h1[KC], h2[KC], xa[KC], xb[KC];
#pragma unroll
        for (int j = 0; j < KC; j++) {
            const int k = k0 + j < L ? k0 + j : L - 1;
            h1[j] = ldg(a.hR + k * Cp + cc.x);
            h2[j] = ldg(a.hR + k * Cp + cc.y);
            xa[j] = ldg(a.utA + k * Ep + e);
            xb[j] = twoB ? ldg(a.utB + k * Ep + e) : R(0);
        }
#pragma unroll
        for (int j = 0; j < KC; j++) {
            if (k0 + j >= L) break;
            const R he = R(0.5) * (h1[j] + h2[j]);
            R v = wA * (ubA + xa[j]);
            if (twoB) v += wB * (ubB + xb[j]);
            Sacc.add(v * he);
            if (PB) hacc.add(he);
        }
    }
    const double S = a.S_in ? a.S_in[e] : Sacc.value();
    const double hs =
        PB ? hacc.value() : 0.5 * ((a.zeta[cc.x] + m.H[cc.x]) + (a.zeta[cc.y] + m.H[cc.y]));
    double Fh = a.cF * S;
    if (a.ex1) Fh += a.cE * a.ex1[e];
    if (a.ex2) Fh += a.cE * a.ex2[e];
    const double uA = a.recon ? a.cA * (a.Fz[e] - Fh) / hs : 0.0;
    if (a.S_out) a.S_out[e] = S;
    a.Fcol[e] = S + uA * hs;
    uA_out[e] = (R)uA;
}

// ---------------------------------------------------------------------------
// The fused thickness/tracer stage.  One CTA of NT threads per patch; owned
// cell l is thread l.  Per layer, with flux_e = h_e (v_e + u^A_e):
//   w_{k+1} = w_k + div(flux)_k - s_k D,  D = div(F_col)   (z-star, from the top)
//   h1 = h_s - s_k dt D (FP64),  h_out = a h^n + b h1
//   (h phi)1 = h phi + dt (-div(flux phi_e) - (phibar_k w_k - phibar_{k+1} w_{k+1})
//              + div(h_e kappa_h grad phi) + kappa_v (D_zt phi_k - D_zt phi_{k+1}))
//   phi_out = (a h^n phi^n + b h1 phi1) / h_out
// the same operators as k_thickness, in the same precisions, arranged so that
// each quantity is formed once (the FP64 kernel is bound by the FP64 pipe: 78%
// of its active cycles, 200 FP64 instructions per cell-layer as k_thickness
// writes them, about 100 here):
//   g_j = (n l / A) h_e v at the cell's edges; div = sum g_j, and the advective
//     divergence of a tracer is (phi div + sum g_j phi_j) / 2;
//   the exchange through a layer's bottom, phibar w - kappa_v D_zt phi, is the
//     next layer's through its top;
//   (h phi)1 enters the combination directly (b h1 phi1 = b (h phi)1), so one
//     division per tracer remains, and the tracers share its reciprocal;
// Level-7 sphere (114,689 cells x 60 layers, T and S), three launches: FP64
// 10.23 -> 5.47 ms, FP32 0.809 -> 0.781 ms per step (the FP32 kernel waits on
// loads and barriers, not on arithmetic); errors against the FP64 scheme unchanged.
// ---------------------------------------------------------------------------
// Two layers per pass: every index, coefficient and address serves both, their
// chains are independent, and half the barriers remain (with patches dealt evenly
// to the SMs: FP64 5.47 -> 3.87 ms, FP32 0.781 -> 0.542 ms).  Every fused
// multiply-add is written out, so that each instantiation of the body rounds
// alike (KH: horizontal tracer diffusion is on in some state of the launch; a
// state without it adds a zero).
//
// PB: partial bottom cells.  The column's own layers end at kc[i], its z-star
// shares are its own, and an edge carries no flux below the layers both its
// cells have; nothing is written below the column's bottom.  (In place of the
// unfused kernels, level 6 x 60 layers, mixed: transport and thickness 1.27 ->
// 0.45 ms per step.)  Such meshes hold absolute tracers, which h phi and its
// Runge-Kutta weights round three times a stage; in FP32 (INC) the tracer is an
// increment of the old level's t (of its own in stage 1),
//   phi_out = t + b ((h phi)1 - h1 t) / h_out,
//   (h phi)1 - h1 t = h (phi - t) + (h - h1) t + dt (...),
// which rounds it once: the errors of a step against 64 bits go from u 1.9e-6, T
// 7.3e-8, S 8.0e-8 to 6.1e-7, 4.1e-8, 4.7e-8 in the same time.  Full columns keep
// h phi: their anomalies are small, and a tracer divided by the rounded h_out
// compensates its error in rho' h, where the increments' does not (u on 512 cells
// 3.3e-7 against 3.5e-7).
template <class R, bool KH, bool PB>
__device__ __forceinline__ void thick_fused_patch(const DMesh &m, const DParams &p, const DThick &t,
                                                  const ThickFArgs<R> &a, const int pid) {
    using R2 = V2<R>;
    const int l = threadIdx.x, NT = blockDim.x;
    const int *cn = t.cnt + 4 * pid;
    const int nO = cn[0], nEO = cn[1], nC1 = cn[2];
    const int *eg_g = t.eogid + t.off_eo[pid];
    const int *cg_g = t.c1gid + t.off_c1[pid];

    const int Ep = m.Ep, Cp = m.Cp, L = m.L, Pc = t.Pc;
    const int NP = (L + 1) / 2;   // layer pairs (the second layer of the last is absent if L is odd)
    const int nT = p.nT;
    const bool twoB = a.utB != nullptr, comb = a.a != 0.0;
    constexpr bool INC = PB && sizeof(R) == 4;
    const PhysR<R> &q = phys<R>(p);

    extern __shared__ __align__(16) char smem[];
    char *sp = smem;
    const int sE = pad16<R2>(t.maxEO + 1), sC = pad16<R2>(t.maxC1);
    R *vb_s = carve<R>(sp, t.maxEO + 1);       // wA ubA + wB ubB + u^A per edge (0: zero slot)
    R2 *uA_r = carve<R2>(sp, NBUF * sE);            // utA
    R2 *uB_r = carve<R2>(sp, twoB ? NBUF * sE : 1); // utB
    R2 *h_r = carve<R2>(sp, NBUF * sC);             // hR_s at C1
    R2 *tr_r = carve<R2>(sp, NBUF * nT * sC);       // tracers at C1, [pair][t][C1]
    int *eg = carve<int>(sp, t.maxEO);   // the patch's internal indices
    int *cg = carve<int>(sp, t.maxC1);
    for (int j = l; j < nEO; j += NT) eg[j] = eg_g[j];
    for (int j = l; j < nC1; j += NT) cg[j] = cg_g[j];
    __syncthreads();

    // one pair's copies into buffer b (the second layer's only if it exists)
    auto issue = [&](int pp, int b) {
        const int k0 = 2 * pp;
        const bool has1 = k0 + 1 < L;
        R *uA = reinterpret_cast<R *>(uA_r + b * sE), *uB = reinterpret_cast<R *>(uB_r + b * sE);
        const R *gA = a.utA + (size_t)k0 * Ep, *gB = twoB ? a.utB + (size_t)k0 * Ep : nullptr;
        for (int j = l; j < nEO; j += NT) {
            const int e = eg[j];
            cp_async(uA + 2 * j, gA + e);
            if (has1) cp_async(uA + 2 * j + 1, gA + Ep + e);
            if (twoB) {
                cp_async(uB + 2 * j, gB + e);
                if (has1) cp_async(uB + 2 * j + 1, gB + Ep + e);
            }
        }
        R *hd = reinterpret_cast<R *>(h_r + b * sC), *td = reinterpret_cast<R *>(tr_r + b * nT * sC);
        const R *gh = a.hR_s + (size_t)k0 * Cp, *gt = a.tr_s + (size_t)k0 * Cp;
        for (int j = l; j < nC1; j += NT) {
            const int c = cg[j];
            cp_async(hd + 2 * j, gh + c);
            if (has1) cp_async(hd + 2 * j + 1, gh + Cp + c);
            for (int tt = 0; tt < nT; tt++) {
                R *d = td + 2 * (tt * sC + j);
                const R *g = gt + (size_t)tt * L * Cp + c;
                cp_async(d, g);
                if (has1) cp_async(d + 1, g + Cp);
            }
        }
        cp_async_commit();
    };
    issue(0, 0);
    // the per-edge 2-D part of the transport velocity
    const R wA = (R)a.wA, wB = (R)a.wB;
    for (int j = l; j < nEO; j += NT) {
        const int e = eg[j];
        R v = wA * ldg(a.ubA + e) + ldg(a.uA + e);
        if (twoB) v += wB * ldg(a.ubB + e);
        vb_s[j] = v;
    }
    if (l == 0) {
        // the zero slot that stands in for a pentagon's absent sixth edge
        R2 z;
        z.x = R(0); z.y = R(0);
        vb_s[nEO] = R(0);
        for (int b = 0; b < NBUF; b++) {
            uA_r[b * sE + nEO] = z;
            if (twoB) uB_r[b * sE + nEO] = z;
        }
    }

    // the owned cell's connectivity (byte offsets into the pairs of edges and
    // cells) and column data
    const bool own = l < nO;
    const int i = own ? cg[l] : 0;
    unsigned eo[BCL_NCEP];
    int kj[PB ? BCL_NCEP : 1];   // the layers of the cell's edges
    const int K = !own ? 0 : PB ? m.kc[i] : L;
    R dcf[BCL_NCEP], dif_c[KH ? BCL_NCEP : 1];
    double D = 0.0;
#pragma unroll
    for (int j = 0; j < BCL_NCEP; j++) {
        eo[j] = 0;
        dcf[j] = R(0);
        if (KH) dif_c[j] = R(0);
        if (PB) kj[j] = 0;
        if (own) {
            const size_t x = (size_t)BCL_NCEP * Pc * pid + (size_t)j * Pc + l;
            const int es = t.o_e[x], os = t.o_o[x];
            eo[j] = (unsigned)(es * sizeof(R2)) | ((unsigned)(os * sizeof(R2)) << 16);
            if (j < m.neoc[i]) {
                const int e = eg[es];
                const R dc = coef<R>(m).divc[j * Cp + i];
                dcf[j] = R(0.5) * dc;   // with the 1/2 of h_e
                if (KH) dif_c[j] = fabs(dcf[j]) * q.kappa_h * coef<R>(m).invdc[e];
                if (PB) kj[j] = m.ke[e];
                D += m.divc_d[j * Cp + i] * a.Fcol[e];
            }
        }
    }
    const R Dr = (R)D;
    const double dtD = a.dt * D;
    const R *sfr = sfr_of<R>(m), *sfcR = sfc_of<R>(m);
    const R dtR = (R)a.dt, aR = (R)a.a, bR = (R)a.b, kv = q.kappa_v;
    const R dtDr = dtR * Dr;
    double hsum = 0.0;
    R wk = R(0);
    R X0 = R(0), X1 = R(0);   // the tracers' exchange through the layer's top

    for (int pp = 0; pp < NP; pp++) {
        const int k0 = 2 * pp, bc = pp & 1;
        const bool has1 = k0 + 1 < K, has2 = k0 + 2 < K;
        cp_async_wait_all();
        __syncthreads();   // pair pp staged; pair pp - 1's readers done
        if (pp + 1 < NP) issue(pp + 1, bc ^ 1);
        if (k0 >= K) continue;
        // the owned cell's own stage and old levels and the layer below the
        // pair: coalesced loads (the owned cells are consecutive), used after
        // the flux loop below
        const size_t x = (size_t)k0 * Cp + i;
        double hs_d[2], hn[2] = {0.0, 0.0};
        R hnr[2] = {R(0), R(0)}, trn[2][2] = {{R(0), R(0)}, {R(0), R(0)}};
        R h_b = R(0), tr_b[2] = {R(0), R(0)};
#pragma unroll
        for (int r = 0; r < 2; r++) {
            hs_d[r] = 0.0;
            if (r && !has1) continue;
            const size_t y = x + (size_t)r * Cp;
            hs_d[r] = a.h_s[y];
            if (comb) {
                hn[r] = a.h_n[y];
                if constexpr (sizeof(R) == 4) hnr[r] = a.hR_n[y];
                else hnr[r] = hn[r];
                trn[r][0] = a.tr_n[y];
                if (nT > 1) trn[r][1] = a.tr_n[(size_t)L * Cp + y];
            }
        }
        if (has2) {
            h_b = a.hR_s[x + 2 * (size_t)Cp];
            tr_b[0] = a.tr_s[x + 2 * (size_t)Cp];
            if (nT > 1) tr_b[1] = a.tr_s[(size_t)(L + 2) * Cp + x];
        }
        const R2 *uA_c = uA_r + bc * sE, *uB_c = uB_r + bc * sE, *h_c = h_r + bc * sC;
        const R2 hc = h_c[l];
        // flux at the cell's edges and its divergence
        R2 fl[BCL_NCEP], dv;
        dv.x = R(0); dv.y = R(0);
#pragma unroll
        for (int j = 0; j < BCL_NCEP; j++) {
            const unsigned oe = eo[j] & 0xffffu, oc = eo[j] >> 16;
            const R vb = at(vb_s, oe / 2);
            const R2 u = at(uA_c, oe), ho = at(h_c, oc);
            R2 v;
            v.x = fma_r(wA, u.x, vb);
            v.y = fma_r(wA, u.y, vb);
            if (twoB) {
                const R2 w = at(uB_c, oe);
                v.x = fma_r(wB, w.x, v.x);
                v.y = fma_r(wB, w.y, v.y);
            }
            fl[j].x = mul_r(dcf[j], mul_r(add_r(hc.x, ho.x), v.x));
            fl[j].y = mul_r(dcf[j], mul_r(add_r(hc.y, ho.y), v.y));
            if (PB && k0 >= kj[j]) fl[j].x = R(0);
            if (PB && k0 + 1 >= kj[j]) fl[j].y = R(0);
            dv.x = add_r(dv.x, fl[j].x);
            dv.y = add_r(dv.y, fl[j].y);
        }
        const R sk0 = PB ? sfcR[x] : sfr[k0];
        const R sk1 = !has1 ? R(0) : PB ? sfcR[x + Cp] : sfr[k0 + 1];
        // w at the tops of layers k0 + 1 and k0 + 2 (0 at the bottom)
        const R w1 = has1 ? fma_r(-sk0, Dr, add_r(wk, dv.x)) : R(0);
        const R w2 = has2 ? fma_r(-sk1, Dr, add_r(w1, dv.y)) : R(0);
        // kappa_v / the distances to the next layers' middles
        const R kvd1 = has1 ? mul_r(kv, rcp_r(mul_r(R(0.5), add_r(hc.x, hc.y)))) : R(0);
        const R kvd2 = has2 ? mul_r(kv, rcp_r(mul_r(R(0.5), add_r(hc.y, h_b)))) : R(0);
        // the new thickness: FP64 from the column-integrated flux (volume
        // conservation), and in the tendency precision for the tracers
        R hor[2], rout[2], bh[2], dh[2];   // bh = a h^n; dh = h - h1 (increments)
#pragma unroll
        for (int r = 0; r < 2; r++) {
            hor[r] = R(1); rout[r] = R(1); bh[r] = R(0); dh[r] = R(0);
            if (r && !has1) continue;
            const double share = PB ? m.sfc[x + (size_t)r * Cp] : m.sfrac[k0 + r];
            const double h1 = fma_r(-share, dtD, hs_d[r]);
            const double ho = comb ? fma_r(a.a, hn[r], a.b * h1) : h1;
            a.h_out[x + (size_t)r * Cp] = ho;
            hsum += ho;
            if constexpr (sizeof(R) == 8) {
                hor[r] = ho;
            } else {
                const R h1r = fma_r(-(r ? sk1 : sk0), dtDr, r ? hc.y : hc.x);
                hor[r] = comb ? fma_r(aR, hnr[r], mul_r(bR, h1r)) : h1r;
                a.hR_out[x + (size_t)r * Cp] = hor[r];
                dh[r] = mul_r(r ? sk1 : sk0, dtDr);
            }
            rout[r] = rcp_r(hor[r]);
            if (!INC) bh[r] = mul_r(aR, hnr[r]);
        }
#pragma unroll
        for (int tt = 0; tt < 2; tt++) {
            if (tt >= nT) break;
            const R2 *phi = tr_r + (bc * nT + tt) * sC;
            const R2 ph = phi[l];
            R2 adv, dif;
            adv.x = mul_r(ph.x, dv.x);
            adv.y = mul_r(ph.y, dv.y);
            dif.x = R(0); dif.y = R(0);
#pragma unroll
            for (int j = 0; j < BCL_NCEP; j++) {
                const R2 po = at(phi, eo[j] >> 16);
                adv.x = fma_r(fl[j].x, po.x, adv.x);
                adv.y = fma_r(fl[j].y, po.y, adv.y);
                if (KH) {
                    const R2 ho = at(h_c, eo[j] >> 16);
                    if (!PB || k0 < kj[j]) dif.x = fma_r(mul_r(dif_c[j], add_r(hc.x, ho.x)), add_r(po.x, -ph.x), dif.x);
                    if (!PB || k0 + 1 < kj[j]) dif.y = fma_r(mul_r(dif_c[j], add_r(hc.y, ho.y)), add_r(po.y, -ph.y), dif.y);
                }
            }
            // phibar w - kappa_v D_zt phi at the two layers' bottoms
            const R pb = tt ? tr_b[1] : tr_b[0];
            const R Xt = tt ? X1 : X0;
            R Xm = R(0), Xb = R(0);
            if (has1)
                Xm = fma_r(mul_r(R(0.5), add_r(ph.x, ph.y)), w1, -mul_r(kvd1, add_r(ph.x, -ph.y)));
            if (has2)
                Xb = fma_r(mul_r(R(0.5), add_r(ph.y, pb)), w2, -mul_r(kvd2, add_r(ph.y, -pb)));
            if (tt) X1 = Xb; else X0 = Xb;
#pragma unroll
            for (int r = 0; r < 2; r++) {
                if (r && !has1) continue;
                R rate = fma_r(R(-0.5), r ? adv.y : adv.x, r ? add_r(Xb, -Xm) : add_r(Xm, -Xt));
                if (KH) rate = add_r(rate, r ? dif.y : dif.x);
                const R hr = r ? hc.y : hc.x, phr = r ? ph.y : ph.x;
                R out;
                if constexpr (!INC) {
                    const R hphi = fma_r(dtR, rate, mul_r(hr, phr));
                    const R num = comb ? fma_r(bh[r], trn[r][tt], mul_r(bR, hphi)) : hphi;
                    out = quot(num, hor[r], rout[r]);
                } else {
                    const R t0 = comb ? trn[r][tt] : phr;
                    const R inc = fma_r(dtR, rate, fma_r(hr, add_r(phr, -t0), mul_r(dh[r], t0)));
                    out = add_r(t0, quot(comb ? mul_r(bR, inc) : inc, hor[r], rout[r]));
                }
                a.tr_out[(size_t)tt * L * Cp + x + (size_t)r * Cp] = out;
            }
        }
        wk = w2;
    }
    if (own) a.zeta_out[i] = hsum - m.H[i];
}


constexpr int THICK_NT = 128;   // cells per patch and threads per CTA, at most

// ---------------------------------------------------------------------------
// batched launches (see bcl_fused.cu): job j owns blocks [first[j], first[j+1])
// ---------------------------------------------------------------------------
__device__ __forceinline__ int job_of_block_t(const int *first, int njobs) {
    int lo = 0, hi = njobs - 1;
    const int b = blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}
template <class T> __device__ __forceinline__ void copy_job_t(T &dst, const T &src) {
    static_assert(sizeof(T) % 4 == 0, "job descriptors are copied in 4-byte words");
    const int *s = reinterpret_cast<const int *>(&src);
    int *d = reinterpret_cast<int *>(&dst);
    for (int i = threadIdx.x; i < (int)(sizeof(T) / 4); i += blockDim.x) d[i] = s[i];
}
// single-state and batched kernels run the body on a shared-memory copy of
// their descriptor, so that the body compiles identically in both (a state's
// results are the same bits alone or in a batch)
//
// Resident CTAs per SM asked of the compiler (THICK_NT threads each): the
// registers that leaves are 80 in FP32 (6 CTAs).  0 leaves the FP64 body's
// register count to the compiler.
template <class R> constexpr int thick_min_blocks() { return sizeof(R) == 4 ? 6 : 0; }
template <class R, bool KH, bool PB>
__global__ void __launch_bounds__(THICK_NT, thick_min_blocks<R>()) k_thick_fused(const ThickJob<R> job) {
    __shared__ ThickJob<R> J;
    copy_job_t(J, job);
    __syncthreads();
    thick_fused_patch<R, KH, PB>(J.m, J.p, J.t, J.a, blockIdx.x);
}
template <class R, bool KH>
__global__ void __launch_bounds__(THICK_NT, thick_min_blocks<R>()) k_thick_fused_batch(const ThickJob<R> *__restrict__ jobs,
                                                          const int *__restrict__ first,
                                                          int njobs) {
    __shared__ ThickJob<R> J;
    const int j = job_of_block_t(first, njobs);
    copy_job_t(J, jobs[j]);
    __syncthreads();
    thick_fused_patch<R, KH, false>(J.m, J.p, J.t, J.a, blockIdx.x - first[j]);
}
template <class R, bool PB>
__global__ void __launch_bounds__(128) k_transport_cols(const TransportJob<R> job) {
    __shared__ TransportJob<R> J;
    copy_job_t(J, job);
    __syncthreads();
    transport_cols_edge<R, PB>(J.m, J.a, J.uA, blockIdx.x * blockDim.x + threadIdx.x);
}
template <class R>
__global__ void __launch_bounds__(128) k_transport_cols_batch(const TransportJob<R> *__restrict__ jobs,
                                                              const int *__restrict__ first,
                                                              int njobs) {
    __shared__ TransportJob<R> J;
    const int j = job_of_block_t(first, njobs);
    copy_job_t(J, jobs[j]);
    __syncthreads();
    transport_cols_edge<R, false>(J.m, J.a, J.uA, (blockIdx.x - first[j]) * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------
size_t thick_smem_bytes(const DThick &plan, int nT, bool twoB, size_t sR) {
    auto a16 = [](size_t b) { return (b + 15) / 16 * 16; };
    size_t b = a16(sR * (plan.maxEO + 1));
    b += NBUF * a16(2 * sR * (plan.maxEO + 1)) * (twoB ? 2 : 1) + (twoB ? 0 : a16(2 * sR));
    b += NBUF * a16(2 * sR * plan.maxC1) * (1 + nT);
    b += a16(4 * (size_t)plan.maxEO) + a16(4 * (size_t)plan.maxC1);
    return b;
}
int thick_cells_per_patch() { return THICK_NT; }
template <class R> const void *thick_fused_kernel_ptr(bool kh, bool pb) {
    if (pb) return kh ? (const void *)k_thick_fused<R, true, true>
                      : (const void *)k_thick_fused<R, false, true>;
    return kh ? (const void *)k_thick_fused<R, true, false>
              : (const void *)k_thick_fused<R, false, false>;
}

template <class R>
void launch_transport_cols(const DMesh &m, const TransportArgs<R> &a, R *uA, cudaStream_t s) {
    const TransportJob<R> job{m, a, uA};
    if (m.partial) k_transport_cols<R, true><<<(m.E + 127) / 128, 128, 0, s>>>(job);
    else k_transport_cols<R, false><<<(m.E + 127) / 128, 128, 0, s>>>(job);
}
template <class R>
void launch_thick_fused(const DThick &t, const DMesh &m, const DParams &p, const ThickFArgs<R> &a,
                        size_t smem, cudaStream_t s) {
    const ThickJob<R> job{m, p, t, a};
    const bool kh = p.kappa_h != 0.0;
    if (m.partial) {
        if (kh) k_thick_fused<R, true, true><<<t.P, t.Pc, smem, s>>>(job);
        else k_thick_fused<R, false, true><<<t.P, t.Pc, smem, s>>>(job);
    } else {
        if (kh) k_thick_fused<R, true, false><<<t.P, t.Pc, smem, s>>>(job);
        else k_thick_fused<R, false, false><<<t.P, t.Pc, smem, s>>>(job);
    }
}

template <class R>
void launch_transport_cols_batch(const TransportJob<R> *jobs, const int *first, int njobs,
                                 int blocks, cudaStream_t s) {
    k_transport_cols_batch<R><<<blocks, 128, 0, s>>>(jobs, first, njobs);
}
template <class R>
void launch_thick_fused_batch(const ThickJob<R> *jobs, const int *first, int njobs, int blocks,
                              size_t smem, bool kh, cudaStream_t s) {
    if (kh) k_thick_fused_batch<R, true><<<blocks, THICK_NT, smem, s>>>(jobs, first, njobs);
    else k_thick_fused_batch<R, false><<<blocks, THICK_NT, smem, s>>>(jobs, first, njobs);
}
template <class R> const void *thick_fused_batch_kernel_ptr(bool kh) {
    return kh ? (const void *)k_thick_fused_batch<R, true>
              : (const void *)k_thick_fused_batch<R, false>;
}
template void launch_transport_cols_batch<float>(const TransportJob<float> *, const int *, int,
                                                 int, cudaStream_t);
template void launch_transport_cols_batch<double>(const TransportJob<double> *, const int *, int,
                                                  int, cudaStream_t);
template void launch_thick_fused_batch<float>(const ThickJob<float> *, const int *, int, int,
                                              size_t, bool, cudaStream_t);
template void launch_thick_fused_batch<double>(const ThickJob<double> *, const int *, int, int,
                                               size_t, bool, cudaStream_t);
template const void *thick_fused_batch_kernel_ptr<float>(bool);
template const void *thick_fused_batch_kernel_ptr<double>(bool);
template const void *thick_fused_kernel_ptr<float>(bool, bool);
template const void *thick_fused_kernel_ptr<double>(bool, bool);
template void launch_transport_cols<float>(const DMesh &, const TransportArgs<float> &, float *,
                                           cudaStream_t);
template void launch_transport_cols<double>(const DMesh &, const TransportArgs<double> &, double *,
                                            cudaStream_t);
template void launch_thick_fused<float>(const DThick &, const DMesh &, const DParams &,
                                        const ThickFArgs<float> &, size_t, cudaStream_t);
template void launch_thick_fused<double>(const DThick &, const DMesh &, const DParams &,
                                         const ThickFArgs<double> &, size_t, cudaStream_t);

}  // namespace sse
