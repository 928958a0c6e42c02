// Device helpers of the solver passes, shared by the translation units that hold their kernels: mask
// decisions, the Adam step, record layouts, and the per-unit work of the Active Set passes after their
// sums (f, x*, z* and snapshots of an input; supergradient and dual updates of a row).
#pragma once
#include "cb_common.cuh"
#include "cb_walk.cuh"

namespace cb {

// Active Set mask bits of every slot for one (i, j) pair (eq. 3 at binary iterates).
// zs: bit b = z*_k[i] when slot b was added; xs: bit b = (x*_{k-1}[j] was at its upper bound).
// With z = 1 the row is all ones; with z = 0 the bit is 1 where the coefficient
// ((1-z) Lcheck + z Ucheck - x) W is >= 0: W > 0 and x at its lower bound, W < 0 and x at its
// upper bound, W = 0, or l = u (fixed input, coefficient exactly 0). An input strictly inside its
// box (interior: layer 0 over an ellipsoid) is at neither end: the bit is z, or 1 where W = 0 or l = u.
__device__ __forceinline__ unsigned cb_slot_mask(unsigned zs, unsigned xs, bool fixed, float w,
                                                 bool interior = false) {
    unsigned xm = fixed ? 0xFFu
                        : (w > 0.f ? (interior ? 0u : (~xs & 0xFFu)) : (w < 0.f ? (interior ? 0u : xs) : 0xFFu));
    return zs | xm;
}

// Saddle Point oracle bit, eq. (3) with continuous (x, z), in the threshold form: W > 0 ->
// z (u - l) >= x - l, W < 0 -> z (u - l) >= u - x (eq. 3 with the sign of W multiplied out), i.e.
// z >= tau for tau = (x - l) / (u - l), resp. (u - x) / (u - l); W = 0 or l = u -> 1 (fixed inputs
// carry thresholds of -inf). The thresholds are cb_tau_up's, so each float32 compare is exact.
__device__ __forceinline__ bool cb_sp_mask(float z, float tp, float tn, float w) {
    return w > 0.f ? (z >= tp) : (w < 0.f ? (z >= tn) : true);
}

// The smallest float32 at or above the real quotient (a - b) / (hi - lo), for float32 a, b, lo <
// hi: the differences are exact in float64 (float32 operands whose magnitudes lie within 2^28 of
// each other), the quotient is rounded up in float64 and again to float32. Rounding up twice
// gives the float32 rounding up of the real quotient (a float32 is a float64), so for every
// float32 z, z >= tau (real) exactly when z >= this value: the mask decision of eq. (3) is exact.
__device__ __forceinline__ float cb_tau_up(float a, float b, float lo, float hi) {
    return __double2float_ru(__ddiv_ru((double)a - (double)b, (double)hi - (double)lo));
}

// Block-to-segment lookup for launches that cover several layers.
struct Segs {
    int n;
    int layer[CB_MAXL];   // 0-based layer index
    int start[CB_MAXL + 1];
};
__device__ __forceinline__ int seg_of(const Segs& sg, int blk) {
    int q = 0;
    while (q + 1 < sg.n && blk >= sg.start[q + 1]) ++q;
    return q;
}

// One projected Adam ascent step (Kingma and Ba) of a dual variable: returns the new value and
// updates the moments. Fast reciprocal square root and division (a few float32 ulps).
__device__ __forceinline__ float adam_step(float th, float& m, float& v, float g, float lr, float ibc1,
                                           float ibc2, const DSched& sc) {
    m = sc.b1 * m + sc.omb1 * g;
    v = sc.b2 * v + sc.omb2 * g * g;
    const float mh = m * ibc1, vh = v * ibc2;
    const float sq = vh > 0.f ? vh * rsqrtf(vh) : 0.f;
    return fmaxf(th + lr * __fdividef(mh, sq + sc.eps), 0.f);
}

struct TSegs {
    int n;
    int layer[CB_MAXL];
    int start[CB_MAXL + 1];   // first block of each segment
    int T[CB_MAXL];           // team size (1, 2, 4, 8, 16 or 32)
    const int* perm[CB_MAXL]; // col pass of a strided conv: unit order -> input index (or null)
};

__device__ __forceinline__ float team_sum(float v, int T) {
    for (int o = T >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------- Active Set walks
// Group and base position of row-pass unit i (output neuron i of layer L).
__device__ __forceinline__ void row_group(const DLayer& L, int i, int& g, int& base) {
    if (L.kind == 0) {
        g = i;
        base = 0;
        return;
    }
    const int hw = L.ho * L.wo;
    const int co = i / hw, rem = i - co * hw;
    const int oy = rem / L.wo, ox = rem - oy * L.wo;
    g = co;
    base = oy * L.st * L.Wp + ox * L.st;
}

// Group and base position of col-pass unit j (input neuron j of layer L).
__device__ __forceinline__ void col_group(const DLayer& L, int j, int& g, int& base) {
    if (L.kind == 0) {
        g = j;
        base = 0;
        return;
    }
    const int hw = L.hi * L.wi;
    const int c = j / hw, rem = j - c * hw;
    const int y = rem / L.wi, x = rem - y * L.wi;
    const int ty = y + L.pd, tx = x + L.pd;
    const int Y0 = ty / L.st, X0 = tx / L.st;
    const int py = ty - Y0 * L.st, px = tx - X0 * L.st;
    g = (c * L.st + py) * L.st + px;
    base = (Y0 + L.hl) * L.Wpo + X0 + L.wl;
}

// Record position of input neuron j (row-pass input records) and output neuron i (col-pass
// output records) of layer L.
__device__ __forceinline__ int xin_pos(const DLayer& L, int j) {
    if (L.kind == 0) return j;
    const int hw = L.hi * L.wi;
    const int c = j / hw, rem = j - c * hw;
    const int y = rem / L.wi, x = rem - y * L.wi;
    return (c * L.Hp + y + L.pd) * L.Wp + x + L.pd;
}
__device__ __forceinline__ int arec_pos(const DLayer& L, int i) {
    if (L.kind == 0) return i;
    const int hw = L.ho * L.wo;
    const int co = i / hw, rem = i - co * hw;
    const int oy = rem / L.wo, ox = rem - oy * L.wo;
    return (co * L.Hpo + oy + L.hl) * L.Wpo + ox + L.wl;
}

// Output records of layer L for subproblem s: RS / 4 planes of float4, plane q holding entries
// 4q .. 4q + 3 of every position, so that lanes reading neighbouring positions read one
// contiguous run per plane.
__device__ __forceinline__ float4* arec_planes(const DNet& net, const DState& st, const DLayer& L, int s) {
    return reinterpret_cast<float4*>(st.arec + (size_t)s * net.AT + L.ao);
}
__device__ __forceinline__ float* arec_entry(const DNet& net, const DState& st, const DLayer& L, int s, int p, int e) {
    return reinterpret_cast<float*>(arec_planes(net, st, L, s) + (size_t)(e >> 2) * L.apos + p) + (e & 3);
}
// Subproblem s's first Active Set input record of layer L.
__device__ __forceinline__ float2* xin_recs(const DNet& net, const DState& st, const DLayer& L, int s) {
    return reinterpret_cast<float2*>(st.xin + (size_t)s * net.XT + L.xo);
}

// Records of the float32 slot row sums (k_slot_sums_t below): per input {l, u, p bits | q bits
// << 8} in the first Saddle Point input plane, which Active Set leaves unused.
__device__ __forceinline__ float4* slot_rec_plane(const DNet& net, const DState& st, const DLayer& L, int s) {
    return st.spin + (size_t)s * net.XT + (size_t)L.xo;
}
// The record of an input with box [lo, hi] and snapshot bits xs (bit b: at its upper end when slot b
// was added); a fixed input (lo = hi) is selected by every mask, an interior one (layer 0 over an
// ellipsoid) by none: its bit is z alone.
__device__ __forceinline__ float4 slot_rec(float lo, float hi, unsigned xs, bool fixed, bool interior) {
    const unsigned fxm = fixed ? 0xFFu : 0u;
    const unsigned pm = (interior ? 0u : (~xs & 0xFFu)) | fxm, qm = (interior ? 0u : (xs & 0xFFu)) | fxm;
    return make_float4(lo, hi, __uint_as_float(pm | (qm << 8)), 0.f);
}

// Slot bits p_b, q_b of an input with snapshot bits xs: an interior input (layer 0 over an ellipsoid)
// is at neither end of its box (eq. 3 gives z), a fixed one at both.
__device__ __forceinline__ void slot_bits(const DNet& net, const DLayer& L, unsigned xs, bool fixed, unsigned& pm,
                                          unsigned& qm) {
    const bool interior = net.ball && L.in_off == 0;
    const unsigned fxm = fixed ? 0xFFu : 0u;
    pm = (interior ? 0u : ((~xs) & 0xFFu)) | fxm;
    qm = (interior ? 0u : xs) | fxm;
}

// What the col pass reads for input j of layer L (m = k - 1 its own hidden layer) beside its sum.
template <int NS>
struct ColState {
    float lo, hi, al, b0, b1, uh, lh, bm;
    float bs[NS > 0 ? NS : 1], kap[NS > 0 ? NS : 1], lam[NS > 0 ? NS : 1];
    unsigned xs;
    bool fixed;
    int cap_s;
};
template <int NS>
__device__ __forceinline__ ColState<NS> as_colA_load(const DNet& net, const DState& st, const StepNow& sp, const DLayer& L,
                                                     int k, int s, int j, int mode) {
    ColState<NS> c;
    const size_t xo = (size_t)s * net.NT + L.in_off + j;
    c.lo = st.lo[xo];
    c.hi = st.hi[xo];
    c.xs = st.xsnap[sp.nadd_before & 1][xo];
    c.fixed = st.efix[xo];
    c.cap_s = st.caps[s];
    if (k < 2) return c;
    const size_t h = (size_t)s * net.NH + L.h_in + j, hs = (size_t)s * net.cap * net.NH + L.h_in + j;
    c.al = st.alpha[h];
    c.b0 = st.beta0[h];
    c.b1 = st.beta1[h];
    c.uh = st.uhat[h];
    c.lh = st.lhat[h];
    const int nsl = min(sp.nadd_before, c.cap_s);
#pragma unroll
    for (int b = 0; b < NS; ++b) {
        c.bs[b] = c.kap[b] = c.lam[b] = 0.f;
        if (b < nsl) {
            c.bs[b] = st.bs[hs + (size_t)b * net.NH];
            c.kap[b] = st.kap[hs + (size_t)b * net.NH];
            if (mode != 2) c.lam[b] = st.lam[hs + (size_t)b * net.NH];
        }
    }
    if (mode != 2) c.bm = net.L[k - 2].b[j];
    return c;
}

// Col pass, one input j of layer L after its walk: f is the masked backward product (minus the output
// row's entry for the inputs of the last layer), c the input's state.
template <int NS>
__device__ __forceinline__ void as_colA_unit(const DNet& net, const DState& st, const StepNow& sp, const DLayer& L, int k,
                                             int s, int j, float f, const ColState<NS>& c, int mode) {
    const bool want_terms = mode != 2;
    const int nsl = min(sp.nadd_before, c.cap_s);
    const int bo = sp.nadd_before & 1;
    const bool add_iter = (mode != 1) && sp.b_new >= 0;
    const bool add = add_iter && sp.b_new < c.cap_s;
    const size_t xo = (size_t)s * net.NT + L.in_off + j;
    const unsigned fxm = c.fixed ? 0xFFu : 0u;
    double term = 0.0;
    if (k >= 2) {
        const size_t h = (size_t)s * net.NH + L.h_in + j;
        float sb = 0.f, gk = c.b0 * c.uh + c.b1 * c.lh;
        double cterm = 0.0;
#pragma unroll
        for (int b = 0; b < NS; ++b)
            if (b < nsl) {
                sb += c.bs[b];
                gk += c.bs[b] * c.kap[b];
                if (want_terms) cterm += (double)c.bs[b] * c.lam[b];
            }
        f += c.al - c.b0 - c.b1 - sb;
        const bool z = gk >= 0.f;
        st.zcur[h] = z;
        if (want_terms)
            term = (double)c.bm * c.al + (double)c.b1 * ((double)c.lh - c.bm) + cterm - (z ? (double)gk : 0.0);
        if (add_iter) {
            const unsigned zs_old = st.zsnap[bo][h];
            st.zsnap[bo ^ 1][h] = (uint8_t)(zs_old | ((add && z) ? (1u << sp.b_new) : 0u));
        }
    }
    const bool up = f >= 0.f;
    const float xv = up ? c.hi : c.lo;
    st.xval[xo] = xv;
    // f is read by the gradient (after a mode 1 evaluation) and by the ellipsoid's x_0*
    if (mode == 1 || net.ball) st.fval[xo] = f;
    if (want_terms) st.terms[xo] = term - (double)f * xv;
    unsigned xs_new = c.xs;
    if (add_iter) {
        xs_new = c.xs | ((add && up) ? (1u << sp.b_new) : 0u);
        st.xsnap[bo ^ 1][xo] = (uint8_t)xs_new;
    }
    if (k <= net.n - 1) {
        const unsigned mpos = ((~xs_new) & 0xFFu) | fxm, mneg = (xs_new & 0xFFu) | fxm;
        // row-pass input record: x* and the slot masks p_b (bits 0-7) and q_b (bits 8-15)
        xin_recs(net, st, L, s)[xin_pos(L, j)] = make_float2(xv, __uint_as_float(mpos | (mneg << 8)));
    }
}

// What the row pass reads for row i of layer L beside its sums: its duals and moments (alpha, beta_0,
// beta_1), and with SLOTS its slots' too.
template <int NS>
struct RowState {
    float th[3], m[3], v[3], uh, lh, x, z, bi;
    float bs[NS > 0 ? NS : 1], ms[NS > 0 ? NS : 1], vs[NS > 0 ? NS : 1], lam[NS > 0 ? NS : 1], kap[NS > 0 ? NS : 1];
    unsigned zs;
    int cap_s;
};
// Slot b of a row: the slot the iteration adds (newb) takes its lambda and kappa from this iteration.
template <int NS, bool ADD>
__device__ __forceinline__ void row_load_slot(const DNet& net, const DState& st, size_t hs0, int b, int nsl, int newb,
                                              RowState<NS>& r) {
    r.bs[b] = r.ms[b] = r.vs[b] = r.lam[b] = r.kap[b] = 0.f;
    if (b >= nsl) return;
    const size_t hs = hs0 + (size_t)b * net.NH;
    r.bs[b] = st.bs[hs];
    r.ms[b] = st.ms[hs];
    r.vs[b] = st.vs[hs];
    if (!(ADD && b == newb)) {
        r.lam[b] = st.lam[hs];
        r.kap[b] = st.kap[hs];
    }
}
template <int NS, bool ADD, bool SLOTS>
__device__ __forceinline__ RowState<NS> as_rowB_load(const DNet& net, const DState& st, const DLayer& L, int s, int i,
                                                     const StepNow& sp) {
    RowState<NS> r;
    const int bn = (sp.nadd_before + (sp.b_new >= 0 ? 1 : 0)) & 1;
    const size_t h = (size_t)s * net.NH + L.h_out + i;
    r.th[0] = st.alpha[h];
    r.th[1] = st.beta0[h];
    r.th[2] = st.beta1[h];
    r.m[0] = st.ma[h];
    r.m[1] = st.m0[h];
    r.m[2] = st.m1[h];
    r.v[0] = st.va[h];
    r.v[1] = st.v0[h];
    r.v[2] = st.v1[h];
    r.uh = st.uhat[h];
    r.lh = st.lhat[h];
    r.x = st.xval[(size_t)s * net.NT + L.out_off + i];
    r.z = st.zcur[h] ? 1.f : 0.f;
    r.zs = st.zsnap[bn][h];
    r.bi = L.b[i];
    r.cap_s = st.caps[s];
    if constexpr (SLOTS && NS > 0) {
        const int nsl = min(sp.nadd_before + (sp.b_new >= 0 ? 1 : 0), r.cap_s);
        const int newb = (ADD && sp.b_new < r.cap_s) ? sp.b_new : -1;
        const size_t hs0 = (size_t)s * net.cap * net.NH + L.h_out + i;
#pragma unroll
        for (int b = 0; b < NS; ++b) row_load_slot<NS, ADD>(net, st, hs0, b, nsl, newb, r);
    }
    return r;
}

// Row pass, one unit by one lane after its sums (acc0 = W x*, acc[b] the masked products): the
// supergradient, Adam steps and projection of every dual of row i, and the row's output record. SLOTS:
// r holds the slots as well; without, they are loaded in pairs here (a kernel of 64 registers).
template <int NS, bool ADD, bool SLOTS>
__device__ __forceinline__ void as_rowB_unit(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int s,
                                             int i, const StepNow& sp, float acc0, const float* acc,
                                             RowState<NS>& r) {
    const size_t NH = net.NH;
    const int newb = (ADD && sp.b_new < r.cap_s) ? sp.b_new : -1;
    const size_t h = (size_t)s * NH + L.h_out + i;
    const int nsl = min(sp.nadd_before + (sp.b_new >= 0 ? 1 : 0), r.cap_s);
    const float x = r.x, z = r.z;
    const float xhat = acc0 + r.bi;
    const size_t hs0 = (size_t)s * net.cap * NH + L.h_out + i;
    const int ap = arec_pos(L, i);
    auto put = [&](int e, float v) { *arec_entry(net, st, L, s, ap, e) = v; };
    const float2 ib = cb_bias(st);
    const float g3[3] = {xhat - x, x - z * r.uh, x - xhat + (1.f - z) * r.lh};
#pragma unroll
    for (int v = 0; v < 3; ++v) r.th[v] = adam_step(r.th[v], r.m[v], r.v[v], g3[v], sp.lr, ib.x, ib.y, sc);
    st.alpha[h] = r.th[0]; st.beta0[h] = r.th[1]; st.beta1[h] = r.th[2];
    st.ma[h] = r.m[0]; st.m0[h] = r.m[1]; st.m1[h] = r.m[2];
    st.va[h] = r.v[0]; st.v0[h] = r.v[1]; st.v1[h] = r.v[2];
    float contrib = r.th[2] - r.th[0];
#pragma unroll
    for (int b0 = 0; b0 < NS; b0 += 2) {
        if constexpr (!SLOTS) {   // a pair's loads first, then its updates (larger groups spill)
#pragma unroll
            for (int b = b0; b < b0 + 2 && b < NS; ++b) row_load_slot<NS, ADD>(net, st, hs0, b, nsl, newb, r);
        }
#pragma unroll
        for (int b = b0; b < b0 + 2 && b < NS; ++b) {
            if (b >= nsl) {
                put(1 + b, 0.f);
                continue;
            }
            const size_t hs = hs0 + (size_t)b * NH;
            const bool zb = (r.zs >> b) & 1u;
            float lam = r.lam[b], kap = r.kap[b];
            if (ADD && b == newb) {
                const float lzh = st.lz[h];
                lam = zb ? lzh : acc[b];
                // kappa = lambda + sum W (1 - I) Ucheck + b: W x* + b at box vertices; over
                // interior inputs (layer 0, ellipsoid) the z = 0 mask holds fixed inputs only
                kap = zb ? lzh + r.bi : (net.ball && L.in_off == 0 ? st.uz[h] + r.bi : xhat);
                st.lam[hs] = lam;
                st.kap[hs] = kap;
            }
            const float prod = zb ? acc0 : acc[b];
            const float gb = x - prod + lam * (1.f - z) - z * (kap - lam);
            const float2 sib = cb_slot_bias(st, b);
            const float nv = adam_step(r.bs[b], r.ms[b], r.vs[b], gb, sp.lr, sib.x, sib.y, sc);
            st.bs[hs] = nv; st.ms[hs] = r.ms[b]; st.vs[hs] = r.vs[b];
            if (zb) contrib += nv;
            put(1 + b, zb ? 0.f : nv);
        }
    }
    put(0, contrib);
}

// ---------------------------------------------------------------- Saddle Point units
// Saddle Point records, in the Active Set walks' layouts (Active Set and Saddle Point do not run on
// one context at the same time, so the output records reuse the Active Set's array):
//  per output position (the first float4 plane of the output records): {alpha, beta_bar on beta_1,
//      beta_bar on I*, z} of the current iterate, written by the row pass (alpha also by k_sp_prep);
//  per input position, two float4 planes (st.spin): {x, tau+, l, u} for W > 0 and {x, tau-, u, l}
//      for W < 0, i.e. {x, threshold, Lcheck, Ucheck} for the sign of the taps that read it.
__device__ __forceinline__ float4* sp_orec(const DNet& net, const DState& st, const DLayer& L, int s, int i) {
    return arec_planes(net, st, L, s) + arec_pos(L, i);
}
// the W > 0 plane of layer L (the W < 0 plane follows, xpos float4 later): in float4 units a
// layer takes 2 xpos, as it takes 2 xpos floats in the Active Set input records
__device__ __forceinline__ float4* sp_iplane(const DNet& net, const DState& st, const DLayer& L, int s) {
    return st.spin + (size_t)s * net.XT + (size_t)L.xo;
}

// Phase A epilogue for input j of layer L (k = li + 1, m = k - 1): f_m from acc = (W_k^T alpha_k)[j]
// (Sec. 5.1), the primal conditional gradient (eqs. 7-8 with B = E), the bound terms, and the
// records of input j for the row pass: the thresholds of the oracle eq. (3) at the primal iterate
// x (buffer cur), rounded up to float32 (cb_tau_up) so that the row pass's compares are exact.
// init != 0 also starts the primal iterate at the conditional gradient.
__device__ __forceinline__ void sp_phaseA_epilogue(const DNet& net, const DState& st, const DLayer& L, int k,
                                                   int s, int j, float acc, int cur, int init) {
    const int m = k - 1;
    const size_t NT = net.NT, NH = net.NH;
    const size_t xo = (size_t)s * NT + L.in_off + j;
    float f = k <= net.n - 1 ? st.P[xo] - acc : -net.Wout[(size_t)s * L.n_in + j];
    const float lo = st.lo[xo], hi = st.hi[xo];
    double term = 0.0;
    if (m >= 1) {
        const size_t h = (size_t)s * NH + L.h_in + j;
        f += st.alpha[h] - st.Sb[h];
        const float G = st.G[h];
        const bool z = G >= 0.f;
        st.zbar[h] = z;
        if (init) st.spz[cur][h] = z ? 1.f : 0.f;
        term = (double)net.L[m - 1].b[j] * st.alpha[h] + (double)st.C[h] - (z ? (double)G : 0.0);
    }
    const float xb = f >= 0.f ? hi : lo;
    st.xbar[xo] = xb;
    term -= (double)f * xb;
    st.terms[xo] = term;
    if (net.ball && L.in_off == 0) st.fval[xo] = f;   // for the ellipsoid vertex (k_ball_sp)
    const float x = init ? xb : st.spx[cur][xo];
    if (init) st.spx[cur][xo] = xb;
    if (k <= net.n - 1) {
        float tp = -INFINITY, tn = -INFINITY;
        if (lo != hi) {
            tp = cb_tau_up(x, lo, lo, hi);
            tn = cb_tau_up(hi, x, lo, hi);
        }
        float4* r = sp_iplane(net, st, L, s) + xin_pos(L, j);
        r[0] = make_float4(x, tp, lo, hi);
        r[L.xpos] = make_float4(x, tn, hi, lo);
    }
}

// Phase B of one row after its sums (a0 = W x, A = (W o I*) x, Lam, Mu the row sums of the oracle mask,
// nout its unselected free inputs): conditional gradients alpha_bar (eq. 11) and beta_bar (eq. 12), the
// convex combination of alpha, Sb, G, C at iteration t, and the output record. h: the row's index in a hidden
// vector, z its primal value (worked out again here, the lane teams' kernel took 64 registers instead of 48: 25
// iterations on the Wide conv net's nine properties 1500 us instead of 1473).
__device__ __forceinline__ void sp_rowB_unit(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int s,
                                             int i, size_t h, int t, float z, float a0, float A, float Lam, float Mu, int nout) {
    const int cur = t & 1;
    const size_t NT = net.NT;
    // a row selecting none or all of its free inputs is the all-zero / all-ones constraint, a
    // looser copy of beta_0 / beta_1: it does not compete in the choice of eq. (12)
    const bool degenerate = nout == 0 || nout == st.nfree[h];
    const float gamma = 1.f / ((float)t + sc.gamma0);
    const float bi = L.b[i];
    const float xhat = a0 + bi;
    const float x = st.spx[cur][(size_t)s * NT + L.out_off + i];
    const float uh = st.uhat[h], lh = st.lhat[h];
    const float abar = (xhat - x >= 0.f) ? st.mua[h] : 0.f;
    const float v0 = x - z * uh;
    const float v1 = x - xhat + (1.f - z) * lh;
    const float vI = x - A + (1.f - z) * Lam - z * (bi + Mu);
    int sel = 0;
    float vm = v0;
    if (v1 > vm) { sel = 1; vm = v1; }
    if (!degenerate && vI > vm) { sel = 2; vm = vI; }
    const bool on = vm >= 0.f;
    const float bb = on ? st.mub[h] : 0.f;
    const float gsel = sel == 0 ? uh : (sel == 1 ? lh : Lam + Mu + bi);
    const float csel = sel == 0 ? 0.f : (sel == 1 ? lh - bi : Lam);
    const float om = 1.f - gamma;
    const float an = om * st.alpha[h] + gamma * abar;
    st.alpha[h] = an;
    st.Sb[h] = om * st.Sb[h] + gamma * bb;
    st.G[h] = om * st.G[h] + gamma * (bb * gsel);
    st.C[h] = om * st.C[h] + gamma * (bb * csel);
    st.sel[h] = on ? (uint8_t)sel : (uint8_t)3;
    *sp_orec(net, st, L, s, i) = make_float4(an, sel == 1 ? bb : 0.f, sel == 2 ? bb : 0.f, z);
}

// Phase C of one input after its sums at iteration t, fused with phase A of the next (k_sp_colCA_t): the
// convex combination of P_k (accC the masked backward product of the chosen masks) and of the primal
// iterate into the other buffer, then phase A there (accA = (W^T alpha)[j]).
__device__ __forceinline__ void sp_colC_unit(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int k,
                                             int s, int j, int t, float accC, float accA) {
    const int cur = t & 1, nxt = cur ^ 1;
    const float gamma = 1.f / ((float)t + sc.gamma0);
    const float om = 1.f - gamma;
    const size_t xo = (size_t)s * net.NT + L.in_off + j;
    if (k <= net.n - 1) st.P[xo] = om * st.P[xo] + gamma * accC;
    st.spx[nxt][xo] = om * st.spx[cur][xo] + gamma * st.xbar[xo];
    if (k >= 2) {
        const size_t hh = (size_t)s * net.NH + L.h_in + j;
        st.spz[nxt][hh] = om * st.spz[cur][hh] + gamma * (st.zbar[hh] ? 1.f : 0.f);
    }
    sp_phaseA_epilogue(net, st, L, k, s, j, accA, nxt, 0);
}

// Primal initialisation (App. C.2), one row after its sum a0 = W x: the inner maximisers at (x, z); returns
// alpha* - beta_1*, the row's entry of the col pass.
__device__ __forceinline__ float spi_row_unit(const DNet& net, const DState& st, const DLayer& L, int s, int i, int cur,
                                              float a0) {
    const size_t h = (size_t)s * net.NH + L.h_out + i;
    const float xhat = a0 + L.b[i];
    const float x = st.spx[cur][(size_t)s * net.NT + L.out_off + i];
    const float z = st.spz[cur][h];
    const float ab = (xhat - x >= 0.f) ? st.mua[h] : 0.f;
    const float v0 = x - z * st.uhat[h];
    const float v1 = x - xhat + (1.f - z) * st.lhat[h];
    const bool on = fmaxf(v0, v1) >= 0.f;
    const bool p0 = v0 >= v1;
    const float b0 = (on && p0) ? st.mub[h] : 0.f;
    const float b1 = (on && !p0) ? st.mub[h] : 0.f;
    st.ab[h] = ab;
    st.b0i[h] = b0;
    st.b1i[h] = b1;
    return ab - b1;
}

// Primal initialisation, one input after its sum acc = (W^T (alpha* - beta_1*))[j]: one step of x_m and z_m,
// projected on the boxes (over an ellipsoid, k_ball_retract brings x_0 back into it); returns the new x.
__device__ __forceinline__ float spi_col_unit(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int k,
                                              int s, int j, int step, float acc) {
    const int cur = st.ctr[1] & 1;
    const float eta = sc.sp_lr0 + (sc.sp_lr1 - sc.sp_lr0) * (float)step / (float)max(1, sc.sp_init_steps - 1);
    float f = k <= net.n - 1 ? -acc : -net.Wout[(size_t)s * L.n_in + j];
    const size_t xo = (size_t)s * net.NT + L.in_off + j;
    if (k >= 2) {
        const size_t h = (size_t)s * net.NH + L.h_in + j;
        f += st.ab[h] - st.b0i[h] - st.b1i[h];
        const float g = st.b0i[h] * st.uhat[h] + st.b1i[h] * st.lhat[h];
        st.spz[cur][h] = fminf(fmaxf(st.spz[cur][h] + eta * g, 0.f), 1.f);
    }
    float x = st.spx[cur][xo] + eta * f;
    if (!(net.ball && L.in_off == 0)) x = fminf(fmaxf(x, st.lo[xo]), st.hi[xo]);
    st.spx[cur][xo] = x;
    return x;
}

}  // namespace cb
