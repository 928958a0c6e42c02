// The BF16 form's per-neuron passes, four neighbouring neurons per thread.
//
// The passes stream the duals, moments, slots and products (about 430 bytes per hidden neuron and box, 27 GB
// a pass pair at 1024 conv4 boxes) and are bound by memory in the end, but one neuron per thread spent 1200
// instructions a neuron on 4-byte copies, 64-bit addresses and 2-byte stores: issue 51 to 64% active, DRAM
// 39 to 59%. Here every vector is read and written 16 bytes at a time (the snapshot bytes 4), and a conv
// layer's bf16 operand planes are put together from two staged words per position pair.
//
// A layer takes these kernels where the offsets of its vectors and its positions are multiples of four
// (bf_vec_row, bf_vec_col); the others keep one neuron per thread (cb_team.cuh). The arithmetic per
// neuron is the same, in the same order. At 128 conv4 boxes and five slots the col pass takes 256 us (395 by
// one neuron per thread; 59% of the DRAM rate, 0.32 of the instructions), the row pass 380 us (471; 73%).
#include <cuda_bf16.h>

#include "cb_vec.cuh"

namespace cb {

namespace {

constexpr int VP = 128;   // positions of a conv block (8 channels x 128 positions, four per thread)

__device__ __forceinline__ int vseg_of(const VSegs& v, int blk) {
    int q = 0;
    while (q + 1 < v.n && blk >= v.start[q + 1]) ++q;
    return q;
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void get(const float4& v, float (&o)[4]) {
    o[0] = v.x;
    o[1] = v.y;
    o[2] = v.z;
    o[3] = v.w;
}
__device__ __forceinline__ unsigned ld_b4(const uint8_t* p) { return *reinterpret_cast<const unsigned*>(p); }
__device__ __forceinline__ void st_b4(uint8_t* p, unsigned v) { *reinterpret_cast<unsigned*>(p) = v; }
__device__ __forceinline__ uint16_t bf(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }
__device__ __forceinline__ unsigned bf2(float a, float b) { return bf(a) | ((unsigned)bf(b) << 16); }

// A thread's four units: subproblem, first neuron (and, conv, channel, position); none: s < 0.
struct Quad {
    int s, i, c, p;
};
__device__ __forceinline__ Quad quad_of(int blk, bool conv, int C, int P, int S) {
    Quad q{-1, 0, 0, 0};
    if (conv) {
        const int ncb = (C + 7) >> 3, npb = (P + VP - 1) / VP;
        const int s = blk / (ncb * npb), rem = blk - s * (ncb * npb);
        const int cb = rem / npb, pb = rem - cb * npb;
        q.c = cb * 8 + (threadIdx.x >> 5);
        q.p = pb * VP + (threadIdx.x & 31) * 4;
        if (q.c < C && q.p < P) q.s = s;
        q.i = q.c * P + q.p;
    } else {
        const long long u = (long long)blk * CB_THREADS + threadIdx.x;
        const int n4 = C >> 2, s = (int)(u / n4);
        q.i = q.c = (int)(u - (long long)s * n4) * 4;
        if (s < S) q.s = s;
    }
    return q;
}

// Two neighbouring positions' 16-byte pieces of a channels-last plane from eight channels' words (each
// the two positions' bf16 values).
__device__ __forceinline__ void pieces(const unsigned (&w)[8], uint4& a, uint4& b) {
    a = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410), __byte_perm(w[4], w[5], 0x5410),
                   __byte_perm(w[6], w[7], 0x5410));
    b = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632), __byte_perm(w[4], w[5], 0x7632),
                   __byte_perm(w[6], w[7], 0x7632));
}

// ---------------------------------------------------------------- row pass
template <int NS, bool ADD>
__device__ __forceinline__ void row_quad(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int li,
                                         const StepNow& sp, const Quad& q, uint16_t (*stage)[8][VP]) {
    const size_t NH = net.NH;
    const int s = q.s, P = L.ho * L.wo;
    const size_t h = (size_t)s * NH + L.h_out + q.i, hs0 = (size_t)s * net.cap * NH + L.h_out + q.i;
    const int bn = (sp.nadd_before + (sp.b_new >= 0 ? 1 : 0)) & 1;
    const int cap_s = st.caps[s];
    const int newb = (ADD && sp.b_new < cap_s) ? sp.b_new : -1;
    const int nsl = min(sp.nadd_before + (sp.b_new >= 0 ? 1 : 0), cap_s);
    const BfLayer& B = net.bf[li];
    const size_t slot = (size_t)net.S * P * L.co;
    const float* d = B.Drow + ((size_t)s * L.co + q.c) * P + q.p;
    float acc[1 + NS][4], x[4], z[4], bi[4];
    {
        float4 t[1 + NS];
#pragma unroll
        for (int b = 0; b <= NS; ++b) t[b] = ld4(d + b * slot);
#pragma unroll
        for (int b = 0; b <= NS; ++b) get(t[b], acc[b]);
    }
    const unsigned zs4 = ld_b4(st.zsnap[bn] + h), z4 = ld_b4(st.zcur + h);
    get(ld4(st.xval + (size_t)s * net.NT + L.out_off + q.i), x);
    get(ld4(L.b + q.i), bi);
    float con[4];
    {
        const float* src[9] = {st.alpha, st.beta0, st.beta1, st.ma, st.m0, st.m1, st.va, st.v0, st.v1};
        float4 t[11];
#pragma unroll
        for (int v = 0; v < 9; ++v) t[v] = ld4(src[v] + h);
        t[9] = ld4(st.uhat + h);
        t[10] = ld4(st.lhat + h);
        float th[9][4], uh[4], lh[4];
#pragma unroll
        for (int v = 0; v < 9; ++v) get(t[v], th[v]);
        get(t[9], uh);
        get(t[10], lh);
        const float2 ib = cb_bias(st);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            z[u] = (z4 >> (8 * u)) & 255u ? 1.f : 0.f;
            const float xhat = acc[0][u] + bi[u];
            const float g[3] = {xhat - x[u], x[u] - z[u] * uh[u], x[u] - xhat + (1.f - z[u]) * lh[u]};
#pragma unroll
            for (int v = 0; v < 3; ++v) th[v][u] = adam_step(th[v][u], th[3 + v][u], th[6 + v][u], g[v], sp.lr, ib.x, ib.y, sc);
            con[u] = th[2][u] - th[0][u];
        }
#pragma unroll
        for (int v = 0; v < 9; ++v) st4(const_cast<float*>(src[v]) + h, th[v]);
    }
    // plane e of the next col products' operands: staged (conv), or stored at once (linear)
    auto put = [&](int e, const float (&v)[4]) {
        const uint2 w = make_uint2(bf2(v[0], v[1]), bf2(v[2], v[3]));
        if (stage) {
            *reinterpret_cast<uint2*>(&stage[e][threadIdx.x >> 5][(threadIdx.x & 31) * 4]) = w;
        } else {
            *reinterpret_cast<uint2*>(B.R + ((long long)e * net.S + s) * B.PR + q.i) = w;
        }
    };
#pragma unroll
    for (int b = 0; b < NS; ++b) {
        float nv[4] = {0.f, 0.f, 0.f, 0.f};
        if (b < nsl) {
            const size_t hs = hs0 + (size_t)b * NH;
            float bs[4], ms[4], vs[4], lam[4], kap[4];
            const float4 t0 = ld4(st.bs + hs), t1 = ld4(st.ms + hs), t2 = ld4(st.vs + hs);
            if (ADD && b == newb) {
                float lz[4], uz[4];
                get(ld4(st.lz + h), lz);
                const bool in = net.ball && L.in_off == 0;
                get(in ? ld4(st.uz + h) : make_float4(0.f, 0.f, 0.f, 0.f), uz);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool zb = (zs4 >> (8 * u + b)) & 1u;
                    lam[u] = zb ? lz[u] : acc[1 + b][u];
                    // kappa = lambda + sum W (1 - I) Ucheck + b: W x* + b at box vertices; over interior
                    // inputs (layer 0, ellipsoid) the z = 0 mask holds fixed inputs only
                    kap[u] = zb ? lz[u] + bi[u] : (in ? uz[u] + bi[u] : acc[0][u] + bi[u]);
                }
                st4(st.lam + hs, lam);
                st4(st.kap + hs, kap);
            } else {
                const float4 t3 = ld4(st.lam + hs), t4 = ld4(st.kap + hs);
                get(t3, lam);
                get(t4, kap);
            }
            get(t0, bs);
            get(t1, ms);
            get(t2, vs);
            const float2 sib = cb_slot_bias(st, b);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool zb = (zs4 >> (8 * u + b)) & 1u;
                const float prod = zb ? acc[0][u] : acc[1 + b][u];
                const float gb = x[u] - prod + lam[u] * (1.f - z[u]) - z[u] * (kap[u] - lam[u]);
                bs[u] = adam_step(bs[u], ms[u], vs[u], gb, sp.lr, sib.x, sib.y, sc);
                if (zb) con[u] += bs[u];
                nv[u] = zb ? 0.f : bs[u];
            }
            st4(st.bs + hs, bs);
            st4(st.ms + hs, ms);
            st4(st.vs + hs, vs);
        }
        put(1 + b, nv);
    }
    put(0, con);
}

template <int NS, bool ADD>
__device__ __forceinline__ void row_block(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int li,
                                          const StepNow& sp, int blk, char* smem) {
    const bool conv = L.kind == 1;
    const int P = L.ho * L.wo;
    const Quad q = quad_of(blk, conv, conv ? L.co : L.n_out, P, net.S);
    uint16_t(*stage)[8][VP] = conv ? reinterpret_cast<uint16_t(*)[8][VP]>(smem) : nullptr;
    if (q.s >= 0) {
        row_quad<NS, ADD>(net, st, sc, L, li, sp, q, stage);
    } else if (conv) {   // no unit here (channel padding): zeros
#pragma unroll
        for (int e = 0; e <= NS; ++e)
            *reinterpret_cast<uint2*>(&stage[e][threadIdx.x >> 5][(threadIdx.x & 31) * 4]) = make_uint2(0u, 0u);
    }
    if (!conv) return;
    __syncthreads();
    const BfLayer& B = net.bf[li];
    const int ncb = (L.co + 7) >> 3, npb = (P + VP - 1) / VP;
    const int ts = blk / (ncb * npb), rem = blk - ts * (ncb * npb), cb = rem / npb, pb = rem - cb * npb;
    const int pp = threadIdx.x & 63, p = pb * VP + 2 * pp;   // P is a multiple of 4: both positions or neither
    if (p >= P) return;
    const int y0 = p / L.wo, x0 = p - y0 * L.wo, y1 = (p + 1) / L.wo, x1 = p + 1 - y1 * L.wo;
    const long long o0 = ((long long)(y0 + L.hl) * L.Wpo + (x0 + L.wl)) * B.Cop + cb * 8;
    const long long o1 = ((long long)(y1 + L.hl) * L.Wpo + (x1 + L.wl)) * B.Cop + cb * 8;
    for (int e = threadIdx.x >> 6; e <= NS; e += CB_THREADS / 64) {
        unsigned w[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) w[c] = *reinterpret_cast<const unsigned*>(&stage[e][c][2 * pp]);
        uint4 a, b;
        pieces(w, a, b);
        uint16_t* R = B.R + ((long long)e * net.S + ts) * B.PR;
        *reinterpret_cast<uint4*>(R + o0) = a;
        *reinterpret_cast<uint4*>(R + o1) = b;
    }
}

__global__ void __launch_bounds__(CB_THREADS, 2) k_bf_rowB(DNet net, DState st, DSched sc, const __grid_constant__ VSegs v) {
    extern __shared__ __align__(16) char vec_smem[];
    const int q = vseg_of(v, blockIdx.x), li = v.layer[q], blk = blockIdx.x - v.start[q];
    const DLayer& L = net.L[li];
    const StepNow sp = cb_step(st);
    const int ns = min(sp.nadd_before + (sp.b_new >= 0 ? 1 : 0), sc.maxcut);
    if (sp.b_new >= 0) {
        switch (ns) {
            case 1: row_block<1, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 2: row_block<2, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 3: row_block<3, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 4: row_block<4, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 5: row_block<5, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 6: row_block<6, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 7: row_block<7, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
            default: row_block<8, true>(net, st, sc, L, li, sp, blk, vec_smem); break;
        }
    } else {
        switch (ns) {
            case 0: row_block<0, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 1: row_block<1, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 2: row_block<2, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 3: row_block<3, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 4: row_block<4, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 5: row_block<5, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 6: row_block<6, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            case 7: row_block<7, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
            default: row_block<8, false>(net, st, sc, L, li, sp, blk, vec_smem); break;
        }
    }
}

// ---------------------------------------------------------------- col pass
// The products of slot b and sign sg for four neighbouring inputs of a conv layer or four of a linear one.
struct ColProducts {
    const float* d[2];      // of even and odd positions (stride 2); of all (stride 1, linear)
    size_t slot[2], neg[2];
    bool two;
    __device__ __forceinline__ void init(const DNet& net, const DLayer& L, const BfLayer& B, const Quad& q) {
        two = L.kind == 1 && L.st == 2;
        if (L.kind == 0) {
            slot[0] = (size_t)net.S * 2 * L.ci;
            neg[0] = L.ci;
            d[0] = B.Dcol[0] + (size_t)q.s * 2 * L.ci + q.c;
            return;
        }
        const int y = q.p / L.wi, x = q.p - y * L.wi;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (e && !two) return;
            const int ty = y + L.pd, tx = x + e + L.pd;
            const int Y0 = two ? ty >> 1 : ty, X0 = two ? tx >> 1 : tx;
            const int ph = two ? (ty & 1) * 2 + (tx & 1) : 0;
            const int P = B.nY[ph] * B.nX[ph];
            slot[e] = (size_t)net.S * 2 * L.ci * P;
            neg[e] = (size_t)L.ci * P;
            d[e] = B.Dcol[ph] + ((size_t)q.s * 2 * L.ci + q.c) * P + (Y0 - B.Y0a[ph]) * B.nX[ph] + (X0 - B.X0a[ph]);
        }
    }
    __device__ __forceinline__ float4 load(int b, int sg) const {
        if (!two) return ld4(d[0] + b * slot[0] + sg * neg[0]);
        const float2 e = *reinterpret_cast<const float2*>(d[0] + b * slot[0] + sg * neg[0]);
        const float2 o = *reinterpret_cast<const float2*>(d[1] + b * slot[1] + sg * neg[1]);
        return make_float4(e.x, o.x, e.y, o.y);
    }
};

template <int NS>
__device__ __forceinline__ void col_quad(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int k,
                                         const StepNow& sp, const Quad& q, int mode, uint16_t (*sx)[VP],
                                         uint16_t (*sb_)[VP]) {
    const size_t NT = net.NT, NH = net.NH;
    const int s = q.s, j = q.i;
    const bool want_terms = mode != 2, prod = k <= net.n - 1;
    const int cap_s = st.caps[s];
    const int nsl = min(sp.nadd_before, cap_s), bo = sp.nadd_before & 1;
    const bool add_iter = (mode != 1) && sp.b_new >= 0;
    const bool add = add_iter && sp.b_new < cap_s;
    const size_t xo = (size_t)s * NT + L.in_off + j;
    const size_t h = (size_t)s * NH + L.h_in + j, hs = (size_t)s * net.cap * NH + L.h_in + j;
    const unsigned xs4 = ld_b4(st.xsnap[bo] + xo), fx4 = ld_b4(st.efix + xo);
    float lo[4], hi[4], f[4];
    float4 tl = ld4(st.lo + xo), thi = ld4(st.hi + xo);
    unsigned pm[4], qm[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) slot_bits(net, L, (xs4 >> (8 * u)) & 255u, (fx4 >> (8 * u)) & 255u, pm[u], qm[u]);
    if (prod) {
        ColProducts cp;
        cp.init(net, L, net.bf[k - 1], q);
        float4 t[2 * (1 + NS)];
#pragma unroll
        for (int b = 0; b <= NS; ++b) {
            t[2 * b] = cp.load(b, 0);
            t[2 * b + 1] = cp.load(b, 1);
        }
        float a[4], c[4];
        get(t[0], a);
        get(t[1], c);
#pragma unroll
        for (int u = 0; u < 4; ++u) f[u] = a[u] + c[u];
#pragma unroll
        for (int b = 0; b < NS; ++b) {
            get(t[2 + 2 * b], a);
            get(t[3 + 2 * b], c);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if ((pm[u] >> b) & 1u) f[u] += a[u];
                if ((qm[u] >> b) & 1u) f[u] += c[u];
            }
        }
    } else {
        float w[4];
        get(ld4(net.Wout + (size_t)s * L.n_in + j), w);
#pragma unroll
        for (int u = 0; u < 4; ++u) f[u] = -w[u];
    }
    get(tl, lo);
    get(thi, hi);
    double term[4] = {0.0, 0.0, 0.0, 0.0};
    if (k >= 2) {
        float al[4], b0[4], b1[4], uh[4], lh[4], bs[NS > 0 ? NS : 1][4], kp[NS > 0 ? NS : 1][4];
        {
            const float4 t0 = ld4(st.alpha + h), t1 = ld4(st.beta0 + h), t2 = ld4(st.beta1 + h), t3 = ld4(st.uhat + h),
                         t4 = ld4(st.lhat + h);
            float4 tb[NS > 0 ? NS : 1], tk[NS > 0 ? NS : 1];
#pragma unroll
            for (int b = 0; b < NS; ++b) {
                tb[b] = tk[b] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (b < nsl) {
                    tb[b] = ld4(st.bs + hs + (size_t)b * NH);
                    tk[b] = ld4(st.kap + hs + (size_t)b * NH);
                }
            }
            get(t0, al);
            get(t1, b0);
            get(t2, b1);
            get(t3, uh);
            get(t4, lh);
#pragma unroll
            for (int b = 0; b < NS; ++b) {
                get(tb[b], bs[b]);
                get(tk[b], kp[b]);
            }
        }
        unsigned z4 = 0u, zn = 0u;
        const unsigned zo = add_iter ? ld_b4(st.zsnap[bo] + h) : 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float sb = 0.f, gk = b0[u] * uh[u] + b1[u] * lh[u];
#pragma unroll
            for (int b = 0; b < NS; ++b)
                if (b < nsl) {
                    sb += bs[b][u];
                    gk += bs[b][u] * kp[b][u];
                }
            f[u] += al[u] - b0[u] - b1[u] - sb;
            const bool z = gk >= 0.f;
            z4 |= (z ? 1u : 0u) << (8 * u);
            zn |= (((zo >> (8 * u)) & 255u) | ((add && z) ? (1u << sp.b_new) : 0u)) << (8 * u);
            if (want_terms) {
                const float bm = net.L[k - 2].b[j + u];
                double ct = 0.0;
#pragma unroll
                for (int b = 0; b < NS; ++b)
                    if (b < nsl) ct += (double)bs[b][u] * st.lam[hs + (size_t)b * NH + u];
                term[u] = (double)bm * al[u] + (double)b1[u] * ((double)lh[u] - bm) + ct - (z ? (double)gk : 0.0);
            }
        }
        st_b4(st.zcur + h, z4);
        if (add_iter) st_b4(st.zsnap[bo ^ 1] + h, zn);
    }
    float xv[4];
    unsigned xn = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const bool up = f[u] >= 0.f;
        xv[u] = up ? hi[u] : lo[u];
        if (want_terms) st.terms[xo + u] = term[u] - (double)f[u] * xv[u];
        xn |= (((xs4 >> (8 * u)) & 255u) | ((add && up) ? (1u << sp.b_new) : 0u)) << (8 * u);
    }
    st4(st.xval + xo, xv);
    if (mode == 1 || net.ball) st4(st.fval + xo, f);
    if (add_iter) st_b4(st.xsnap[bo ^ 1] + xo, xn);
    if (!prod) return;
    // the row products' operands: x*, and where each slot's masks keep it under positive and negative weights
    unsigned mp[4], mq[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const unsigned xs = (xn >> (8 * u)) & 255u, fx = (fx4 >> (8 * u)) & 255u ? 255u : 0u;
        mp[u] = ((~xs) & 255u) | fx;
        mq[u] = xs | fx;
    }
    if (sx) {
        const int w = threadIdx.x >> 5, l = (threadIdx.x & 31) * 4;
        *reinterpret_cast<uint2*>(&sx[w][l]) = make_uint2(bf2(xv[0], xv[1]), bf2(xv[2], xv[3]));
        *reinterpret_cast<uint2*>(&sb_[w][l]) = make_uint2(mp[0] | mq[0] << 8 | mp[1] << 16 | mq[1] << 24,
                                                           mp[2] | mq[2] << 8 | mp[3] << 16 | mq[3] << 24);
    } else {
        const BfLayer& B = net.bf[k - 1];
        const int nt = NS + (add_iter ? 1 : 0);
        for (int t = 0; t <= nt; ++t) {
            float v[4], n[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                v[u] = t == 0 || ((mp[u] >> (t - 1)) & 1u) ? xv[u] : 0.f;
                n[u] = t == 0 || ((mq[u] >> (t - 1)) & 1u) ? xv[u] : 0.f;
            }
            uint16_t* X = B.X + ((long long)t * net.S + s) * 2 * B.PX + j;
            *reinterpret_cast<uint2*>(X) = make_uint2(bf2(v[0], v[1]), bf2(v[2], v[3]));
            *reinterpret_cast<uint2*>(X + B.PX) = make_uint2(bf2(n[0], n[1]), bf2(n[2], n[3]));
        }
    }
    // the new slot's float32 lambda, kappa (k_slot_sums_t after the row pass) walk these records
    if (add_iter)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            slot_rec_plane(net, st, L, s)[xin_pos(L, j + u)] =
                slot_rec(lo[u], hi[u], (xn >> (8 * u)) & 255u, (fx4 >> (8 * u)) & 255u, net.ball && L.in_off == 0);
}

template <int NS>
__device__ __forceinline__ void col_block(const DNet& net, const DState& st, const DSched& sc, const DLayer& L, int li,
                                          const StepNow& sp, int blk, int mode, uint16_t (*sx)[VP], uint16_t (*sb)[VP]) {
    const bool conv = L.kind == 1;
    const int P = L.hi * L.wi;
    const Quad q = quad_of(blk, conv, conv ? L.ci : L.n_in, P, net.S);
    if (q.s >= 0) {
        col_quad<NS>(net, st, sc, L, li + 1, sp, q, mode, conv ? sx : nullptr, sb);
    } else if (conv) {
        const int w = threadIdx.x >> 5, l = (threadIdx.x & 31) * 4;
        *reinterpret_cast<uint2*>(&sx[w][l]) = make_uint2(0u, 0u);
        *reinterpret_cast<uint2*>(&sb[w][l]) = make_uint2(0u, 0u);
    }
    if (!conv) return;
    __syncthreads();
    const BfLayer& B = net.bf[li];
    const int ncb = (L.ci + 7) >> 3, npb = (P + VP - 1) / VP;
    const int ts = blk / (ncb * npb), rem = blk - ts * (ncb * npb), cb = rem / npb, pb = rem - cb * npb;
    const int pp = threadIdx.x & 63, p = pb * VP + 2 * pp;
    if (p >= P) return;
    const int y = p / L.wi, x = p - y * L.wi;   // wi is a multiple of 4: both positions in one row
    const long long o0 = ((long long)(y + L.pd) * L.Wp + (x + L.pd)) * B.Cip + cb * 8, o1 = o0 + B.Cip;
    unsigned xw[8], bw[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        xw[c] = *reinterpret_cast<const unsigned*>(&sx[c][2 * pp]);
        bw[c] = *reinterpret_cast<const unsigned*>(&sb[c][2 * pp]);
    }
    const int nt = NS + (mode != 1 && sp.b_new >= 0 ? 1 : 0);
    for (int e = threadIdx.x >> 6; e < 2 * (1 + nt); e += CB_THREADS / 64) {
        const int t = e >> 1, sg = e & 1;
        unsigned w[8];
        if (t == 0) {
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = xw[c];
        } else {
            const int sh = t - 1 + 8 * sg;
#pragma unroll
            for (int c = 0; c < 8; ++c) w[c] = xw[c] & (((bw[c] >> sh) & 0x00010001u) * 0xFFFFu);
        }
        uint4 a, b;
        pieces(w, a, b);
        uint16_t* X = B.X + (((long long)t * net.S + ts) * 2 + sg) * B.PX;
        *reinterpret_cast<uint4*>(X + o0) = a;
        *reinterpret_cast<uint4*>(X + o1) = b;
    }
}

__global__ void __launch_bounds__(CB_THREADS, 2) k_bf_colA(DNet net, DState st, DSched sc, const __grid_constant__ VSegs v,
                                                           int mode) {
    __shared__ __align__(16) uint16_t sx[8][VP], sb[8][VP];
    const int q = vseg_of(v, blockIdx.x), li = v.layer[q], blk = blockIdx.x - v.start[q];
    const DLayer& L = net.L[li];
    const StepNow sp = cb_step(st);
    switch (min(sp.nadd_before, sc.maxcut)) {
        case 0: col_block<0>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 1: col_block<1>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 2: col_block<2>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 3: col_block<3>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 4: col_block<4>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 5: col_block<5>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 6: col_block<6>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        case 7: col_block<7>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
        default: col_block<8>(net, st, sc, L, li, sp, blk, mode, sx, sb); break;
    }
}

}  // namespace

// Offsets of a layer's vectors, subproblems and positions that are multiples of four.
bool bf_vec_row(const DNet& D, int li) {
    const DLayer& L = D.L[li];
    return D.NT % 4 == 0 && D.NH % 4 == 0 && L.out_off % 4 == 0 && L.h_out % 4 == 0 &&
           (L.kind == 0 ? L.n_out % 4 == 0 : (L.ho * L.wo) % 4 == 0);
}
bool bf_vec_col(const DNet& D, int li) {
    const DLayer& L = D.L[li];
    if (D.NT % 4 || D.NH % 4 || L.in_off % 4 || (li > 0 && L.h_in % 4)) return false;
    return L.kind == 0 ? L.n_in % 4 == 0 : L.wi % 4 == 0 && L.st <= 2;
}
int bf_vec_blocks(const DNet& D, int li, bool col) {
    const DLayer& L = D.L[li];
    if (L.kind == 0) return (int)(((long long)D.S * (col ? L.n_in : L.n_out) / 4 + CB_THREADS - 1) / CB_THREADS);
    const int C = col ? L.ci : L.co, P = col ? L.hi * L.wi : L.ho * L.wo;
    return D.S * ((C + 7) / 8) * ((P + VP - 1) / VP);
}

void launch_bf_colA(int blocks, const DNet& net, const DState& st, const DSched& sc, const VSegs& v, int mode, cudaStream_t s) {
    k_bf_colA<<<blocks, CB_THREADS, 0, s>>>(net, st, sc, v, mode);
}
void launch_bf_rowB(int blocks, const DNet& net, const DState& st, const DSched& sc, const VSegs& v, cudaStream_t s) {
    k_bf_rowB<<<blocks, CB_THREADS, (1 + net.cap) * 8 * VP * (int)sizeof(uint16_t), s>>>(net, st, sc, v);
}

}  // namespace cb
