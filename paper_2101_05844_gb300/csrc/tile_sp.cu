// Interval propagation and Saddle Point passes on tiles (cb_tile.cuh).
#include <algorithm>

#include "cb_tile.cuh"

namespace cb {

// ---------------------------------------------------------------- interval propagation
// Interval propagation (App. E) of one hidden layer on tiles: lhat = W+ l + W- u + b, uhat = W+ u + W- l + b
// by compensated float32 sums, from records {l, u} of the layer's inputs kept in the first Saddle Point input
// plane. A warp per row (k_ibp) reads every weight and bound of a row from L1 for that row alone: 26.6 ms for
// 256 conv4 boxes, where the sums' 20 operations per tap take about 1.6 ms at the float32 rate. On tiles 4.7
// ms (the layers of few tiles split over their sources, tl_ibp_splits).
//
// Accuracy: a pair (CompSum) loses about k 2^-48 over k terms, so one pair over a whole row is worse than the
// warp's 32 pairs that meet in float64 (rms over rows of 576 terms 1.1e-15 against 3.4e-16 of the terms'
// magnitudes). A thread's pair therefore ends where a lane's would, after a 32nd of the row, and goes into a
// three-word total (CompTotal): no larger error than the warp's at any of 27 to 8192 terms. That costs 20
// operations per 32nd of a row (4.0 -> 4.7 ms: of the batch's set-up 3.52 -> 4.14, 3.69 with the totals left out).
// Adding into float64 instead asks for 4 G conversions and additions, 6 ms at the nominal float64 rate.
template <int CH>
struct IbpOp : TlOp {
    static constexpr int RB = 8, EB = 0, WB = 4, SWEEPS = 1;
    const float4* src;      // the layer's input records of subproblem 0
    size_t ss;              // records per subproblem
    CompSum a[CH], c[CH];
    CompTotal ta[CH], tc[CH];
    int nf[CH];
    int part, room;         // taps of a pair; taps the present one has left
    __device__ __forceinline__ void copy(uint32_t buf, int, int slot, int s, int i) const {
        tl_copy<8>(buf + slot * 8, src + (size_t)s * ss + i);
    }
    __device__ __forceinline__ const char* weights(const TlSeg& g) const { return reinterpret_cast<const char*>(g.w); }
    __device__ __forceinline__ void begin(int) {
#pragma unroll
        for (int k = 0; k < CH; ++k) nf[k] = 0;
        room = part;
    }
    __device__ __forceinline__ bool singly() const { return part < 4; }
    __device__ __forceinline__ void taken(int n) {
        room -= n;
        if (room < (part < 4 ? 1 : 4)) {
            end(0);
            room = part;
        }
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int, int slot, const char* w) {
        const float2 r = *reinterpret_cast<const float2*>(rec + slot * 8);
        const int free = r.x != r.y ? 1 : 0;
#pragma unroll
        for (int k = 0; k < CH; k += 4) {
            const float4 q = *reinterpret_cast<const float4*>(w + 4 * k);
            const float v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool pos = v[e] >= 0.f;
                a[k + e].add_prod(v[e], pos ? r.x : r.y);
                c[k + e].add_prod(v[e], pos ? r.y : r.x);
                nf[k + e] += v[e] != 0.f ? free : 0;
            }
        }
    }
    __device__ __forceinline__ void end(int) {   // the pairs into the totals
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            ta[k].add(a[k]);
            tc[k].add(c[k]);
            a[k] = c[k] = CompSum{};
        }
    }
};

// Layer k's records {l, u} of its inputs from the input box (k = 0; later layers' are written by the
// layer before).
__global__ void k_ibp_box(DNet net, DState st) {
    const DLayer& L = net.L[0];
    const size_t n = (size_t)net.S * L.n_in;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < n; u += (size_t)gridDim.x * blockDim.x) {
        const int s = (int)(u / L.n_in), j = (int)(u - (size_t)s * L.n_in);
        const size_t xo = (size_t)s * net.NT + j;
        slot_rec_plane(net, st, L, s)[xin_pos(L, j)] = make_float4(st.lo[xo], st.hi[xo], 0.f, 0.f);
    }
}

// One hidden layer: the segment's tiles; the row constants lz, uz and the free counts as k_ibp, the
// post-activation box, and the next layer's input records.
template <int CH>
__device__ __forceinline__ void ibp_tile(const DNet& net, const DState& st, const TlSegs& segs, const TlSeg& g,
                                         const signed char* splits, char* smem) {
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    float* sums = reinterpret_cast<float*>(smem);
    {
        IbpOp<CH> op;
        op.src = slot_rec_plane(net, st, L, 0);
        op.ss = net.XT;
        // a pair takes the terms that a lane of the warp walk takes (conv: rows of kernel columns)
        op.part = max(g.SC * g.kt / 32, L.kw);
        tl_walk(g, t, net.S, smem, op);
        float v[CH][5];
#pragma unroll
        for (int k = 0; k < CH; ++k) {   // the float64 sums as words
            const double a = op.ta[k].total(), c = op.tc[k].total();
            v[k][0] = __int_as_float(__double2loint(a));
            v[k][1] = __int_as_float(__double2hiint(a));
            v[k][2] = __int_as_float(__double2loint(c));
            v[k][3] = __int_as_float(__double2hiint(c));
            v[k][4] = __int_as_float(op.nf[k]);
        }
        tl_put<5, CH>(g, t, sums, v);
    }
    // the splits' sums of a row are added in float64 by the block that arrives last
    if (g.ks > 1 && !tl_arrive<5>(segs, g, t, sums)) return;
    __syncthreads();
    const int TC = tl_channels(g), row = tl_lanes(g) + 1;
    const float* part = reinterpret_cast<const float*>(tl_partials<5>(segs, g, t));
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        int ch, lane, s, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, s, p) || t.ct * TC + ch >= g.C) continue;
        const int i = (t.ct * TC + ch) * g.P + p, at = ch * row + lane;
        double a = 0.0, c = 0.0;
        int nf = 0;
        if (g.ks == 1) {
            auto val = [&](int e) { return __float_as_int(sums[e * TC * row + at]); };
            a = __hiloint2double(val(1), val(0));
            c = __hiloint2double(val(3), val(2));
            nf = val(4);
        } else {
#pragma unroll 4
            for (int q = 0; q < g.ks; ++q) {
                const float* v = part + q * tl_split(g, 5) + at;
                auto val = [&](int e) { return __float_as_int(__ldcg(v + e * TC * row)); };
                a += __hiloint2double(val(1), val(0));
                c += __hiloint2double(val(3), val(2));
                nf += val(4);
            }
        }
        const size_t h = (size_t)s * net.NH + L.h_out + i;
        st.lz[h] = (float)a;
        st.uz[h] = (float)c;
        st.nfree[h] = nf;
        a += (double)L.b[i];
        c += (double)L.b[i];
        if (splits && a < 0.0 && c > 0.0) {
            if (splits[h] > 0) a = 0.0;
            if (splits[h] < 0) c = 0.0;
        }
        const float lh = __double2float_rd(a), uh = __double2float_ru(c);
        st.lhat[h] = lh;
        st.uhat[h] = uh;
        const float lo = fmaxf(lh, 0.f), hi = fmaxf(uh, 0.f);
        const size_t o = (size_t)s * net.NT + L.out_off + i;
        st.lo[o] = lo;
        st.hi[o] = hi;
        if (g.li + 2 < net.n) {
            const DLayer& N = net.L[g.li + 1];
            slot_rec_plane(net, st, N, s)[xin_pos(N, i)] = make_float4(lo, hi, 0.f, 0.f);
        }
    }
}
__global__ void __launch_bounds__(CB_THREADS, 2) k_ibp_tl(DNet net, DState st, const __grid_constant__ TlSegs segs,
                                                          const signed char* splits) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[0];
    if (g.ch == 8) ibp_tile<8>(net, st, segs, g, splits, tile_smem);
    else ibp_tile<4>(net, st, segs, g, splits, tile_smem);
}

// ---------------------------------------------------------------- Saddle Point
// Phase B (cb_team.cuh: k_sp_rowB_t) on tiles: the oracle mask of eq. (3) by comparing the row's z with the
// threshold of the tap's sign, a few selects per tap and channel; a record {x, tau+, tau-, l, u} is staged
// once per tile where the lane teams loaded 16 bytes per unit and tap. Bound by issue.
template <int CH>
struct SpRowOp : TlOp {
    static constexpr int RB = 20, EB = 0, WB = 4, SWEEPS = 1;
    const float4* src;      // the layer's records of subproblem 0: {x, tau+, l, u}, and xpos on {x, tau-, u, l}
    size_t ss;
    int xpos;
    float z[CH], v[CH][4];  // W x, (W o I) x, Lam, Mu
    int nout[CH];
    __device__ __forceinline__ void copy(uint32_t buf, int nrec, int slot, int s, int i) const {
        const float4* p = src + (size_t)s * ss + i;
        tl_copy<16>(buf + slot * 16, p);
        tl_copy<4>(buf + nrec * 16 + slot * 4, &p[xpos].y);
    }
    __device__ __forceinline__ const char* weights(const TlSeg& g) const { return reinterpret_cast<const char*>(g.w); }
    __device__ __forceinline__ void begin(int) {
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            v[c][0] = v[c][1] = v[c][2] = v[c][3] = 0.f;
            nout[c] = 0;
        }
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int nrec, int slot, const char* w) {
        const float4 r = *reinterpret_cast<const float4*>(rec + slot * 16);
        const float tn = *reinterpret_cast<const float*>(rec + nrec * 16 + slot * 4);
#pragma unroll
        for (int c4 = 0; c4 < CH; c4 += 4) {
            const float4 q = *reinterpret_cast<const float4*>(w + 4 * c4);
            const float wv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = c4 + e;
                const float wt = wv[e], wx = wt * r.x;
                const bool pos = wt > 0.f;
                // I = [z >= threshold] (fixed inputs, padding and zero weights: 1)
                const bool I = z[c] >= (pos ? r.y : tn) || wt == 0.f;
                v[c][0] += wx;
                if (I) {
                    v[c][1] += wx;
                    v[c][2] = fmaf(wt, pos ? r.z : r.w, v[c][2]);
                } else {
                    v[c][3] = fmaf(wt, pos ? r.w : r.z, v[c][3]);
                    ++nout[c];
                }
            }
        }
    }
    __device__ __forceinline__ void end(int) {}
};

template <int CH>
__device__ __forceinline__ void sp_row_tile(const DNet& net, const DState& st, const DSched& sc, const TlSegs& segs,
                                            const TlSeg& g, char* smem) {
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const int it = st.ctr[1], TC = tl_channels(g), row = tl_lanes(g) + 1;
    float* sums = reinterpret_cast<float*>(smem);
    {
        SpRowOp<CH> op;
        op.src = sp_iplane(net, st, L, 0);
        op.ss = net.XT;
        op.xpos = L.xpos;
        int s, p;
        const bool ok = tl_unit(g, t, t.lane, net.S, s, p);
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int ch = t.ct * TC + t.c0 + c;
            op.z[c] = ok && ch < g.C ? st.spz[it & 1][(size_t)s * net.NH + L.h_out + ch * g.P + p] : 0.f;
        }
        tl_walk(g, t, net.S, smem, op);
        float v[CH][5];
#pragma unroll
        for (int c = 0; c < CH; ++c) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[c][e] = op.v[c][e];
            v[c][4] = (float)op.nout[c];   // a count below 2^24: exact, and exact when splits are added
        }
        tl_put<5, CH>(g, t, sums, v);
    }
    if (g.ks > 1 && !tl_join<5>(segs, g, t, sums)) return;
    __syncthreads();
#pragma unroll 1
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        int ch, lane, s, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, s, p) || t.ct * TC + ch >= g.C) continue;
        const float* v = sums + ch * row + lane;
        const int n = TC * row;
        const int i = (t.ct * TC + ch) * g.P + p;
        const size_t h = (size_t)s * net.NH + L.h_out + i;
        sp_rowB_unit(net, st, sc, L, s, i, h, it, st.spz[it & 1][h], v[0], v[n], v[2 * n], v[3 * n], (int)v[4 * n]);
    }
}
__global__ void __launch_bounds__(CB_THREADS, 2) k_sp_rowB_tl(DNet net, DState st, DSched sc,
                                                              const __grid_constant__ TlSegs segs) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    if (g.ch == 8) sp_row_tile<8>(net, st, sc, segs, g, tile_smem);
    else sp_row_tile<4>(net, st, sc, segs, g, tile_smem);
}

// Phase C fused with the next phase A (k_sp_colCA_t): the output records {alpha, beta_bar on beta_1, beta_bar on I*, z}.
template <int CH>
struct SpColOp : TlOp {
    static constexpr int RB = 16, EB = 0, WB = 4, SWEEPS = 1;
    const float4* src;
    size_t ss;
    float tp[CH], tn[CH], c[CH], a[CH];
    __device__ __forceinline__ void copy(uint32_t buf, int, int slot, int s, int i) const {
        tl_copy<16>(buf + slot * 16, src + (size_t)s * ss + i);
    }
    __device__ __forceinline__ const char* weights(const TlSeg& g) const { return reinterpret_cast<const char*>(g.w); }
    __device__ __forceinline__ void begin(int) {
#pragma unroll
        for (int k = 0; k < CH; ++k) c[k] = a[k] = 0.f;
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int, int slot, const char* w) {
        const float4 r = *reinterpret_cast<const float4*>(rec + slot * 16);
        const float in = r.y + r.z;   // one of the two is zero: the sum is exact
#pragma unroll
        for (int k4 = 0; k4 < CH; k4 += 4) {
            const float4 q = *reinterpret_cast<const float4*>(w + 4 * k4);
            const float wv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = k4 + e;
                c[k] = fmaf(wv[e], r.w >= (wv[e] > 0.f ? tp[k] : tn[k]) ? in : r.y, c[k]);
                a[k] = fmaf(wv[e], r.x, a[k]);
            }
        }
    }
    __device__ __forceinline__ void end(int) {}
};

// W x or W^T y of the first entries of float4 records: phase A alone (alpha), the primal initialisation's
// products (x; alpha* - beta_1*).
template <int CH>
struct DotOp : TlOp {
    static constexpr int RB = 4, EB = 0, WB = 4, SWEEPS = 1;
    const float4* src;
    size_t ss;
    float v[CH];
    __device__ __forceinline__ void copy(uint32_t buf, int, int slot, int s, int i) const {
        tl_copy<4>(buf + slot * 4, src + (size_t)s * ss + i);
    }
    __device__ __forceinline__ const char* weights(const TlSeg& g) const { return reinterpret_cast<const char*>(g.w); }
    __device__ __forceinline__ void begin(int) {
#pragma unroll
        for (int c = 0; c < CH; ++c) v[c] = 0.f;
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int, int slot, const char* w) {
        const float x = *reinterpret_cast<const float*>(rec + slot * 4);
#pragma unroll
        for (int c = 0; c < CH; c += 4) {
            const float4 q = *reinterpret_cast<const float4*>(w + 4 * c);
            v[c] = fmaf(q.x, x, v[c]);
            v[c + 1] = fmaf(q.y, x, v[c + 1]);
            v[c + 2] = fmaf(q.z, x, v[c + 2]);
            v[c + 3] = fmaf(q.w, x, v[c + 3]);
        }
    }
    __device__ __forceinline__ void end(int) {}
};

template <int CH>
__device__ __forceinline__ void sp_col_sums(const DNet& net, const DState& st, const DLayer& L, const TlSeg& g,
                                            const TlTile& t, char* smem) {
    SpColOp<CH> op;
    op.src = arec_planes(net, st, L, 0);
    op.ss = net.AT / 4;
    int s, p;
    const bool ok = tl_unit(g, t, t.lane, net.S, s, p);
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        const int ch = t.ct * tl_channels(g) + t.c0 + c;
        op.tp[c] = op.tn[c] = 0.f;
        if (ok && ch < g.C) {
            const float4* own = sp_iplane(net, st, L, s) + xin_pos(L, tl_col_neuron(L, g, ch, p));
            op.tp[c] = own[0].y;
            op.tn[c] = own[L.xpos].y;
        }
    }
    tl_walk(g, t, net.S, smem, op);
    float v[CH][2];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        v[c][0] = op.c[c];
        v[c][1] = op.a[c];
    }
    tl_put<2, CH>(g, t, reinterpret_cast<float*>(smem), v);
}
template <int CH>
__device__ __forceinline__ void dot_sums(const DNet& net, const float4* src, size_t ss, const TlSeg& g, const TlTile& t,
                                         char* smem) {
    DotOp<CH> op;
    op.src = src;
    op.ss = ss;
    tl_walk(g, t, net.S, smem, op);
    float v[CH][1];
#pragma unroll
    for (int c = 0; c < CH; ++c) v[c][0] = op.v[c];
    tl_put<1, CH>(g, t, reinterpret_cast<float*>(smem), v);
}
__device__ __forceinline__ void dot_tile(const DNet& net, const float4* src, size_t ss, const TlSeg& g, const TlTile& t,
                                         char* smem) {
    if (g.ch == 8) dot_sums<8>(net, src, ss, g, t, smem);
    else dot_sums<4>(net, src, ss, g, t, smem);
}

// What a col pass does with its inputs' sums.
enum SpCol { SP_PHASE_CA, SP_PHASE_A, SP_START, SP_INIT };
template <SpCol WHAT>
__global__ void __launch_bounds__(CB_THREADS, 3) k_sp_col_tl(DNet net, DState st, DSched sc,
                                                             const __grid_constant__ TlSegs segs) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const int k = g.li + 1, it = st.ctr[1], TC = tl_channels(g), row = tl_lanes(g) + 1;
    float* sums = reinterpret_cast<float*>(tile_smem);
    if (g.nch) {
        if constexpr (WHAT == SP_PHASE_CA) {
            if (g.ch == 8) sp_col_sums<8>(net, st, L, g, t, tile_smem);
            else sp_col_sums<4>(net, st, L, g, t, tile_smem);
            if (g.ks > 1 && !tl_join<2>(segs, g, t, sums)) return;
        } else {
            dot_tile(net, arec_planes(net, st, L, 0), net.AT / 4, g, t, tile_smem);
            if (g.ks > 1 && !tl_join<1>(segs, g, t, sums)) return;
        }
        __syncthreads();
    }
#pragma unroll 1
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        int ch, lane, s, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, s, p) || t.ct * TC + ch >= g.C) continue;
        const int j = tl_col_neuron(L, g, t.ct * TC + ch, p);
        const float v0 = g.nch ? sums[ch * row + lane] : 0.f;
        if constexpr (WHAT == SP_PHASE_CA) {
            sp_colC_unit(net, st, sc, L, k, s, j, it, v0, g.nch ? sums[(TC + ch) * row + lane] : 0.f);
        } else if constexpr (WHAT == SP_INIT) {
            const float x = spi_col_unit(net, st, sc, L, k, s, j, st.ctr[2], v0);
            if (k <= net.n - 1) sp_iplane(net, st, L, s)[xin_pos(L, j)].x = x;   // the row pass reads the records
        } else {
            sp_phaseA_epilogue(net, st, L, k, s, j, v0, it & 1, WHAT == SP_START);
        }
    }
}

// Primal initialisation, row pass.
__global__ void __launch_bounds__(CB_THREADS, 3) k_spi_row_tl(DNet net, DState st, const __grid_constant__ TlSegs segs) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const int cur = st.ctr[1] & 1, TC = tl_channels(g), row = tl_lanes(g) + 1;
    float* sums = reinterpret_cast<float*>(tile_smem);
    dot_tile(net, sp_iplane(net, st, L, 0), net.XT, g, t, tile_smem);
    if (g.ks > 1 && !tl_join<1>(segs, g, t, sums)) return;
    __syncthreads();
#pragma unroll 1
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        int ch, lane, s, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, s, p) || t.ct * TC + ch >= g.C) continue;
        const int i = (t.ct * TC + ch) * g.P + p;
        *sp_orec(net, st, L, s, i) = make_float4(spi_row_unit(net, st, L, s, i, cur, sums[ch * row + lane]), 0.f, 0.f, 0.f);
    }
}

// ---------------------------------------------------------------- launches
int tl_sp_row_smem(const TlSeg& g) { return tl_smem(g, 20, 4, 0, 5); }
int tl_sp_col_smem(const TlSeg& g) { return tl_smem(g, 16, 4, 0, 2); }

void tl_launch_sp_row(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                      cudaStream_t s) {
    k_sp_rowB_tl<<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t);
}
void tl_launch_sp_col(int what, int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                      cudaStream_t s) {
    switch (what) {
        case SP_PHASE_CA: k_sp_col_tl<SP_PHASE_CA><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t); break;
        case SP_PHASE_A: k_sp_col_tl<SP_PHASE_A><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t); break;
        case SP_START: k_sp_col_tl<SP_START><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t); break;
        default: k_sp_col_tl<SP_INIT><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t); break;
    }
}
void tl_launch_spi_row(int blocks, int smem, const DNet& net, const DState& st, const TlSegs& t, cudaStream_t s) {
    k_spi_row_tl<<<blocks, CB_THREADS, smem, s>>>(net, st, t);
}
int tl_ibp_smem(const TlSeg& g) { return tl_smem(g, 8, 4, 0, 5); }

cudaError_t tl_sp_prepare() {
    cudaError_t e = cudaSuccess;
    auto allow = [&](const void* k) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM_MAX);
    };
    allow((const void*)k_ibp_tl);
    allow((const void*)k_sp_rowB_tl);
    allow((const void*)k_spi_row_tl);
    allow((const void*)k_sp_col_tl<SP_PHASE_CA>);
    allow((const void*)k_sp_col_tl<SP_PHASE_A>);
    allow((const void*)k_sp_col_tl<SP_START>);
    allow((const void*)k_sp_col_tl<SP_INIT>);
    return e;
}

void tl_launch_ibp_box(int grid, const DNet& net, const DState& st, cudaStream_t s) {
    k_ibp_box<<<grid, CB_THREADS, 0, s>>>(net, st);
}

// Splits of a layer's walks: a layer is one launch, and one with fewer tiles than two per SM (linear layers:
// 64 at 256 subproblems and 512 rows) leaves most of the chip idle while its blocks walk all their sources. At
// least 64 taps per split. Without splits 13 conv4 boxes took 1.61 ms, a warp per row 1.53, split 0.60 (one pair a
// row; the totals changed nothing at this size: the batch's set-up takes 0.54 ms before, 0.53 after).
int tl_ibp_splits(const TlSeg& g, int S) {
    return std::max(1, std::min({152 * 2 / tl_tiles(g, S), g.nch, 16, g.SC * g.kt / 64}));
}

void tl_launch_ibp(const DNet& net, const DState& st, const TlSegs& segs, int q, const signed char* splits, cudaStream_t s) {
    TlSegs one{};
    one.n = 1;
    one.s[0] = segs.s[q];
    one.s[0].first = 0;
    one.s[0].ks = tl_ibp_splits(segs.s[q], net.S);
    one.s[0].part = 0;   // one launch at a time uses the context's scratch
    one.s[0].ctr = 0;
    one.part = segs.part;
    one.ctr = segs.ctr;
    k_ibp_tl<<<tl_tiles(segs.s[q], net.S) * one.s[0].ks, CB_THREADS, tl_ibp_smem(segs.s[q]), s>>>(net, st, one, splits);
}

}  // namespace cb
