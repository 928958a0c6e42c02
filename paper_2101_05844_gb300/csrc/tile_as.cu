// Active Set passes on tiles (cb_tile.cuh): the col and row pass of the float32 form, and the weights
// their segments read.
//
// The masked products ask for the sums over the positive and over the negative weights of a row or
// column separately (cb_team.cuh), and every channel has its own sign pattern. The taps are walked in
// their natural order with the weight split into the pair {max(w, 0), min(w, 0)}: col pass, one packed
// fma.rn.f32x2 adds to both sums; row pass, both sides go into one sum by scalar FMAs (an exact zero times
// the operand adds nothing). That spends two multiply-adds per one asked for. A warp-uniform branch on the
// sign instead, and packed pairs of slots, halved the FMA pipe's share (28 to 32% active) but waited on the
// branches and measured slower (col 546 -> 630 us, row 708 -> 719 us).
//
// Measured at 64 boxes of the conv4 net with five slots (packed FMA rate about 63 TFLOP/s): col pass 1555
// us by lane teams, 544 us; row pass 1047, 678 us. Bound by issue and the FMA pipe (43 to 53% active, 16
// warps per SM); 2048 subproblems of the Wide conv net: an iteration 6.4 -> 3.9 ms.
#include <algorithm>

#include "cb_tile.cuh"

namespace cb {

__global__ void k_tl_weights(DLayer L, int col, int py, int px, int rows, int C, int CP, float* w, float2* wpm) {
    // row segments: weight row t is the t-th input of a receptive field (conv: (channel, ky, kx)),
    // columns are output channels; col segments: (output channel, dky, dkx) of the stride phase, columns
    // are input channels
    const size_t n = (size_t)rows * CP;
    const int kk = L.kh * L.kw;
    const int nkx = (L.kw - px + L.st - 1) / L.st, nky = (L.kh - py + L.st - 1) / L.st;
    for (size_t u = blockIdx.x * (size_t)blockDim.x + threadIdx.x; u < n; u += (size_t)gridDim.x * blockDim.x) {
        const int t = (int)(u / CP), c = (int)(u - (size_t)t * CP);
        float v = 0.f;
        if (c < C) {
            if (L.kind == 0) {
                v = col ? L.W[(size_t)t * L.n_in + c] : L.W[(size_t)c * L.n_in + t];
            } else if (!col) {
                v = L.W[(size_t)c * L.ci * kk + t];
            } else {
                const int co = t / (nky * nkx), r = t - co * nky * nkx;
                const int dy = r / nkx, dx = r - dy * nkx;
                v = L.W[((size_t)co * L.ci + c) * kk + (py + L.st * dy) * L.kw + px + L.st * dx];
            }
        }
        w[u] = v;
        wpm[u] = make_float2(fmaxf(v, 0.f), fminf(v, 0.f));
    }
}

// ---------------------------------------------------------------- col pass
// Output records {rp, bz_b}: plane q holds entries 4q .. 4q + 3; only the 1 + NS entries in use are staged.
template <int NS>
struct ColRecords : TlOp {
    static constexpr int E = 1 + NS, RB = tl_arec_bytes(E), EB = 0;
    const float4* src;      // the layer's records of subproblem 0
    size_t ss;              // float4 per subproblem
    int apos;
    __device__ __forceinline__ void copy(uint32_t buf, int nrec, int slot, int s, int i) const {
        const float4* p = src + (size_t)s * ss + i;
        tl_copy<tl_piece(E)>(buf + slot * tl_piece(E), p);
        if constexpr (E > 4) tl_copy<tl_piece(E - 4)>(buf + nrec * 16 + slot * tl_piece(E - 4), p + apos);
        if constexpr (E > 8) tl_copy<tl_piece(E - 8)>(buf + nrec * 32 + slot * tl_piece(E - 8), p + 2 * (size_t)apos);
    }
    template <int N>
    static __device__ __forceinline__ void piece(const char* p, float* v) {
        if constexpr (N >= 3) {
            const float4 a = *reinterpret_cast<const float4*>(p);
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        } else if constexpr (N == 2) {
            const float2 a = *reinterpret_cast<const float2*>(p);
            v[0] = a.x; v[1] = a.y;
        } else {
            v[0] = *reinterpret_cast<const float*>(p);
        }
    }
    static __device__ __forceinline__ void load(const char* rec, int nrec, int slot, float (&v)[12]) {
        piece<E>(rec + slot * tl_piece(E), v);
        if constexpr (E > 4) piece<E - 4>(rec + nrec * 16 + slot * tl_piece(E - 4), v + 4);
        if constexpr (E > 8) piece<E - 8>(rec + nrec * 32 + slot * tl_piece(E - 8), v + 8);
    }
};

// More than five slots at eight channels per thread hold more accumulators than registers: such a walk
// sweeps the taps twice, four channels a sweep.
__host__ __device__ constexpr int as_halves(int ns, int ch) { return ns > 5 && ch > 4 ? 2 : 1; }

// Two neighbouring pairs of a weight row.
__device__ __forceinline__ void load_pairs(const char* w, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(w);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}

template <int NS, int CH>
struct ColOp : ColRecords<NS> {
    static constexpr int WB = NS ? 8 : 4, SWEEPS = as_halves(NS, CH), CW = CH / SWEEPS, NA = NS ? CW : CW / 2;
    unsigned pm[CH], qm[CH];   // the inputs' slot bits
    float f[CH];
    float2 acc[NA][1 + NS];    // {positive, negative taps} of a channel; NS = 0: channel pairs
    int c0 = 0;
    __device__ __forceinline__ const char* weights(const TlSeg& g) const {
        return NS ? reinterpret_cast<const char*>(g.wpm) : reinterpret_cast<const char*>(g.w);
    }
    __device__ __forceinline__ void begin(int sweep) {
        c0 = sweep * CW;
#pragma unroll
        for (int c = 0; c < NA; ++c)
#pragma unroll
            for (int b = 0; b <= NS; ++b) acc[c][b] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int nrec, int slot, const char* w) {
        float v[12];
        this->load(rec, nrec, slot, v);
        if constexpr (NS == 0) {
#pragma unroll
            for (int c = 0; c < NA; c += 2) {
                float2 p0, p1;
                load_pairs(w + 8 * c, p0, p1);
                acc[c][0] = fma2(p0, make_float2(v[0], v[0]), acc[c][0]);
                acc[c + 1][0] = fma2(p1, make_float2(v[0], v[0]), acc[c + 1][0]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < CW; c += 2) {
                float2 p0, p1;
                load_pairs(w + (c0 + c) * 8, p0, p1);
#pragma unroll
                for (int b = 0; b <= NS; ++b) {
                    acc[c][b] = fma2(p0, make_float2(v[b], v[b]), acc[c][b]);
                    acc[c + 1][b] = fma2(p1, make_float2(v[b], v[b]), acc[c + 1][b]);
                }
            }
        }
    }
    __device__ __forceinline__ void end(int sweep) {
#pragma unroll
        for (int h = 0; h < SWEEPS; ++h) {
            if (h != sweep) continue;
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const int o = h * CW + c;
                if constexpr (NS == 0) {
                    f[o] = c & 1 ? acc[c >> 1][0].y : acc[c >> 1][0].x;
                } else {
                    f[o] = acc[c][0].x + acc[c][0].y;
#pragma unroll
                    for (int b = 0; b < NS; ++b) {
                        if ((pm[o] >> b) & 1u) f[o] += acc[c][1 + b].x;
                        if ((qm[o] >> b) & 1u) f[o] += acc[c][1 + b].y;
                    }
                }
            }
        }
    }
};

// The same sums in the order of a lane per unit (cb_team.cuh): the positive taps of a channel, then its
// negative ones, into one accumulator of the unmasked product. Two sweeps over the taps for every four
// channels, for the gradient, which an input at a tie of f moves (the bound is continuous there and takes the
// packed sums: 16.2 against 8.9 ms at 1024 conv4 boxes and five slots). Equal bit for bit to a lane per unit
// where a tile is not split; a team of several lanes and a split tile add their parts' sums, and an input whose
// f is within rounding of zero may take its other end there.
template <int NS, int CH>
struct ColSeqOp : ColRecords<NS> {
    static constexpr int WB = 4, CW = 4, SWEEPS = 2 * CH / CW;
    unsigned pm[CH], qm[CH];
    float f[CH];
    float acc[CW], part[CW][NS > 0 ? NS : 1], pos[CW][NS > 0 ? NS : 1];
    bool neg = false;
    int c0 = 0;
    __device__ __forceinline__ const char* weights(const TlSeg& g) const { return reinterpret_cast<const char*>(g.w); }
    __device__ __forceinline__ void begin(int sweep) {
        neg = sweep & 1;
        c0 = sweep / 2 * CW;
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            if (!neg) acc[c] = 0.f;
#pragma unroll
            for (int b = 0; b < NS; ++b) part[c][b] = 0.f;
        }
    }
    __device__ __forceinline__ void step(const char* rec, const char*, int nrec, int slot, const char* w) {
        float v[12];
        this->load(rec, nrec, slot, v);
        const float4 q = *reinterpret_cast<const float4*>(w + c0 * 4);
        const float wv[CW] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            const float ws = neg ? fminf(wv[c], 0.f) : fmaxf(wv[c], 0.f);
            acc[c] = fmaf(ws, v[0], acc[c]);
#pragma unroll
            for (int b = 0; b < NS; ++b) part[c][b] = fmaf(ws, v[1 + b], part[c][b]);
        }
    }
    __device__ __forceinline__ void end(int sweep) {
        if (!neg) {
#pragma unroll
            for (int c = 0; c < CW; ++c)
#pragma unroll
                for (int b = 0; b < NS; ++b) pos[c][b] = part[c][b];
            return;
        }
#pragma unroll
        for (int h = 0; h < CH / CW; ++h) {
            if (h != sweep / 2) continue;
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                const int o = h * CW + c;
                f[o] = acc[c];
#pragma unroll
                for (int b = 0; b < NS; ++b) {
                    if ((pm[o] >> b) & 1u) f[o] += pos[c][b];
                    if ((qm[o] >> b) & 1u) f[o] += part[c][b];
                }
            }
        }
    }
};

// The tile's sums f of its inputs, their bits applied, into the staged sums.
template <int NS, int CH, class Op>
__device__ __forceinline__ void col_sums(const DNet& net, const DState& st, const DLayer& L, const TlSeg& g,
                                         const TlTile& t, int bo, char* smem) {
    Op op;
    op.src = arec_planes(net, st, L, 0);
    op.ss = net.AT / 4;
    op.apos = L.apos;
    int s, p;
    const bool ok = tl_unit(g, t, t.lane, net.S, s, p);
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        op.pm[c] = op.qm[c] = 0u;
        const int ch = t.ct * tl_channels(g) + t.c0 + c;
        if (NS && ok && ch < g.C) {
            const size_t xo = (size_t)s * net.NT + L.in_off + tl_col_neuron(L, g, ch, p);
            slot_bits(net, L, st.xsnap[bo][xo], st.efix[xo], op.pm[c], op.qm[c]);
        }
    }
    tl_walk(g, t, net.S, smem, op);
    float v[CH][1];
#pragma unroll
    for (int c = 0; c < CH; ++c) v[c][0] = op.f[c];
    tl_put<1, CH>(g, t, reinterpret_cast<float*>(smem), v);
}

// The epilogues run over the tile's units a step ahead of themselves: the next unit's state is loaded
// before this one's is worked through (with two blocks per SM one unit's round trips to DRAM at a time
// left the epilogue, not the walk, to bound the pass).
template <int NS>
__device__ __forceinline__ void col_epilogue(const DNet& net, const DState& st, const StepNow& sp, const DLayer& L,
                                             const TlSeg& g, const TlTile& t, int mode, const float* sums) {
    const int k = g.li + 1;
    const int TC = tl_channels(g), row = tl_lanes(g) + 1;
    struct Unit {
        int s, j, at;
        ColState<NS> c;
    };
    auto load = [&](int u, Unit& q) {
        int ch, lane, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, q.s, p) || t.ct * TC + ch >= g.C) return false;
        q.j = tl_col_neuron(L, g, t.ct * TC + ch, p);
        q.at = ch * row + lane;
        q.c = as_colA_load<NS>(net, st, sp, L, k, q.s, q.j, mode);
        return true;
    };
    Unit cur, nxt;
    bool on = load(threadIdx.x, cur);
#pragma unroll 1
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        const bool more = u + CB_THREADS < tl_units(g) && load(u + CB_THREADS, nxt);
        if (on) {
            const float f = k <= net.n - 1 ? sums[cur.at] : -net.Wout[(size_t)cur.s * L.n_in + cur.j];
            as_colA_unit<NS>(net, st, sp, L, k, cur.s, cur.j, f, cur.c, mode);
        }
        cur = nxt;
        on = more;
    }
}

template <int NS, bool SEQ>
__device__ __forceinline__ void col_tile(const DNet& net, const DState& st, const StepNow& sp, const DLayer& L,
                                         const TlSegs& segs, const TlSeg& g, const TlTile& t, int mode, char* smem) {
    if (g.nch) {
        const int bo = sp.nadd_before & 1;
        if (g.ch == 8) {
            if constexpr (SEQ) col_sums<NS, 8, ColSeqOp<NS, 8>>(net, st, L, g, t, bo, smem);
            else col_sums<NS, 8, ColOp<NS, 8>>(net, st, L, g, t, bo, smem);
        } else {
            if constexpr (SEQ) col_sums<NS, 4, ColSeqOp<NS, 4>>(net, st, L, g, t, bo, smem);
            else col_sums<NS, 4, ColOp<NS, 4>>(net, st, L, g, t, bo, smem);
        }
        if (g.ks > 1 && !tl_join<1>(segs, g, t, reinterpret_cast<float*>(smem))) return;
        __syncthreads();
    }
    col_epilogue<NS>(net, st, sp, L, g, t, mode, reinterpret_cast<const float*>(smem));
}

template <bool SEQ>
__global__ void __launch_bounds__(CB_THREADS, 2) k_as_colA_tl(DNet net, DState st, DSched sc,
                                                              const __grid_constant__ TlSegs segs, int mode) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const StepNow sp = cb_step(st);
    switch (min(sp.nadd_before, sc.maxcut)) {
        case 0: col_tile<0, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 1: col_tile<1, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 2: col_tile<2, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 3: col_tile<3, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 4: col_tile<4, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 5: col_tile<5, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 6: col_tile<6, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        case 7: col_tile<7, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
        default: col_tile<8, SEQ>(net, st, sp, L, segs, g, t, mode, tile_smem); break;
    }
}

// Saddle Point's start (eq. 10): P_k = W^T beta_{k,1} + sum_b (W o I_b)^T beta_{k,b}, the col pass's masked
// product over records that hold beta_1 in the place of -(alpha - beta_1) (k_rowprep).
template <int NS>
__device__ __forceinline__ void convert_tile(const DNet& net, const DState& st, const DLayer& L, const TlSegs& segs,
                                             const TlSeg& g, const TlTile& t, int bo, char* smem) {
    if (g.ch == 8) col_sums<NS, 8, ColOp<NS, 8>>(net, st, L, g, t, bo, smem);
    else col_sums<NS, 4, ColOp<NS, 4>>(net, st, L, g, t, bo, smem);
    const float* sums = reinterpret_cast<const float*>(smem);
    if (g.ks > 1 && !tl_join<1>(segs, g, t, reinterpret_cast<float*>(smem))) return;
    __syncthreads();
    const int TC = tl_channels(g), row = tl_lanes(g) + 1;
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        int ch, lane, s, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, s, p) || t.ct * TC + ch >= g.C) continue;
        st.P[(size_t)s * net.NT + L.in_off + tl_col_neuron(L, g, t.ct * TC + ch, p)] = sums[ch * row + lane];
    }
}
__global__ void __launch_bounds__(CB_THREADS, 2) k_sp_convert_tl(DNet net, DState st, DSched sc,
                                                                 const __grid_constant__ TlSegs segs) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    if (!g.nch) return;   // the output layer's inputs carry no P
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const StepNow sp = cb_step(st);
    const int bo = sp.nadd_before & 1;
    switch (min(sp.nadd_before, sc.maxcut)) {
        case 0: convert_tile<0>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 1: convert_tile<1>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 2: convert_tile<2>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 3: convert_tile<3>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 4: convert_tile<4>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 5: convert_tile<5>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 6: convert_tile<6>(net, st, L, segs, g, t, bo, tile_smem); break;
        case 7: convert_tile<7>(net, st, L, segs, g, t, bo, tile_smem); break;
        default: convert_tile<8>(net, st, L, segs, g, t, bo, tile_smem); break;
    }
}

// ---------------------------------------------------------------- row pass
// W x* and the masked products from the input records {x*, p bits | q bits << 8}: under a positive weight
// a slot takes x* where its p bit is set, under a negative one where its q bit is. The records are
// spread into one pair {x* p_b, x* q_b} per slot when a chunk has arrived: picked per tap, the bits cost
// as many instructions as the products (conv4 net, 64 boxes, five slots: 526 M instructions a pass).
template <int NS, int CH>
struct RowOp : TlOp {
    static constexpr int RB = 8, EB = 8 * NS, WB = NS ? 8 : 4, SWEEPS = 1;
    const float2* src;
    size_t ss;              // records per subproblem
    float v[CH][1 + NS];
    __device__ __forceinline__ void copy(uint32_t buf, int, int slot, int s, int i) const {
        tl_copy<8>(buf + slot * 8, src + (size_t)s * ss + i);
    }
    __device__ __forceinline__ const char* weights(const TlSeg& g) const {
        return NS ? reinterpret_cast<const char*>(g.wpm) : reinterpret_cast<const char*>(g.w);
    }
    __device__ __forceinline__ void begin(int) {
#pragma unroll
        for (int c = 0; c < CH; ++c)
#pragma unroll
            for (int b = 0; b <= NS; ++b) v[c][b] = 0.f;
    }
    __device__ __forceinline__ void expand(const char* rec, char* ex, int nrec, int i) const {
        const float2 r = *reinterpret_cast<const float2*>(rec + i * 8);
        const unsigned bits = __float_as_uint(r.y);
#pragma unroll
        for (int b = 0; b < NS; ++b)
            *reinterpret_cast<float2*>(ex + (b * nrec + i) * 8) =
                make_float2(bits & (1u << b) ? r.x : 0.f, bits & (256u << b) ? r.x : 0.f);
    }
    __device__ __forceinline__ void step(const char* rec, const char* ex, int nrec, int slot, const char* w) {
        const float x = *reinterpret_cast<const float*>(rec + slot * 8);
        if constexpr (NS == 0) {
#pragma unroll
            for (int c = 0; c < CH; c += 4) {
                const float4 q = *reinterpret_cast<const float4*>(w + 4 * c);
                v[c][0] = fmaf(q.x, x, v[c][0]);
                v[c + 1][0] = fmaf(q.y, x, v[c + 1][0]);
                v[c + 2][0] = fmaf(q.z, x, v[c + 2][0]);
                v[c + 3][0] = fmaf(q.w, x, v[c + 3][0]);
            }
        } else {
            float2 xb[NS];   // x* under positive and under negative weights
#pragma unroll
            for (int b = 0; b < NS; ++b) xb[b] = *reinterpret_cast<const float2*>(ex + (b * nrec + slot) * 8);
#pragma unroll
            for (int c = 0; c < CH; c += 2) {
                float2 p[2];
                load_pairs(w + c * 8, p[0], p[1]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    v[c + e][0] = fmaf(p[e].x + p[e].y, x, v[c + e][0]);
#pragma unroll
                    for (int b = 0; b < NS; ++b)
                        v[c + e][1 + b] = fmaf(p[e].y, xb[b].y, fmaf(p[e].x, xb[b].x, v[c + e][1 + b]));
                }
            }
        }
    }
    __device__ __forceinline__ void end(int) {}
};

template <int NS, int CH>
__device__ __forceinline__ void row_sums(const DNet& net, const DState& st, const DLayer& L, const TlSeg& g,
                                         const TlTile& t, char* smem) {
    RowOp<NS, CH> op;
    op.src = xin_recs(net, st, L, 0);
    op.ss = net.XT / 2;
    tl_walk(g, t, net.S, smem, op);
    tl_put<1 + NS, CH>(g, t, reinterpret_cast<float*>(smem), op.v);
}

template <int NS, bool ADD>
__device__ __forceinline__ void row_epilogue(const DNet& net, const DState& st, const DSched& sc, const StepNow& sp,
                                             const DLayer& L, const TlSeg& g, const TlTile& t, const float* sums) {
    const int TC = tl_channels(g), row = tl_lanes(g) + 1;
    struct Unit {
        int s, i, at;
        RowState<NS> r;
    };
    auto load = [&](int u, Unit& q) {
        int ch, lane, p;
        tl_order(g, L.kind == 0, u, ch, lane);
        if (!tl_unit(g, t, lane, net.S, q.s, p) || t.ct * TC + ch >= g.C) return false;
        q.i = (t.ct * TC + ch) * g.P + p;
        q.at = ch * row + lane;
        q.r = as_rowB_load<NS, ADD, true>(net, st, L, q.s, q.i, sp);
        return true;
    };
    Unit cur, nxt;
    bool on = load(threadIdx.x, cur);
#pragma unroll 1
    for (int u = threadIdx.x; u < tl_units(g); u += CB_THREADS) {
        const bool more = u + CB_THREADS < tl_units(g) && load(u + CB_THREADS, nxt);
        if (on) {
            float v[1 + NS];
#pragma unroll
            for (int b = 0; b <= NS; ++b) v[b] = sums[b * TC * row + cur.at];
            as_rowB_unit<NS, ADD, true>(net, st, sc, L, cur.s, cur.i, sp, v[0], v + 1, cur.r);
        }
        cur = nxt;
        on = more;
    }
}

template <int NS>
__device__ __forceinline__ void row_tile(const DNet& net, const DState& st, const DSched& sc, const StepNow& sp,
                                         const DLayer& L, const TlSegs& segs, const TlSeg& g, const TlTile& t, char* smem) {
    if (g.ch == 8) row_sums<NS, 8>(net, st, L, g, t, smem);
    else row_sums<NS, 4>(net, st, L, g, t, smem);
    if (g.ks > 1 && !tl_join<1 + NS>(segs, g, t, reinterpret_cast<float*>(smem))) return;
    __syncthreads();
    const float* sums = reinterpret_cast<const float*>(smem);
    if constexpr (NS > 0) {
        if (sp.b_new >= 0) {
            row_epilogue<NS, true>(net, st, sc, sp, L, g, t, sums);
            return;
        }
    }
    row_epilogue<NS, false>(net, st, sc, sp, L, g, t, sums);
}

__global__ void __launch_bounds__(CB_THREADS, 2) k_as_rowB_tl(DNet net, DState st, DSched sc,
                                                              const __grid_constant__ TlSegs segs) {
    extern __shared__ __align__(16) char tile_smem[];
    const TlSeg& g = segs.s[tlseg_of(segs, blockIdx.x)];
    const DLayer& L = net.L[g.li];
    const TlTile t = tl_tile(g);
    const StepNow sp = cb_step(st);
    switch (min(sp.nadd_before + (sp.b_new >= 0 ? 1 : 0), sc.maxcut)) {
        case 0: row_tile<0>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 1: row_tile<1>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 2: row_tile<2>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 3: row_tile<3>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 4: row_tile<4>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 5: row_tile<5>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 6: row_tile<6>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        case 7: row_tile<7>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
        default: row_tile<8>(net, st, sc, sp, L, segs, g, t, tile_smem); break;
    }
}

// ---------------------------------------------------------------- launches
void tl_weights(const DLayer& L, bool col, const TlSeg& g, float* w, float2* wpm, cudaStream_t s) {
    const int CP = g.nct * tl_channels(g);
    const size_t cells = (size_t)g.SC * g.kt * CP;
    const int grid = (int)std::min<size_t>((cells + CB_THREADS - 1) / CB_THREADS, 152 * 16);
    k_tl_weights<<<grid, CB_THREADS, 0, s>>>(L, col, g.py, g.px, g.SC * g.kt, g.C, CP, w, wpm);
}

cudaError_t tl_as_prepare() {
    cudaError_t e = cudaFuncSetAttribute(k_as_colA_tl<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_as_colA_tl<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sp_convert_tl, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_as_rowB_tl, cudaFuncAttributeMaxDynamicSharedMemorySize, TL_SMEM_MAX);
    return e;
}

void tl_launch_colA(bool seq, int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                    int mode, cudaStream_t s) {
    if (seq) k_as_colA_tl<true><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t, mode);
    else k_as_colA_tl<false><<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t, mode);
}

void tl_launch_rowB(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                    cudaStream_t s) {
    k_as_rowB_tl<<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t);
}

void tl_launch_sp_convert(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                          cudaStream_t s) {
    k_sp_convert_tl<<<blocks, CB_THREADS, smem, s>>>(net, st, sc, t);
}

}  // namespace cb
