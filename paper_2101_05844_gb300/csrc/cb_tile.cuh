// Tiled walks: the products of a pass from records staged in shared memory.
//
// A block takes one tile of a layer (or of a stride phase of a layer): LT = 32 lw positions, from one
// subproblem or, where a plane is smaller, from several, times TC = ch (8 / lw) channels; a thread holds
// ch = 8 channels of one position (4 for layers of up to four channels). The walk's source channels go through shared memory in chunks, double
// buffered with cp.async: the window of records the tile's positions reach (whole rows of the padded
// planes, one contiguous run) and the chunk's weights. A record then comes from L2 once per tile and
// from shared memory once per tap for eight channels.
//
// What this replaces: a lane team per unit (cb_team.cuh) loads a record from L1 for every (unit, tap),
// which bound it (conv4 net: 42 bytes per (box, nonzero), 92% L1 throughput, 8% of the float32 rate);
// lanes over four or eight channels straight from L1 cut that traffic but waited on it (a third of the
// issue slots used with one tap loaded ahead, 16 warps per SM).
//
// With few tiles (small batches, the wide linear layers of a conv net) a tile's chunks are split over ks
// blocks: each leaves its sums in global scratch, and the block that arrives last adds them in split
// order and does the tile's epilogue. No block waits for another.
#pragma once
#include "cb_dev.cuh"

namespace cb {

constexpr int TL_MAXSEG = 28;       // segments of a launch
// Dynamic shared memory a tiled kernel may ask for (two blocks per SM). The limit that a kernel is given belongs
// to the kernel, not to a context: it is this value for every context, never one context's own need, which would
// have the launches of another context with larger tiles refused.
constexpr int TL_SMEM_MAX = 100 * 1024;

struct TlSeg {
    int li, first;          // layer; first block
    int linear;             // a linear layer's: one position, a subproblem's records neighbours
    int P, Wq;              // positions per subproblem and per line of its grid
    int ch;                 // channels per thread
    int lw, nsub, npt;      // lane warps; subproblems per tile; tiles per subproblem (nsub = 1)
    int C, nct;             // channels; channel tiles
    int SC, CK, nch, ks;    // source channels, per chunk (a power of two for linear layers); chunks; split
    int kt;                 // taps per source channel
    int WX, WN, CS;         // window: records per row, per subproblem, and per source channel
    int step, base;         // window records per line and per column step; offset of a tile's first position
    int row0, rows;         // plane row of line 0's window; rows of a plane
    int cs;                 // records per source channel
    int py, px, y0, x0;     // col pass of a conv: input (y, x) = ((y0 + Y) st + py - pad, (x0 + X) st + px - pad)
    int ctr;                // first of the tiles' arrival counters (ks > 1)
    size_t part;            // first float of the tiles' partial sums (ks > 1)
    const int* kofs;        // [CK kt rounded up to 4] window offset of each tap of a chunk
    const float* w;         // [SC kt][nct TC] weights
    const float2* wpm;      // [SC kt][nct TC] {max(w, 0), min(w, 0)}
};
struct TlSegs {
    int n;
    TlSeg s[TL_MAXSEG];
    float* part;            // partial sums of split tiles
    int* ctr;               // arrivals
};

__host__ __device__ inline int tl_lanes(const TlSeg& g) { return 32 * g.lw; }
__host__ __device__ inline int tl_channels(const TlSeg& g) { return g.ch * (8 / g.lw); }
__host__ __device__ inline int tl_units(const TlSeg& g) { return CB_THREADS * g.ch; }
// records of a chunk, a multiple of 4 (the pieces of a record lie in arrays of this length)
__host__ __device__ inline int tl_records(const TlSeg& g) { return (g.CK * g.CS + 3) & ~3; }
__host__ __device__ inline int tl_offsets(const TlSeg& g) { return (g.CK * g.kt + 3) & ~3; }
// Bytes of one buffer with records of rb and weights of wb bytes, and of a tile's staged sums of nv
// values per unit.
__host__ __device__ inline int tl_buffer(const TlSeg& g, int rb, int wb) {
    return tl_records(g) * rb + g.CK * g.kt * tl_channels(g) * wb;
}

__host__ __device__ inline int tl_sums(const TlSeg& g, int nv) {
    return (nv * tl_channels(g) * (tl_lanes(g) + 1) * (int)sizeof(float) + 15) & ~15;
}
// Bytes of a block's shared memory: two buffers, expanded records of eb bytes and the offsets; the
// sums lie over them.
__host__ __device__ inline int tl_smem(const TlSeg& g, int rb, int wb, int eb, int nv) {
    const int walk = 2 * tl_buffer(g, rb, wb) + tl_records(g) * eb + tl_offsets(g) * (int)sizeof(int);
    const int sums = tl_sums(g, nv);
    return walk > sums ? walk : sums;
}
// floats of one split's sums
__host__ __device__ inline size_t tl_split(const TlSeg& g, int nv) { return tl_sums(g, nv) / sizeof(float); }
__host__ __device__ inline int tl_tiles(const TlSeg& g, int S) {
    return (g.nsub > 1 ? (S + g.nsub - 1) / g.nsub : S * g.npt) * g.nct;
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}

template <int BYTES>
__device__ __forceinline__ void tl_copy(uint32_t dst, const void* src) {
    static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async piece");
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}

__device__ __forceinline__ int tlseg_of(const TlSegs& t, int blk) {
    int q = 0;
    while (q + 1 < t.n && blk >= t.s[q + 1].first) ++q;
    return q;
}

// A block's tile, and this thread's place in it.
struct TlTile {
    int tile, ks;           // tile of the segment; split
    int ct, s0, p0;         // channel tile, first subproblem and position
    int lane, c0;           // lane of the tile; first channel of the thread within the channel tile
    int win;                // window record of the lane's position
};
__device__ __forceinline__ TlTile tl_tile(const TlSeg& g) {
    TlTile t;
    const int blk = blockIdx.x - g.first;
    t.ks = blk % g.ks;
    t.tile = blk / g.ks;
    t.ct = t.tile % g.nct;
    const int lt = t.tile / g.nct;
    if (g.nsub > 1) {
        t.s0 = lt * g.nsub;
        t.p0 = 0;
    } else {
        t.s0 = lt / g.npt;
        t.p0 = (lt - t.s0 * g.npt) * tl_lanes(g);
    }
    const int warp = threadIdx.x >> 5;
    t.lane = (warp % g.lw) * 32 + (threadIdx.x & 31);
    t.c0 = (warp / g.lw) * g.ch;
    int sub = 0, p = t.p0 + t.lane;
    if (g.nsub > 1) {
        sub = t.lane / g.P;
        p = t.lane - sub * g.P;
    }
    if (sub >= g.nsub || p >= g.P) {   // an idle lane walks the tile's first position
        sub = 0;
        p = t.p0;
    }
    const int y = p / g.Wq, x = p - y * g.Wq;
    t.win = g.base + sub * g.WN + ((y - t.p0 / g.Wq) * g.WX + x) * g.step;
    return t;
}

// The subproblem and position of lane l of a tile; false for an idle one.
__device__ __forceinline__ bool tl_unit(const TlSeg& g, const TlTile& t, int l, int S, int& s, int& p) {
    int sub = 0;
    p = t.p0 + l;
    if (g.nsub > 1) {
        sub = l / g.P;
        p = l - sub * g.P;
    }
    s = t.s0 + sub;
    return sub < g.nsub && s < S && p < g.P;
}

// What a walk's op may leave as it is here: taken() hears of the taps after every four of them (a chunk's last
// ones singly), or after each with singly().
struct TlOp {
    __device__ __forceinline__ bool singly() const { return false; }
    __device__ __forceinline__ void taken(int) {}
};

// One chunk into a buffer: op copies record `src` of subproblem s into slot `slot`.
template <class Op>
__device__ __forceinline__ void tl_stage(const TlSeg& g, const TlTile& t, int S, int chunk, uint32_t buf, const Op& op) {
    const int c0 = chunk * g.CK, nc = min(g.CK, g.SC - c0), nrec = tl_records(g);
    // (a conv layer's window can be one record as well: its chunks are no power of two, and its source
    // channels may lie further apart)
    if (g.linear) {   // a subproblem's records are neighbours, source channel fastest
        for (int i = threadIdx.x; i < g.CK * g.nsub; i += CB_THREADS) {
            const int c = i & (g.CK - 1), sub = i >> (31 - __clz(g.CK));
            if (c < nc && t.s0 + sub < S) op.copy(buf, nrec, c * g.CS + sub, t.s0 + sub, c0 + c);
        }
    } else {
        const int row = g.row0 + t.p0 / g.Wq * g.step;
        const int n = min(g.WN, (g.rows - row) * g.WX);
        // a run of n records per (source channel, subproblem), by as many lanes of a warp as it has records
        const int lg = g.WN >= 32 ? 5 : g.WN > 1 ? 32 - __clz(g.WN - 1) : 0;
        const int lane = threadIdx.x & ((1 << lg) - 1);
        for (int q = threadIdx.x >> lg; q < nc * g.nsub; q += CB_THREADS >> lg) {
            const int c = q / g.nsub, sub = q - c * g.nsub;
            if (t.s0 + sub >= S) continue;
            const int src = (c0 + c) * g.cs + row * g.WX, slot = c * g.CS + sub * g.WN;
            for (int i = lane; i < n; i += 1 << lg) op.copy(buf, nrec, slot + i, t.s0 + sub, src + i);
        }
    }
    const int TC = tl_channels(g), lp = 31 - __clz(TC * Op::WB / 16);   // log2 of a weight row's 16-byte pieces
    const uint32_t wdst = buf + nrec * Op::RB;
    const char* wsrc = op.weights(g) + ((size_t)c0 * g.kt * g.nct + t.ct) * TC * Op::WB;
    for (int i = threadIdx.x; i < (nc * g.kt) << lp; i += CB_THREADS) {
        const int r = i >> lp, q = i & ((1 << lp) - 1);
        tl_copy<16>(wdst + i * 16, wsrc + (size_t)r * g.nct * TC * Op::WB + q * 16);
    }
}

// The tile's walk: op accumulates every tap of the block's chunks. smem: two buffers, the expanded
// records (an op with EB > 0 spreads a staged record over EB bytes once per tile, not once per tap),
// then the offsets.
template <class Op>
__device__ __forceinline__ void tl_walk(const TlSeg& g, const TlTile& t, int S, char* smem, Op& op) {
    const int bytes = tl_buffer(g, Op::RB, Op::WB), nrec = tl_records(g), TC = tl_channels(g);
    char* ex = smem + 2 * bytes;
    int* ko = reinterpret_cast<int*>(ex + nrec * Op::EB);
    for (int i = threadIdx.x; i < tl_offsets(g); i += CB_THREADS) ko[i] = __ldg(g.kofs + i);
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
    const int ca = (int)((long long)g.nch * t.ks / g.ks), ce = (int)((long long)g.nch * (t.ks + 1) / g.ks);
    for (int sweep = 0; sweep < Op::SWEEPS; ++sweep) {
        op.begin(sweep);
        if (ca < ce) tl_stage(g, t, S, ca, base, op);
        asm volatile("cp.async.commit_group;" ::: "memory");
        for (int ch = ca; ch < ce; ++ch) {
            const int b = (ch - ca) & 1;
            if (ch + 1 < ce) tl_stage(g, t, S, ch + 1, base + (b ^ 1) * bytes, op);
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();
            const char* rec = smem + b * bytes;
            const char* w = rec + nrec * Op::RB + t.c0 * Op::WB;
            const int nc = min(g.CK, g.SC - ch * g.CK), nk = nc * g.kt;
            if constexpr (Op::EB > 0) {
                for (int i = threadIdx.x; i < nc * g.CS; i += CB_THREADS) op.expand(rec, ex, nrec, i);
                __syncthreads();
            }
            int k = 0;
            const int nk4 = op.singly() ? 0 : nk;
            for (; k + 4 <= nk4; k += 4) {
                const int4 o = *reinterpret_cast<const int4*>(ko + k);
                op.step(rec, ex, nrec, t.win + o.x, w + (k + 0) * TC * Op::WB);
                op.step(rec, ex, nrec, t.win + o.y, w + (k + 1) * TC * Op::WB);
                op.step(rec, ex, nrec, t.win + o.z, w + (k + 2) * TC * Op::WB);
                op.step(rec, ex, nrec, t.win + o.w, w + (k + 3) * TC * Op::WB);
                op.taken(4);
            }
            for (; k < nk; ++k) {
                op.step(rec, ex, nrec, t.win + ko[k], w + k * TC * Op::WB);
                op.taken(1);
            }
            __syncthreads();
        }
        op.end(sweep);
    }
}

// The thread's NV values of its CH channels into the staged sums (value, channel, lane).
template <int NV, int CH>
__device__ __forceinline__ void tl_put(const TlSeg& g, const TlTile& t, float* sums, const float (&v)[CH][NV]) {
    const int TC = tl_channels(g), row = tl_lanes(g) + 1;
#pragma unroll
    for (int c = 0; c < CH; ++c)
#pragma unroll
        for (int e = 0; e < NV; ++e) sums[(e * TC + t.c0 + c) * row + t.lane] = v[c][e];
}

// A split tile's partial sums in the scratch.
template <int NV>
__device__ __forceinline__ float4* tl_partials(const TlSegs& segs, const TlSeg& g, const TlTile& t) {
    return reinterpret_cast<float4*>(segs.part + g.part) + (size_t)t.tile * g.ks * (tl_split(g, NV) / 4);
}

// This block's sums into the scratch; true in the block that arrives last, which then sees every split's.
// Every thread takes part.
template <int NV>
__device__ __forceinline__ bool tl_arrive(const TlSegs& segs, const TlSeg& g, const TlTile& t, const float* sums) {
    const int n4 = (NV * tl_channels(g) * (tl_lanes(g) + 1) + 3) / 4;
    const size_t stride = tl_split(g, NV) / 4;
    float4* part = tl_partials<NV>(segs, g, t);
    __shared__ int last;
    __syncthreads();
    for (int i = threadIdx.x; i < n4; i += CB_THREADS)
        __stcg(part + t.ks * stride + i, reinterpret_cast<const float4*>(sums)[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        int* c = segs.ctr + g.ctr + t.tile;
        last = atomicAdd(c, 1) == g.ks - 1;
        if (last) *c = 0;   // for the next launch
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    return true;
}

// A split tile: true in the block that arrives last, which then holds the tile's sums (added in split order).
template <int NV>
__device__ __forceinline__ bool tl_join(const TlSegs& segs, const TlSeg& g, const TlTile& t, float* sums) {
    if (!tl_arrive<NV>(segs, g, t, sums)) return false;
    const int n4 = (NV * tl_channels(g) * (tl_lanes(g) + 1) + 3) / 4;
    const size_t stride = tl_split(g, NV) / 4;
    const float4* part = tl_partials<NV>(segs, g, t);
    for (int i = threadIdx.x; i < n4; i += CB_THREADS) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < g.ks; q += 8) {   // eight splits in flight
            float4 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (q + e < g.ks) v[e] = __ldcg(part + (q + e) * stride + i);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (q + e < g.ks) a = make_float4(a.x + v[e].x, a.y + v[e].y, a.z + v[e].z, a.w + v[e].w);
        }
        reinterpret_cast<float4*>(sums)[i] = a;
    }
    return true;
}

// Unit u (0 .. tl_units - 1) of a tile in epilogue order: linear layers run over a subproblem's channels,
// conv layers over a channel's positions, so that neighbouring threads take neighbouring neurons.
__device__ __forceinline__ void tl_order(const TlSeg& g, bool linear, int u, int& ch, int& lane) {
    if (linear) {
        const int TC = tl_channels(g);
        lane = u / TC;
        ch = u - lane * TC;
    } else {
        const int LT = tl_lanes(g);
        ch = u / LT;
        lane = u - ch * LT;
    }
}

// Input neuron of channel c at position p of a col segment.
__device__ __forceinline__ int tl_col_neuron(const DLayer& L, const TlSeg& g, int c, int p) {
    if (L.kind == 0) return c;
    const int Y = p / g.Wq, X = p - Y * g.Wq;
    return (c * L.hi + (g.y0 + Y) * L.st + g.py - L.pd) * L.wi + (g.x0 + X) * L.st + g.px - L.pd;
}

// Launches (tile_as.cu). tl_weights fills a segment's weights from its layer's; tl_as_prepare allows
// the passes TL_SMEM_MAX; seq: the col pass's sums in the lane teams' order.
void tl_weights(const DLayer& L, bool col, const TlSeg& g, float* w, float2* wpm, cudaStream_t s);
cudaError_t tl_as_prepare();
void tl_launch_colA(bool seq, int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                    int mode, cudaStream_t s);
void tl_launch_rowB(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                    cudaStream_t s);
// Interval propagation (tile_sp.cu): the input box's records, then a row segment per hidden layer.
int tl_ibp_smem(const TlSeg& g);
int tl_ibp_splits(const TlSeg& g, int S);
cudaError_t tl_sp_prepare();
void tl_launch_ibp_box(int grid, const DNet& net, const DState& st, cudaStream_t s);
void tl_launch_ibp(const DNet& net, const DState& st, const TlSegs& segs, int q, const signed char* splits, cudaStream_t s);
// Saddle Point (tile_sp.cu): its passes, the col pass's work by `what` (0: phase C and the next phase A, 1:
// phase A, 2: phase A starting the primal iterate, 3: a step of the primal initialisation).
int tl_sp_row_smem(const TlSeg& g);
int tl_sp_col_smem(const TlSeg& g);
void tl_launch_sp_row(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                      cudaStream_t s);
void tl_launch_sp_col(int what, int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                      cudaStream_t s);
void tl_launch_spi_row(int blocks, int smem, const DNet& net, const DState& st, const TlSegs& t, cudaStream_t s);
void tl_launch_sp_convert(int blocks, int smem, const DNet& net, const DState& st, const DSched& sc, const TlSegs& t,
                          cudaStream_t s);
// record bytes of the Active Set passes with up to cap slots (pieces of 4, 8 or 16 bytes)
__host__ __device__ constexpr int tl_piece(int entries) { return entries >= 3 ? 16 : 4 * entries; }
__host__ __device__ constexpr int tl_arec_bytes(int entries) {
    return entries <= 4 ? tl_piece(entries) : entries <= 8 ? 16 + tl_piece(entries - 4) : 32 + tl_piece(entries - 8);
}

}  // namespace cb
