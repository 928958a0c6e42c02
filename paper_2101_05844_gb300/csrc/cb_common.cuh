// Device-side descriptors shared by the kernels and the host API of the convex-barrier library.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#define CB_MAXL 10
#define CB_MAXCUT 8
#define CB_THREADS 256
#define CB_WARPS (CB_THREADS / 32)

// Kernel ids for per-kernel timing (as_kernel_times).
enum { CB_K_AS_COLA = 0, CB_K_AS_ROWB, CB_K_REDUCE, CB_K_SP_COLA, CB_K_SP_ROWB, CB_K_SP_COLC,
       CB_K_SPI_ROW, CB_K_SPI_COL, CB_K_TC_COL, CB_K_TC_ROW, CB_K_SLOT_SUMS, CB_K_BALL_X0,
       CB_K_BATCH, CB_K_SP_START, CB_K_COUNTER, CB_NPROF };

// One affine layer k (1-based in the paper; stored at index k-1).
struct DLayer {
    int kind;              // 0 linear, 1 conv2d
    int n_in, n_out;
    int ci, hi, wi, co, ho, wo, kh, kw, st, pd;
    const float* W;        // linear [n_out][n_in], conv [co][ci][kh][kw]
    const float* b;        // per output neuron [n_out]
    int in_off, out_off;   // offsets of the input / output neuron layer in [NT] vectors
    int h_in, h_out;       // offsets in [NH] hidden vectors (-1 when not a hidden layer)
    // Active Set walks (hidden-output layers). Tap lists {offset in floats, weight bits} per group,
    // the group's positive weights first: taps [grp[2g], grp[2g+1]) have W > 0 and
    // [grp[2g+1], grp[2g+2]) have W < 0 (zero weights are left out).
    //  row pass: group = output row (linear) or output channel (conv); offsets index the input
    //            records of this layer in positions (zero-padded input plane for conv)
    //  col pass: group = input (linear) or (input channel, stride phase y, stride phase x) (conv);
    //            offsets index the output records in positions (output plane with a zero halo
    //            for conv)
    const int2* rtap;
    const int* rgrp;
    const int2* ctap;
    const int* cgrp;
    int xo, ao;            // offsets (floats) of this layer's input / output records in a subproblem
    int xpos, apos;        // input / output record positions (padded planes for conv)
    int Hp, Wp;            // padded input plane (conv): in + 2 pad
    int Hpo, Wpo, hl, wl;  // output plane with halo (conv): rows hl .. hl + ho - 1 are the outputs
};

#define CB_MAXPH 9   // stride phases of a conv layer in the BF16 form (stride <= 3)

// BF16 form of the Active Set passes, per hidden-output layer: the tensor-core operands
// (channels-last planes, channels padded to a multiple of 8, zero padding and halo) and products.
// Slot 0 carries the unmasked operand (x*, resp. rp), slot 1 + b the operand of active-set slot b.
struct BfLayer {
    int Cip, Cop;             // input / output channels rounded up to 8
    long long PX, PR;         // elements of an input plane [Hp][Wp][Cip], of an output plane [Hpo][Wpo][Cop]
    uint16_t* X;              // [1 + cap][S][2][Hp][Wp][Cip] bf16: x* (slot 0), x* p_b (sign 0) and x* q_b (sign 1)
    uint16_t* R;              // [1 + cap][S][Hpo][Wpo][Cop] bf16: rp (slot 0), bz_b
    float* Drow;              // [(1 + cap) S][co][Ho Wo]: W x* (slot 0) and (W o I_b) x* per output neuron
    int nph;                  // stride phases (stride^2); input j = (c, y, x) is in phase (y + pad) % st, (x + pad) % st
    float* Dcol[CB_MAXPH];    // per phase [(1 + cap) S][2 ci][nY nX]: W+^T and W-^T products per input
    int Y0a[CB_MAXPH], X0a[CB_MAXPH], nY[CB_MAXPH], nX[CB_MAXPH];   // (y + pad) / st spans nY values from Y0a
};

struct DNet {
    int n;                 // affine layers; hidden layers k = 1..n-1
    int S, NT, NH, cap;    // subproblems, all neurons (layers 0..n-1), hidden neurons, max slots
    int RS;                // floats per Active Set record chunk (1 + cap rounded up to 4)
    int XT, AT;            // floats of input / output records per subproblem (all layers)
    DLayer L[CB_MAXL];
    const float* Wout;     // [S][n_{n-1}] property-folded output row
    const float* bout;     // [S]
    const BfLayer* bf;     // [n - 1] device array, BF16 form only (else null)
    int ball;              // 1: the input set is the ellipsoid inscribed in the box (l2 ball for equal
                           // half-widths); 0: the box
};

// Solver schedule constants (float32 copies prepared on the host from the double options).
struct DSched {
    int TM, TA, omega, vpa, maxcut;
    int ntab;              // entries in the per-step tables
    float b1, omb1, b2, omb2, eps;
    float lr_as_end;       // step size after the planned iterations
    float gamma0;
    int sp_init_steps;
    float sp_lr0, sp_lr1;
};

// Schedule of the Big-M / Active Set loop at global iteration it. Worked out once per iteration by the
// launch that advances the counter (and wherever the counter is set), and read by the passes: worked out
// per unit, its divisions and bias corrections were a third of the passes' instructions.
struct Step {
    int it;
    int as_phase;       // 0 Big-M, 1 Active Set
    int t;              // Active Set local iteration (-1 in Big-M)
    int b_new;          // slot added at this iteration (-1: none)
    int nadd_before;    // slots added before this iteration (global, before per-subproblem caps)
    float lr;
    float2 ib;                 // Adam's 1 / (1 - b1^n), 1 / (1 - b2^n) of alpha, beta_0, beta_1
    float2 sib[CB_MAXCUT];     // and of each slot, by its own step count
};

// Device state. Per-subproblem arrays are [S][NT], [S][NH] or [S][cap][NH].
struct DState {
    float *lo, *hi;                  // post-activation bounds, layer 0 = input box
    float *lhat, *uhat;              // pre-activation bounds (hidden)
    float *alpha, *beta0, *beta1;
    float *ma, *va, *m0, *v0, *m1, *v1;
    float *bs, *ms, *vs, *lam, *kap; // slots
    float *arec;                     // [S][AT] output records of each layer, RS floats per position
                                     // stored as RS / 4 planes of float4 over the positions:
                                     // -(alpha - beta1) + sum_b z_b beta_b, then (1 - z_b) beta_b
    float *xin;                      // [S][XT] input records of each layer, one float2 per position:
                                     // {x*, p_b bits | q_b bits << 8}
    float *lz;                       // [S][NH] sum_j W_ij Lcheck_ij (the all-ones mask's lambda)
    float *brad;                     // [S][NH] ellipsoid inputs: |W_i o e|_2 of layer 1's rows
    double *bnrm;                    // [S] ellipsoid inputs: |e o f_0|_2 of the last x_0* evaluation
    float *uz;                       // [S][NH] sum_j W_ij Ucheck_ij (kappa - b of a z = 0 row whose
                                     // inputs are all interior: the mask is then empty but for
                                     // fixed inputs, where Lcheck = Ucheck)
    uint8_t* efix;                   // [S][NT] l == u
    float *xval;                     // x* of the last evaluation [S][NT]
    float *fval;                     // f of the last evaluation [S][NT]
    uint8_t* zcur;                   // z* of the last evaluation [S][NH]
    uint8_t* xsnap[2];               // [S][NT] slot bitsets (double-buffered by addition count)
    uint8_t* zsnap[2];               // [S][NH]
    double* terms;                   // per-neuron bound terms [S][NT]
    double* best;                    // [S]
    const int* caps;                 // [S]
    int* ctr;                        // [0] AS iteration, [1] SP iteration, [2] SP-init step
    const float* lr_tab;             // [ntab] step size per global iteration
    const float* bc1_tab;            // [ntab] 1 / (1 - b1^step), step = index
    const float* bc2_tab;            // [ntab] 1 / (1 - b2^step)
    // Saddle Point
    float* spx[2];                   // [S][NT]
    float* spz[2];                   // [S][NH]
    float *Sb, *G, *C;               // [S][NH]
    float* P;                        // [S][NT], P_k at the inputs of layer k
    float *mua, *mub;                // [S][NH]
    float* xbar;                     // [S][NT]
    uint8_t* zbar;                   // [S][NH]
    float4* spin;                    // [S][XT] Saddle Point input records: two float4 planes per layer
    int* nfree;                      // [S][NH] nonzero weights of each row on free inputs
    uint8_t* sel;                    // [S][NH] selected beta of the conditional gradient (3 = none)
    float *ab, *b0i, *b1i;           // [S][NH] primal-init inner maximisers
    float* arow;                     // [S][NH] ab - b1i (primal-init row values for the col pass)
    int* status;                     // device error word
    Step* step;                      // schedule of the iteration ctr[0] names
};

__host__ __device__ inline int cb_additions_before(int t, const DSched& d) {
    if (t <= 0) return 0;
    int c;
    if (d.omega > 0) {
        int full = t / d.omega, rem = t % d.omega;
        c = full * d.vpa + (rem < d.vpa ? rem : d.vpa);
    } else {
        c = t < d.vpa ? t : d.vpa;
    }
    return c < d.maxcut ? c : d.maxcut;
}

__host__ __device__ inline int cb_slot_at(int t, const DSched& d) {
    int q, r;
    if (d.omega > 0) { q = t / d.omega; r = t % d.omega; }
    else { q = 0; r = t; }
    if (r >= d.vpa) return -1;
    int b = q * d.vpa + r;
    return b < d.maxcut ? b : -1;
}

// Active Set iteration at which slot b is added.
__host__ __device__ inline int cb_slot_added_at(int b, const DSched& d) {
    return d.omega > 0 ? (b / d.vpa) * d.omega + (b % d.vpa) : b;
}

// 1 / (1 - beta^step), the Adam bias corrections, from a table built in FP64 on the host.
__device__ __forceinline__ float inv_bias_corr(const float* tab, int ntab, int step, float beta) {
    return step < ntab ? tab[step] : 1.f / (1.f - powf(beta, (float)step));
}

// Works out *st.step for iteration `it`: lane b of a warp its slot b, lane 0 the rest.
__device__ inline void cb_set_step(int it, const DSched& d, const DState& st, int lane) {
    Step* s = st.step;
    const int t = it - d.TM;
    if (lane < CB_MAXCUT) {
        // a slot's first step is the iteration that adds it (values of slots not yet added are not read)
        const int n = max(0, t - cb_slot_added_at(lane, d)) + 1;
        s->sib[lane] = make_float2(inv_bias_corr(st.bc1_tab, d.ntab, n, d.b1), inv_bias_corr(st.bc2_tab, d.ntab, n, d.b2));
    }
    if (lane) return;
    s->it = it;
    s->as_phase = t >= 0;
    s->t = t >= 0 ? t : -1;
    s->b_new = t >= 0 ? cb_slot_at(t, d) : -1;
    s->nadd_before = t >= 0 ? cb_additions_before(t, d) : 0;
    s->lr = it < d.ntab ? st.lr_tab[it] : d.lr_as_end;
    s->ib = make_float2(inv_bias_corr(st.bc1_tab, d.ntab, it + 1, d.b1), inv_bias_corr(st.bc2_tab, d.ntab, it + 1, d.b2));
}

// Small batches launch their passes so that a pass is resident before the one before it has ended
// (launch_after on the host): it may start once every block of that one has, and waits here for all of its
// memory. First statement of such a kernel.
__device__ __forceinline__ void cb_after_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The schedule's scalars and a slot's bias corrections. Volatile loads: the launch before may write them,
// and an invariant load (__ldg) could move above the wait for it.
struct StepNow {
    int it, as_phase, t, b_new, nadd_before;
    float lr;
};
__device__ __forceinline__ int cb_load(const int* p) {
    int v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 cb_load(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ StepNow cb_step(const DState& st) {
    const Step* s = st.step;
    return {cb_load(&s->it), cb_load(&s->as_phase), cb_load(&s->t), cb_load(&s->b_new), cb_load(&s->nadd_before),
            __int_as_float(cb_load(reinterpret_cast<const int*>(&s->lr)))};
}
__device__ __forceinline__ float2 cb_bias(const DState& st) { return cb_load(&st.step->ib); }
__device__ __forceinline__ float2 cb_slot_bias(const DState& st, int b) { return cb_load(&st.step->sib[b]); }
