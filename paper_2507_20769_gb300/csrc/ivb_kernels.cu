// ivb_kernels.cu -- sm_103a kernels for Subdomain Lower Bounding (Section 3.1),
// tape interpreter (tile loop, decoding and reductions in ivb_bound_common.cuh):
//   Step 1: subdomain boxes decoded from the thread's global index (never
//           stored), dimension 0 fastest (Section 3.1.1)
//   Step 2: Mean Value Form (Definition 5) per subdomain: rigorous f(c) by an
//           interval sweep on [c,c], gradient enclosure by forward tangents or
//           by a reverse (adjoint) interval sweep
//   Step 3: refinement hull (Section 2.2 item iii) by warp shuffles and
//           ordered-integer atomicMin / atomicMax per node and output
// One persistent kernel serves any number of nodes: blocks grab tiles of the
// global subdomain index space from a device counter and map indices to nodes
// through the node queue's prefix sums.
#include <cmath>
#include <cstdint>
#include <cstring>

// the interpreter's warps are at different instructions: one copy of the long
// primitives keeps its code inside the instruction caches
#define IVB_HEAVY static __noinline__
#include "ivb_bound_common.cuh"
#include "ivb_internal.h"
#include "ivb_iv.cuh"
#include "ivb_kernels.h"

namespace ivb {

// ------------------------------------------------------------------ frame
// this lane's element 0 of its warp's frame (units 32 doubles apart)
struct Frame {
    double* p;
    __device__ __forceinline__ double ld(int u) const { return p[u * 32]; }
    __device__ __forceinline__ void st(int u, double v) const { p[u * 32] = v; }
    __device__ __forceinline__ iv get(int u) const { return mk(ld(u), ld(u + 1)); }
    __device__ __forceinline__ void put(int u, iv v) const { st(u, v.lo); st(u + 1, v.hi); }
    // by element (unit * 32)
    __device__ __forceinline__ iv at(uint32_t e) const { return mk(p[e], p[e + 32]); }
    __device__ __forceinline__ void to(uint32_t e, iv v) const { p[e] = v.lo; p[e + 32] = v.hi; }
};

struct SweepCtx {
    Frame F;
    const double* consts;
    int x_base;
};

// operand word (XIns)
__device__ __forceinline__ iv operand(const SweepCtx& C, uint32_t w) {
    const double* q = (w & kOpConst) ? C.consts : C.F.p;
    q += w & kOpIndex;
    const double lo = *q;
    return mk(lo, (w & kOpPoint) ? lo : q[32]);
}
// value reference of an output: record of `rec` units from `base` on, variable or constant
__device__ __forceinline__ iv load_val(const SweepCtx& C, uint32_t kind, uint32_t idx, int base, int rec) {
    if (kind == K_SLOT) return C.F.get(base + (int)idx * rec);
    if (kind == K_VAR) return C.F.get(C.x_base + 2 * (int)idx);
    const double k = __ldg(C.consts + idx);
    return mk(k, k);
}

__device__ __forceinline__ iv eval_value(uint32_t op, iv A, iv B) {
    switch (op) {
    case OP_ADD: return iv_add(A, B);
    case OP_SUB: return iv_sub(A, B);
    case OP_MUL: return iv_mul(A, B);
    case OP_DIV: return iv_div(A, B);
    case OP_SQR: return iv_sqr(A);
    case OP_SQRT: return iv_sqrt(A);
    case OP_EXP: return iv_exp(A);
    case OP_LOG: return iv_log(A);
    case OP_NEG: return iv_neg(A);
    }
    return entire();
}

// Interval values of a straight-line program. The interpreter is bound by the
// instructions around the arithmetic, not by the FP64 pipe (57 % busy): operands
// come resolved to addresses, the next instruction is fetched ahead, and a
// result that the next instruction reads stays in registers (configuration 3:
// 385 k -> 290 k instructions per warp of subdomains). Barriers that keep the
// warps on one handler cost more than they saved (13.1 ms without, 13.2 with one
// every 16 instructions, 15.7 with one each).
__device__ __noinline__ void run_values(const XIns* __restrict__ ins, int count, const SweepCtx C) {
    uint4 I = __ldg(reinterpret_cast<const uint4*>(ins));
    iv V = zero();
    for (int i = 0; i < count; ++i) {
        const uint4 next = __ldg(reinterpret_cast<const uint4*>(ins + i + 1));
        const uint32_t op = I.x & 31u;
        const iv A = (I.z & kOpLast) ? V : operand(C, I.z);
        const iv B = op > OP_DIV ? A : (I.w & kOpLast) ? V : operand(C, I.w);
        V = eval_value(op, A, B);
        C.F.to(I.y, V);
        I = next;
    }
}

// forward-mode sweep: value + tangent intervals per record (Section 3.2), only in
// the directions an entry depends on (masks of its operands from the host): the
// other tangents are zero, and terms with a zero tangent are exact -- adding
// [0,0] and multiplying by [0,0] change no value, so they are left out, as are
// products with a variable's own tangent [1,1]. The zero's sign may differ from the
// full sweep's; no bound depends on it. Of configuration 2's tangent products and
// sums a third are left (configuration 4, n = 16: an eighth): 12 nodes x 16^4 in
// 2.80 ms instead of 4.63.
__device__ void run_tangents(const XIns* __restrict__ ins, const uint2* __restrict__ masks, int count, const SweepCtx& C) {
    uint4 I = __ldg(reinterpret_cast<const uint4*>(ins));
    for (int i = 0; i < count; ++i) {
        const uint4 next = __ldg(reinterpret_cast<const uint4*>(ins + i + 1));
        const uint2 m = __ldg(masks + i);
        const uint32_t op = I.x & 31u;
        const bool avar = (I.x >> 7) & 1u, bvar = (I.x >> 8) & 1u;
        const uint32_t ea = I.z & ~kOpLast, eb = I.w & ~kOpLast;
        const iv A = operand(C, ea);
        const iv B = op > OP_DIV ? A : operand(C, eb);
        const iv V = eval_value(op, A, B);
        // quotient, sqr, sqrt, exp, log: one factor for every direction
        iv R = one();
        if (op >= OP_DIV && op != OP_NEG) {
            R = op == OP_DIV ? B : op == OP_EXP ? V : op == OP_LOG ? A : iv_twice(op == OP_SQR ? A : V);
            if (op != OP_EXP && op != OP_SQR) R = op == OP_DIV || gt0(R.lo) ? iv_recip(R) : entire();
        }
        // with x the factor of the operand's tangent: MUL B and A, DIV 1 and -V, sums 1 and +-1
        const iv xb = op == OP_DIV ? iv_neg(V) : A;
        for (uint32_t rest = m.x | m.y; rest; rest &= rest - 1u) {
            const int d = __ffs((int)rest) - 1;
            const bool ia = (m.x >> d) & 1u, ib = (m.y >> d) & 1u;
            const uint32_t off = 64u + 64u * (uint32_t)d;
            iv t = zero(), u = zero();
            if (ia) t = avar ? one() : C.F.at(ea + off);
            if (ib) u = bvar ? one() : C.F.at(eb + off);
            switch (op) {
            case OP_ADD:
            case OP_SUB:
                if (op == OP_SUB) u = iv_neg(u);
                t = !ib ? t : !ia ? u : iv_add(t, u);
                break;
            case OP_NEG: t = iv_neg(t); break;
            case OP_MUL:
                if (ia) t = avar ? B : iv_mul(t, B);
                if (ib) t = bvar && !ia ? A : iv_fma(xb, u, t);
                break;
            default:
                if (ib) t = iv_fma(xb, u, t);
                t = avar && !ib ? R : iv_mul(t, R);
            }
            C.F.to(I.y + off, t);
        }
        C.F.to(I.y, V);
        I = next;
    }
}

// reverse sweep of one output (reverse-mode interval AD). Operand a is updated
// before operand b. A product contribution x*y to a slot already written is
// accumulated with one directed rounding per end (iv_fma); the first write
// stores the product.
__device__ __noinline__ void run_reverse(const XRIns* __restrict__ rins, int count, const SweepCtx C) {
    const uint4* q = reinterpret_cast<const uint4*>(rins);
    uint4 I = __ldg(q), J = __ldg(q + 1);
    iv last = zero();   // the adjoint stored last
    for (int i = 0; i < count; ++i) {
        q += 2;
        const uint4 nextI = __ldg(q), nextJ = __ldg(q + 1);
        const uint32_t op = I.x & 31u;
        const iv W = (I.x & kAdjLast) ? last : C.F.at(I.y);
        if (op == OP_VAR) {
            C.F.to(I.z, iv_add(C.F.at(I.z), W));
        } else {
            const bool a_init = (I.x >> 5) & 1u, b_init = (I.x >> 6) & 1u, a_none = (I.x >> 7) & 1u, b_none = (I.x >> 8) & 1u;
            // contribution to operand a: W * ay (a_prod) or +-W; to operand b: bx * by or +-W
            iv ay = W, bx = W, by = W;
            bool prod = true;
            switch (op) {
            case OP_MUL:
                if (!a_none) ay = operand(C, J.y);
                if (!b_none) by = operand(C, J.x);
                break;
            case OP_DIV:
                ay = operand(C, J.y);
                if (!b_none) bx = iv_neg(iv_mul(W, C.F.at(J.z)));   // b gets -(W V) / B
                break;
            case OP_SQR:
            case OP_SQRT: ay = iv_twice(op == OP_SQR ? operand(C, J.x) : C.F.at(J.z)); break;
            case OP_EXP: ay = C.F.at(J.z); break;
            case OP_LOG: ay = operand(C, J.x); break;
            default: prod = false;
            }
            if (op == OP_DIV || op == OP_SQRT || op == OP_LOG) {
                ay = op == OP_DIV || gt0(ay.lo) ? iv_recip(ay) : entire();
                by = ay;
            }
            // a first contribution is fused with [0,0]: the bits of the product
            if (!a_none) {
                if (prod) last = iv_fma(W, ay, a_init ? zero() : C.F.at(I.z));
                else {
                    last = op == OP_NEG ? iv_neg(W) : W;
                    if (!a_init) last = iv_add(C.F.at(I.z), last);
                }
                C.F.to(I.z, last);
            }
            if (!b_none) {
                if (prod) last = iv_fma(bx, by, b_init ? zero() : C.F.at(I.w));
                else {
                    last = op == OP_SUB ? iv_neg(W) : W;
                    if (!b_init) last = iv_add(C.F.at(I.w), last);
                }
                C.F.to(I.w, last);
            }
        }
        I = nextI;
        J = nextJ;
    }
}

// --------------------------------------------------------------- the kernel
template <int MODE>
__global__ void __launch_bounds__(512, 2) k_bound(const KParams P) {
    extern __shared__ double smem[];
    const ProgDesc& G = *P.prog;
    const int n = G.n, n_out = G.n_out;
    const FrameLayout L = G.L;
    SweepCtx C;
    const size_t warp = threadIdx.x >> 5;
    if (P.frame_in_smem) C.F.p = smem + warp * P.frame_units * 32;
    else C.F.p = P.gframe + ((size_t)blockIdx.x * (blockDim.x >> 5) + warp) * P.frame_units * 32;
    C.F.p += threadIdx.x & 31;
    C.consts = G.consts;
    C.x_base = L.x_base;

    // adjoint modes: the outputs of a subdomain shared among warp groups (KParams::groups)
    constexpr bool kAdj = MODE == KM_ADJ_STORE || MODE == KM_ADJ_REDUCE;
    const int groups = kAdj ? P.groups : 1;
    const int per = (int)blockDim.x / groups, first_o = kAdj ? (int)threadIdx.x / per : 0;
    __shared__ unsigned char s_fl[512];
    tile_loop_per(P, per, [&](const Sub& s) {
        const long long g = s.g;
        const bool valid = s.valid;
        if (valid) {
            // ---- Step 1: decode X_k and c
            unsigned int kk = s.k;
            for (int i = 0; i < n; ++i) {
                iv X;
                double c;
                decode_dim(s.rec, n, i, kk, X, c);
                C.F.put(L.x_base + 2 * i, X);
                C.F.st(L.c_base + i, c);
            }
            // ---- Step 2a: rigorous point value f(c) of every output
            if (groups == 1) run_values(G.xins + G.pt_begin, G.pt_count, C);
            for (int o = 0; o < n_out && groups == 1; ++o) {
                const uint32_t kind = G.pt_out_kind[o], ref = G.pt_out_ref[o];
                const double c = kind == K_VAR ? C.F.ld(L.c_base + (int)ref) : 0.0;
                C.F.put(L.fc_base + 2 * o, kind == K_VAR ? mk(c, c) : load_val(C, kind, ref, L.phase_base, 2));
            }
        }
        // ---- Step 2b: gradient enclosures and the Mean Value Form, output by output.
        // With the natural interval extension alone (form 1) a reduce launch needs no
        // gradients: only the value sweep over X_k.
        const bool nie_only = (MODE == KM_FWD_REDUCE || MODE == KM_ADJ_REDUCE) && P.form == 1;
        unsigned fl = 0;   // bit 0: an output proves the subdomain infeasible; bit 1: its centre is not certified feasible
        double obj_lo = from_bits(0x7FF0000000000000LL), obj_c = obj_lo;
        if (MODE == KM_FWD_REDUCE || MODE == KM_FWD_STORE) {
            if (valid) {
                if (nie_only) run_values(G.xtan, G.tan_count, C);
                else run_tangents(G.xtan, G.tan_mask, G.tan_count, C);
            }
        }
        for (int o = first_o; o < n_out; o += groups) {
            iv F = zero(), Fc = zero();
            if (valid) {
                if (groups > 1) {   // f(c) of this output alone
                    const AdjProgram& A = G.adj[o];
                    const int tb = L.phase_base + 2 * n + 2 * A.adj_slots;
                    run_values(G.xcone + A.fw_begin, A.fw_count, C);
                    const double c = A.out_kind_ref == K_VAR ? C.F.ld(L.c_base + A.out_ref) : 0.0;
                    Fc = A.out_kind_ref == K_VAR ? mk(c, c) : load_val(C, A.out_kind_ref, A.out_ref, tb, 2);
                } else {
                    Fc = C.F.get(L.fc_base + 2 * o);
                }
                if (G.out_kind[o] == OUT_INEQ && !le0(Fc.hi)) fl |= 2u;
                if (o == G.obj) obj_c = Fc.hi;
            }
            if (valid && nie_only) {
                iv nie;
                if (MODE == KM_FWD_REDUCE) {
                    nie = load_val(C, G.tan_out_kind[o], G.tan_out_ref[o], L.phase_base, L.tan_rec);
                } else {
                    const AdjProgram& A = G.adj[o];
                    const int tb = L.phase_base + 2 * n + 2 * A.adj_slots;
                    run_values(G.xins + A.fw_begin, A.fw_count, C);
                    nie = load_val(C, A.out_kind_ref, A.out_ref, tb, 2);
                }
                F = final_form(1, nie, nie);
                if (excludes_feasible(G.out_kind[o], F)) fl |= 1u;
                if (o == G.obj) obj_lo = F.lo;
            } else if (valid) {
                iv nie;
                int gunit, gstride;  // gradient of this output: unit of G_0 and stride (0: constant/variable)
                uint32_t dirs = ~0u;  // directions it depends on
                if (MODE == KM_FWD_REDUCE || MODE == KM_FWD_STORE) {
                    const int rec = L.tan_rec;
                    const uint32_t kind = G.tan_out_kind[o], ref = G.tan_out_ref[o];
                    nie = load_val(C, kind, ref, L.phase_base, rec);
                    dirs = G.tan_out_mask[o];
                    if (kind == K_SLOT) { gunit = L.phase_base + (int)ref * rec + 2; gstride = 2; }
                    else { gunit = (kind == K_VAR) ? (int)ref : -1; gstride = 0; }
                } else {
                    const AdjProgram& A = G.adj[o];
                    const int gb = L.phase_base, ab = gb + 2 * n, tb = ab + 2 * A.adj_slots;
                    run_values(G.xins + A.fw_begin, A.fw_count, C);
                    for (int i = 0; i < n; ++i) C.F.put(gb + 2 * i, zero());
                    if (A.out_wslot >= 0) C.F.put(ab + 2 * A.out_wslot, one());
                    run_reverse(G.xrins + A.rv_begin, A.rv_count, C);
                    nie = load_val(C, A.out_kind_ref, A.out_ref, tb, 2);
                    gunit = gb;
                    gstride = 2;
                }
                // Mean Value Form (Definition 5): f(c) + sum_i G_i (X_i - c_i), left to right
                iv mvf = Fc;
                for (int i = 0; i < n; ++i) {
                    const bool dep = (dirs >> i) & 1u;
                    const iv Gi = !dep ? zero() : gstride ? C.F.get(gunit + 2 * i) : one();
                    if (dep) mvf = mvf_term(mvf, Gi, C.F.get(L.x_base + 2 * i), C.F.ld(L.c_base + i));
                    else mvf.hi = is0(mvf.hi) ? 0.0 : mvf.hi;   // mvf + [0,0], in iv_fma's bits
                    if ((MODE == KM_FWD_STORE || MODE == KM_ADJ_STORE) && P.outG) {
                        const long long q0 = g - P.store_first_g;
                        double* q = P.outG + ((size_t)q0 * n_out + o) * n * 2 + 2 * i;
                        q[0] = Gi.lo;
                        q[1] = Gi.hi;
                    }
                }
                F = final_form(P.form, mvf, nie);
                if (excludes_feasible(G.out_kind[o], F)) fl |= 1u;
                if (o == G.obj) obj_lo = F.lo;
            }
            if (MODE == KM_FWD_STORE || MODE == KM_ADJ_STORE) {
                if (valid) {
                    const long long q0 = g - P.store_first_g;
                    P.outF[((size_t)q0 * n_out + o) * 2] = F.lo;
                    P.outF[((size_t)q0 * n_out + o) * 2 + 1] = F.hi;
                    if (P.outFc) {
                        P.outFc[((size_t)q0 * n_out + o) * 2] = Fc.lo;
                        P.outFc[((size_t)q0 * n_out + o) * 2 + 1] = Fc.hi;
                    }
                }
            } else {
                // ---- Step 3: refinement hull per node and output
                reduce_output(P, s, n_out, o, F);
            }
        }
        if (MODE == KM_FWD_REDUCE || MODE == KM_ADJ_REDUCE) {
            if (groups > 1) {   // the objective's group needs every output's tests
                s_fl[threadIdx.x] = (unsigned char)fl;
                __syncthreads();
                for (int h = 0; h < groups; ++h) fl |= s_fl[h * per + (int)threadIdx.x % per];
                __syncthreads();
            }
            if (G.obj % groups == first_o) {
                double ub = from_bits(0x7FF0000000000000LL);
                if (valid && !G.has_eq && !(fl & 2u)) ub = obj_c;
                if (fl & 1u) obj_lo = from_bits(0x7FF0000000000000LL);
                reduce_extras(P, s, n_out, ub, obj_lo);
            }
        }
    });
}

}  // namespace ivb
namespace ivb {

// ------------------------------------------------------------ node results
__global__ void k_init_keys(unsigned long long* keys, const char* queue, int n_out, unsigned long long* counter) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0ULL;
    const int n_nodes = (int)reinterpret_cast<const long long*>(queue)[0];
    const int K = 2 * n_out + 2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes * K; i += gridDim.x * blockDim.x) {
        const int slot = i % K;
        const bool is_max = slot >= n_out && slot < 2 * n_out;
        keys[i] = is_max ? 0ULL : ~0ULL;
    }
}

// Section 3.1 Step 3 and pruning: lb = lower end of the objective's
// refinement (or the filtered minimum), infeasible when an inequality's lower
// end is > 0 or an equality's refinement excludes 0.
__global__ void k_finalize(FinalizeParams F) {
    if (F.out_in_header) {
        const QueueHeader& H = *reinterpret_cast<const QueueHeader*>(F.queue);
        F.lb = H.lb; F.inf = H.inf; F.ub = H.ub; F.minlo = H.minlo; F.maxhi = H.maxhi;
    }
    const int nd = blockIdx.x * blockDim.x + threadIdx.x;
    const int n_nodes = (int)reinterpret_cast<const long long*>(F.queue)[0];
    if (nd >= n_nodes) return;
    const int K = 2 * F.n_out + 2;
    const unsigned long long* k = F.keys + (size_t)nd * K;
    uint8_t inf = 0;
    for (int o = 0; o < F.n_out; ++o) {
        const double lo = unkey(k[o]), hi = unkey(k[F.n_out + o]);
        if (F.out_kind[o] == OUT_INEQ && gt0(lo)) inf = 1;
        if (F.out_kind[o] == OUT_EQ && (gt0(lo) || lt0(hi))) inf = 1;
        if (F.minlo) F.minlo[(size_t)nd * F.n_out + o] = lo;
        if (F.maxhi) F.maxhi[(size_t)nd * F.n_out + o] = hi;
    }
    double lb = unkey(k[F.obj]);
    if (F.filter) {
        lb = unkey(k[2 * F.n_out + 1]);
        if (isinf_(lb) && gt0(lb)) inf = 1;
    }
    if (F.lb) F.lb[nd] = lb;
    if (F.inf) F.inf[nd] = inf;
    if (F.ub) F.ub[nd] = unkey(k[2 * F.n_out]);
}

// ------------------------------------------------- round-to-nearest gradients
// Point value and reverse-mode gradient of every output at x (plain double, same
// local partials as the interval rules), one thread per point. Bound by the FP64
// pipe while quotients, roots, exp and log ran there (three quarters of its FP64
// instructions; configuration 4, 100003 points: 674 us), which is why these are
// in fixed point (ivb_fixed.cuh): 321 us now, and 684 -> 329 us for value and
// gradient through autograd. Now bound by latency: 44 k instructions per warp of
// points, waiting on frame loads and long chains. x goes through the frame, so
// that the strided reads of the caller's array happen once.
__device__ __forceinline__ double point_operand(const double* f, const double* consts, uint32_t w) {
    const double* q = (w & kOpConst) ? consts : f;
    return q[w & kOpIndex];
}

__global__ void __launch_bounds__(64, 16) k_point_grad(const ProgDesc* __restrict__ prog, long long n_points,
                                                      const double* __restrict__ X, double* f, double* grad,
                                                      double* gframe, int frame_units) {
    const ProgDesc& G = *prog;
    const int n = G.n, n_out = G.n_out;
    const double* const consts = G.consts;
    double* const F = gframe + ((size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * frame_units * 32 + (threadIdx.x & 31);
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n_points;
         p += (long long)gridDim.x * blockDim.x) {
        for (int i = 0; i < n; ++i) F[i * 32] = X[(size_t)p * n + i];
        for (int o = 0; o < n_out; ++o) {
            const AdjProgram& A = G.adj[o];
            const int ab = 2 * n, tb = ab + A.adj_slots;
            const uint4* q = reinterpret_cast<const uint4*>(G.pins + A.fw_begin);
            uint4 I = __ldg(q);
            double v = 0.0;
            for (int i = 0; i < A.fw_count; ++i) {
                const uint4 next = __ldg(++q);
                const uint32_t op = I.x;
                const double a = (I.z & kOpLast) ? v : point_operand(F, consts, I.z);
                const double b = op > OP_DIV ? a : (I.w & kOpLast) ? v : point_operand(F, consts, I.w);
                switch (op) {
                case OP_ADD: v = __dadd_rn(a, b); break;
                case OP_SUB: v = __dsub_rn(a, b); break;
                case OP_MUL:
                case OP_SQR: v = __dmul_rn(a, b); break;
                case OP_DIV: v = div_rn(a, b); break;
                case OP_SQRT: v = sqrt_rn(a); break;
                case OP_EXP: v = exp_rn(a); break;
                case OP_LOG: v = log_rn(a); break;
                case OP_NEG: v = -a; break;
                default: v = __longlong_as_double(0x7FF8000000000000LL);
                }
                F[I.y] = v;
                I = next;
            }
            const int r = A.out_ref;
            f[(size_t)p * n_out + o] = A.out_kind_ref == K_CONST ? __ldg(consts + r) : F[(A.out_kind_ref == K_VAR ? r : tb + r) * 32];
            if (!grad) continue;
            for (int i = 0; i < n; ++i) F[(n + i) * 32] = 0.0;
            if (A.out_wslot >= 0) F[(ab + A.out_wslot) * 32] = 1.0;
            q = reinterpret_cast<const uint4*>(G.prins + A.rv_begin);
            uint4 J = __ldg(q + 1);
            I = __ldg(q);
            double last = 0.0;   // the adjoint stored last
            for (int i = 0; i < A.rv_count; ++i) {
                q += 2;
                const uint4 nextI = __ldg(q), nextJ = __ldg(q + 1);
                const uint32_t op = I.x & 31u;
                const double w = (I.x & kAdjLast) ? last : F[I.y];
                if (op == OP_VAR) {
                    F[I.z] = __dadd_rn(F[I.z], w);
                } else {
                    const bool a_init = (I.x >> 5) & 1u, b_init = (I.x >> 6) & 1u;
                    const bool a_none = (I.x >> 7) & 1u, b_none = (I.x >> 8) & 1u;
                    double ca = w, cb = w;
                    switch (op) {
                    case OP_SUB: cb = -w; break;
                    case OP_NEG: ca = -w; break;
                    case OP_MUL:
                        ca = __dmul_rn(w, point_operand(F, consts, J.y));
                        cb = __dmul_rn(w, point_operand(F, consts, J.x));
                        break;
                    case OP_SQR: ca = __dmul_rn(w, __dmul_rn(2.0, point_operand(F, consts, J.x))); break;
                    case OP_EXP: ca = __dmul_rn(w, F[J.z]); break;
                    case OP_DIV:
                    case OP_SQRT:
                    case OP_LOG: {
                        const double r = rcp_rn(op == OP_DIV ? point_operand(F, consts, J.y) :
                                                op == OP_LOG ? point_operand(F, consts, J.x) : __dmul_rn(2.0, F[J.z]));
                        ca = __dmul_rn(w, r);
                        if (op == OP_DIV) cb = -__dmul_rn(__dmul_rn(w, F[J.z]), r);
                    } break;
                    }
                    if (!a_none) {
                        last = a_init ? ca : __dadd_rn(F[I.z], ca);
                        F[I.z] = last;
                    }
                    if (!b_none) {
                        last = b_init ? cb : __dadd_rn(F[I.w], cb);
                        F[I.w] = last;
                    }
                }
                I = nextI;
                J = nextJ;
            }
            for (int i = 0; i < n; ++i) grad[((size_t)p * n_out + o) * n + i] = F[(n + i) * 32];
        }
    }
}

// ------------------------------------------------------------ test hook
// opcode: tape opcodes of the interval operations, 100 for the reciprocal,
// 101..104 for +, -, *, sqr with every endpoint operation emulated on the
// integer pipes (policy 15 of ivb_iv.cuh)
__device__ __forceinline__ iv eval_hook(int opcode, iv X, iv Y) {
    switch (opcode) {
    case 100: return iv_recip(X);
    case 101: return iv_add_t<15>(X, Y);
    case 102: return iv_sub_t<15>(X, Y);
    case 103: return iv_mul_t<15>(X, Y);
    case 104: return iv_sqr_t<15>(X);
    }
    return eval_value((uint32_t)opcode, X, Y);
}

__global__ void k_eval_op(int opcode, long long n, const double* __restrict__ x, const double* __restrict__ y,
                          double* r) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const iv X = mk(x[2 * i], x[2 * i + 1]);
        const iv Y = y ? mk(y[2 * i], y[2 * i + 1]) : X;
        const iv R = opcode == 105 ? iv_fma(X, Y, mk(r[2 * i], r[2 * i + 1])) : eval_hook(opcode, X, Y);
        r[2 * i] = R.lo;
        r[2 * i + 1] = R.hi;
    }
}

cudaError_t launch_eval_op(int opcode, long long n, const double* x, const double* y, double* r, cudaStream_t s) {
    const int block = 256;
    const long long g = (n + block - 1) / block;
    k_eval_op<<<(int)(g < 4096 ? g : 4096), block, 0, s>>>(opcode, n, x, y, r);
    return cudaGetLastError();
}

// ------------------------------------------------------------ own-primitive probe
// throughput of this library's directed primitives (ivb_fp64x.cuh), the
// same shape as ivb_probe.cu: 8 independent chains per thread
template <int W>
__global__ void k_own_probe(double* out, double seed, int iters) {
    double x[8];
    const double y = seed + threadIdx.x * 1e-12;
    for (int j = 0; j < 8; ++j) x[j] = 1.5 + j * 1e-3 + threadIdx.x * 1e-9;
    for (int i = 0; i < iters; ++i) {
        // factors and addends that keep the multiply / add chains near 1.5
        const double f = (i & 1) ? 1.0000001192092896 : 0.99999988079071045;
        const double d = (i & 1) ? 0.0009765625 : -0.0009765625;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (W == 0) x[j] = rcp_dir(x[j], false);
            if (W == 1) x[j] = div_dir(y, x[j], false);
            if (W == 2) x[j] = sqrt_dir(x[j] * 3.1, false);   // one multiply keeps x off powers of two
            if (W == 3) x[j] = exp_dir(-x[j], false);
            if (W == 4) x[j] = __dadd_rn(log_dir(x[j], false), 2.0);
            // integer-pipe emulation (ivb_emu.cuh) alone, and beside the FP64 pipe (half the chains each)
            if (W == 5) x[j] = mul_ru_emu(x[j], f);
            if (W == 6) x[j] = (j & 1) ? mul_ru_emu(x[j], f) : __dmul_ru(x[j], f);
            if (W == 7) x[j] = add_ru_emu(x[j], d);
            if (W == 8) x[j] = (j & 1) ? add_ru_emu(x[j], d) : __dadd_ru(x[j], d);
        }
    }
    double acc = 0.0;
    for (int j = 0; j < 8; ++j) acc += x[j];
    out[blockIdx.x * blockDim.x + threadIdx.x] = acc;
}

template <int W>
static cudaError_t own_probe_run(double* out, int grid, int block, int iters, float* ms) {
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_own_probe<W><<<grid, block>>>(out, 1.0000001, iters / 4 + 1);
    cudaEventRecord(a);
    k_own_probe<W><<<grid, block>>>(out, 1.0000001, iters);
    cudaEventRecord(b);
    cudaError_t e = cudaEventSynchronize(b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

cudaError_t run_own_probe(int which, double* out, int grid, int block, int iters, float* ms) {
    cudaError_t e = init_math_tables();
    if (e != cudaSuccess) return e;
    switch (which) {
    case 0: return own_probe_run<0>(out, grid, block, iters, ms);
    case 1: return own_probe_run<1>(out, grid, block, iters, ms);
    case 2: return own_probe_run<2>(out, grid, block, iters, ms);
    case 3: return own_probe_run<3>(out, grid, block, iters, ms);
    case 4: return own_probe_run<4>(out, grid, block, iters, ms);
    case 5: return own_probe_run<5>(out, grid, block, iters, ms);
    case 6: return own_probe_run<6>(out, grid, block, iters, ms);
    case 7: return own_probe_run<7>(out, grid, block, iters, ms);
    default: return own_probe_run<8>(out, grid, block, iters, ms);
    }
}

// exp/log tables in extended precision on the host (long double: 64-bit
// significand on x86-64, binary128 on AArch64)
cudaError_t math_tables_address(void** ptr, size_t* bytes) {
    *bytes = sizeof(MathTables);
    return cudaGetSymbolAddress(ptr, g_math);
}

cudaError_t init_math_tables() {
    static bool done[256] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 256 && done[dev]) return cudaSuccess;
    static MathTables h;
    const long double two32 = 4294967296.0L;
    for (int j = 0; j < kExpTab; ++j)
        h.exp[j] = (fx64)(exp2l((long double)j / kExpTab) * (two32 * (two32 / 4)) + 0.5L);
    // 1023 ln2 = 710 - frac 2^-64
    const fx64 frac = 0xE91238B093E8CA84ULL;
    for (int j = 0; j < kLogTab; ++j) {
        h.log[j].c = (fx32)(((1u << 30) + (kLogTab + j) - 1) / (kLogTab + j));
        const fx64 v = (fx64)(-logl((long double)h.log[j].c / 1048576.0L) * (two32 * two32) + 0.5L);
        h.log[j].frac = v + frac;
        h.log[j].ip = -710 + (h.log[j].frac < v ? 1 : 0);
    }
    for (int k = 0; k < kNearTab; ++k) {
        // the two intervals next to 1 use c = 1 so that r = y - 1 is exact
        const int j = k - kNearTab / 2;
        const long double F = j >= 0 ? 1.0L + (j + 0.5L) / 2048 : (1.0L + (2048 + j + 0.5L) / 2048) / 2;
        const double c = j == 0 || j == -1 ? 1.0 : (double)(1.0L / F);
        const long double L = -logl((long double)c);
        h.near1[k].c = c;
        h.near1[k].hi = (double)L;
        h.near1[k].lo = (double)(L - (long double)h.near1[k].hi);
    }
    e = cudaMemcpyToSymbol(g_math, &h, sizeof(h));
    if (e == cudaSuccess && dev >= 0 && dev < 256) done[dev] = true;
    return e;
}

// ------------------------------------------------------------ host wrappers
static const void* bound_fn(int mode) {
    switch (mode) {
    case KM_FWD_REDUCE: return (const void*)k_bound<KM_FWD_REDUCE>;
    case KM_ADJ_REDUCE: return (const void*)k_bound<KM_ADJ_REDUCE>;
    case KM_FWD_STORE: return (const void*)k_bound<KM_FWD_STORE>;
    default: return (const void*)k_bound<KM_ADJ_STORE>;
    }
}

cudaError_t set_bound_smem_limit(int mode, int bytes) {
    return cudaFuncSetAttribute(bound_fn(mode), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

int occupancy_blocks(int mode, int block, size_t smem) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, bound_fn(mode), block, smem) != cudaSuccess) return 0;
    return nb;
}

cudaError_t launch_bound(int mode, const KParams& P, int grid, int block, size_t smem, cudaStream_t s) {
    switch (mode) {
    case KM_FWD_REDUCE: k_bound<KM_FWD_REDUCE><<<grid, block, smem, s>>>(P); break;
    case KM_ADJ_REDUCE: k_bound<KM_ADJ_REDUCE><<<grid, block, smem, s>>>(P); break;
    case KM_FWD_STORE: k_bound<KM_FWD_STORE><<<grid, block, smem, s>>>(P); break;
    default: k_bound<KM_ADJ_STORE><<<grid, block, smem, s>>>(P); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_init_keys(unsigned long long* keys, const char* queue, int max_nodes, int n_out,
                             unsigned long long* counter, cudaStream_t s) {
    const int total = max_nodes * (2 * n_out + 2);
    const int block = 256, grid = (total + block - 1) / block < 1024 ? (total + block - 1) / block : 1024;
    k_init_keys<<<grid, block, 0, s>>>(keys, queue, n_out, counter);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const FinalizeParams& F, cudaStream_t s) {
    const int block = 128, grid = (F.max_nodes + block - 1) / block;
    k_finalize<<<grid, block, 0, s>>>(F);
    return cudaGetLastError();
}

cudaError_t launch_point_grad(const ProgDesc* prog, int n, int n_out, int frame_units, long long n_points,
                              const double* x, double* f, double* grad, double* gframe, int grid, int block,
                              cudaStream_t s) {
    (void)n; (void)n_out;
    k_point_grad<<<grid, block, 0, s>>>(prog, n_points, x, f, grad, gframe, frame_units);
    return cudaGetLastError();
}

}  // namespace ivb
