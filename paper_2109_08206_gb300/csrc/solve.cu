// Barzilai-Borwein projected gradient descent (BBPGD) on the CQP
//     min_gamma  1/2 gamma^T (D^T M D) gamma + q^T gamma,   gamma >= 0
// (Appendix Eq. suppcqpdef; Section "Instantiation in a massively parallel
// computing environment": each iteration costs one gradient
// grad f = D^T M D gamma + q, i.e. O(N_u) work).
//
// The paper defers the details of its BBPGD to earlier work, so the
// iteration follows the published projected BB method (Barzilai & Borwein
// 1988; projected form as in Dai & Fletcher 2005):
//   gamma_{k+1} = max(0, gamma_k - alpha_k g_k),
//   s_k = gamma_{k+1} - gamma_k, y_k = g_{k+1} - g_k (= A s_k),
//   alpha_{k+1} from the pair (s_{k-1}, y_{k-1}) of the iteration before,
//     s.s / s.y and s.y / y.y in turn (alternating BB1/BB2): the
//     Barzilai-Borwein step taken one iteration late, a gradient method with
//     retards (Friedlander, Martinez, Molina & Raydan, SIAM J. Numer. Anal.
//     36, 1999), which lets the one-barrier solver below (at most one grid
//     barrier an iteration) form the step length from sums that arrive while
//     another phase runs; every solver kernel uses it, so all of them run
//     one method;
//   alpha_0 = pi.pi / pi.A.pi for the projected gradient pi at gamma_0, for
//   the first two steps and whenever s.y <= 0 or the step is not finite.
// Stop when (h/D) max |pi_c| <= tol (pi the projected gradient) or after
// max_iter iterations.
//
// One persistent cooperative kernel runs the whole loop, one block per SM.
// Rods are numbered in cell order; block b owns an even share of rods
// [r0, r1) and the constraints they own [c0, c1) (owner = lower-ranked end).
// When they fit, the block keeps its own constraints' records, q, gamma and
// g, and its rods' axes and velocities in shared memory for the whole solve
// (at 1e5 rods the mixed working set, about 30 MB, spreads over the SMs'
// shared memory); global memory then carries what other blocks read: the
// velocities, and the state of constraints whose other rod is another
// block's (the rest of the state is written once when the solve ends).
// Without that fit every block works from the global arrays.  Per
// iteration:
//   phase A (one thread per rod, rods taken in ascending order of their
//     entry counts so that a warp's loops have similar lengths):
//     delta_{k+1} of every constraint touching the rod is formed on the fly
//     from (delta_k, g_k, gamma_ref) and alpha_k, summed into the rod's
//     force and torque F = D delta (owned range contiguous, other-side list
//     in CSR order), and dU = M F is stored;
//   grid barrier;
//   phase B (one thread per owned constraint): delta_{k+1} again (same
//     inputs and rounding), g_{k+1} = gref + D^T dU, and the partial sums
//     s.s, s.y, y.y and max |pi| (per thread, per warp and per block in a
//     fixed order);
//   grid barrier; warps 0-3 of every block then reduce the per-block
//     partials in the same fixed order, so all blocks take identical step
//     decisions.
// Two grid barriers per iteration.  Each barrier wait is bounded in time
// and in polls; a wait that runs out raises ALENS_ERR_TIMEOUT in the device
// status word and every block leaves.
//
// Global layout: the state (delta, g, gamma_ref, gamma_lo) of each
// constraint in two ping-pong [m][4] buffers, U as [rod][6], D records SoA
// [9][m] in owner-major order.
// T = double (float64 plain) or float (mixed: the D, M, D^T work, the sums
// and the step sizes in float32).  max |pi| is exact in either, and the
// stopping test takes the float64 decision (h/D) max |pi| <= tol in both:
// in float32 as max |pi| <= pi_tol, the largest float for which the float64
// product stays within tol.  The per-iteration reductions and decisions stay
// off float64 in the mixed solver because this part's float64 latency is
// about ten times float32's (an add 62 cycles, a divide 561).
#include <cooperative_groups.h>
#include <float.h>

#include <algorithm>
#include <cmath>
#include <limits>
#include <type_traits>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace alens {

// CSR entries whose loads a thread issues together (float64 values need the
// registers twice over)
template <typename T> struct Batch { static constexpr int v = 1; };
constexpr int kRefresh = 64;   // float32 iterations between reference refreshes

template <typename T> struct V2;
template <> struct V2<float> { using t = float2; };
template <> struct V2<double> { using t = double2; };

template <typename T>
__device__ __forceinline__ void ld_pair(const T* p, int c, T& a, T& b)
{
    typename V2<T>::t v = reinterpret_cast<const typename V2<T>::t*>(p)[c];
    a = v.x;
    b = v.y;
}

template <typename T>
__device__ __forceinline__ void ld_u6(const T* U, int i, T u[6])
{
    const typename V2<T>::t* p = reinterpret_cast<const typename V2<T>::t*>(U + 6 * (size_t)i);
    typename V2<T>::t a = p[0], b = p[1], c = p[2];
    u[0] = a.x; u[1] = a.y; u[2] = b.x; u[3] = b.y; u[4] = c.x; u[5] = c.y;
}

// Other-side arms of CSR entry k, packed as [m][8] (e, arm x e, 2 pad).
__device__ __forceinline__ void ld_arm(const float* qe, int k, float v[6])
{
    const float4 a = __ldg(reinterpret_cast<const float4*>(qe) + 2 * (size_t)k);
    const float2 b = __ldg(reinterpret_cast<const float2*>(qe) + 4 * (size_t)k + 2);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y;
}
__device__ __forceinline__ void ld_arm(const double* qe, int k, double v[6])
{
    const double2* p = reinterpret_cast<const double2*>(qe) + 4 * (size_t)k;
    const double2 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y; v[4] = c.x; v[5] = c.y;
}

template <typename T>
__device__ __forceinline__ void st_u6(T* U, int i, const T u[6])
{
    typename V2<T>::t* p = reinterpret_cast<typename V2<T>::t*>(U + 6 * (size_t)i);
    typename V2<T>::t a, b, c;
    a.x = u[0]; a.y = u[1]; b.x = u[2]; b.y = u[3]; c.x = u[4]; c.y = u[5];
    p[0] = a; p[1] = b; p[2] = c;
}

// Constraint state (delta, g, gamma_ref, gamma_lo) of constraint c in a
// [m][4] buffer: one vector load (float32) or two (float64).  The iterate
// is gamma = gamma_ref + gamma_lo + delta: in float32 (gamma_ref, gamma_lo)
// is an unevaluated sum carrying about 48 bits (gamma_lo is 0 in float64).
__device__ __forceinline__ void ld_state(const float* p, int c, float& d, float& g, float& gr, float& gl)
{
    const float4 v = reinterpret_cast<const float4*>(p)[c];
    d = v.x; g = v.y; gr = v.z; gl = v.w;
}
__device__ __forceinline__ void ld_state(const double* p, int c, double& d, double& g, double& gr, double& gl)
{
    const double2* q = reinterpret_cast<const double2*>(p) + 2 * (size_t)c;
    const double2 a = q[0], b = q[1];
    d = a.x; g = a.y; gr = b.x; gl = b.y;
}
__device__ __forceinline__ float gl_of_state(const float* p, int c) { return p[4 * (size_t)c + 3]; }
__device__ __forceinline__ double gl_of_state(const double* p, int c) { return p[4 * (size_t)c + 3]; }

// (delta, g) and (gamma_ref, gamma_lo) halves of a state
template <typename T>
__device__ __forceinline__ void st_dg(T* p, int c, T d, T g)
{
    typename V2<T>::t v;
    v.x = d; v.y = g;
    reinterpret_cast<typename V2<T>::t*>(p)[2 * (size_t)c] = v;
}
template <typename T>
__device__ __forceinline__ void st_ref(T* p, int c, T gr, T gl)
{
    typename V2<T>::t v;
    v.x = gr; v.y = gl;
    reinterpret_cast<typename V2<T>::t*>(p)[2 * (size_t)c + 1] = v;
}

// Sums that are never fused with a product they add (the compiler may
// otherwise take a + (rounded p q) as fma(p, q, a), as it likes in each
// place, which breaks the error-free transformations below).
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// Exact sum: a + b = s + e.
template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T& s, T& e)
{
    s = add_rn(a, b);
    const T bb = add_rn(s, -a);
    e = add_rn(add_rn(a, -add_rn(s, -bb)), add_rn(b, -bb));
}

// Sum-of-products accumulator.  COMP (float32 reference passes): an
// unevaluated (hi, lo) pair fed by error-free transformations - the product
// split through one FMA, the sum through TwoSum - so large contact forces
// that cancel on a rod, or q and D^T U that cancel in a gradient entry, lose
// no digits.  Otherwise a plain sum.
template <typename T, bool COMP>
struct Acc {
    T hi, lo;
    __device__ __forceinline__ void init(T v) { hi = v; lo = T(0); }
    __device__ __forceinline__ void add_prod(T a, T b)
    {
        if (!COMP) {
            hi += a * b;
        } else {
            const T p = a * b;
            const T ep = fma(a, b, -p);
            T sum, es;
            two_sum(hi, p, sum, es);
            hi = sum;
            lo += es + ep;
        }
    }
    // a term far below hi (a product with a low part): into lo directly
    __device__ __forceinline__ void add_lo(T x) { lo += x; }
    __device__ __forceinline__ T value() const { return COMP ? hi + lo : hi; }
};

template <typename T>
struct SolveArgs {
    int n, m, np, mp;
    const int* __restrict__ rowP;
    const int* __restrict__ rowQ;
    const int* __restrict__ qlist;
    const int* __restrict__ ci;
    const int* __restrict__ cj;
    const T* __restrict__ rec;
    const T* __restrict__ qe;
    const T* __restrict__ q;
    const T* __restrict__ ax;
    T* gg0;     // [m][4] (delta, g, gamma_ref, 0): written inside the kernel, plain (coherent) loads only
    T* gg1;
    T* U;       // [n][6] velocity increment M D delta
    T* Uref;    // [n][6] reference velocity M D gamma_ref
    T* gref;    // [m] reference gradient q + D^T Uref (blocks working from global memory)
    T* priv;       // one-barrier solver: 2 mp values for what a share's shared memory does not hold (qe's space)
    int* hrank;    // one-barrier solver: ranks of the blocks' halo rods (2 mp)
    size_t dyn_bytes;   // its dynamic shared memory
    uint4* xch;    // one-barrier solver: tagged velocities [2][n] rods, then tagged block sums [kSumSlots][blocks]
    int workers;   // one-barrier solver: threads that hold slots and rods (a further warp, if any, sums the blocks)
    double* partials;
    unsigned* bar;
    int* flags;
    double* out;   // [0] residual, [1] alpha0
    T inv_perp, inv_par, inv_rot, inv_spin;
    const T* __restrict__ mobr;   // [4][np] per-rod inverse drags (batches), or NULL for the uniform ones
    const T* __restrict__ comp;   // [mp] per constraint: < 0 collision, >= 0 spring compliance 1/(h kappa); NULL: all collisions
    const T* __restrict__ rec_lo; // float32: low parts of rec, qe and q for the reference passes (else NULL)
    const T* __restrict__ qe_lo;
    const T* __restrict__ pe;   // [mp][8] owner-side records (null: read rec)
    const T* __restrict__ q_lo;
    const T* __restrict__ lop;    // [mp][8] float32: rec_lo rows, owner side / other side (null: read rec_lo)
    const T* __restrict__ loq;
    const T* __restrict__ isc;    // [mp] 1/sigma_c of the diagonal scaling (1 when unscaled)
    double hD, tol;
    T pi_tol;      // stopping threshold on max |pi| (float32: see above)
    int max_iter;
    int refresh;   // refresh the reference every this many iterations (0: never)
    int zero_start;   // gamma_0 = 0 (the one-barrier solver's initial reference needs no rod pass)
    int sort_ns;   // global-memory blocks sort their rods (shared memory for the order was given)
    int sort_cap;  // rods the order's scratch holds (a larger share keeps the rank order)
    long long wait_cycles;
    int fault;
    // a step recorded as a graph: the one-barrier kernel was launched with
    // fit_cap bytes of shared memory and reads its shares' need here (null:
    // the need was checked on the host)
    const unsigned long long* need1_dev;
    long long fit_cap;
    const int* __restrict__ bstart;   // [gridDim.x + 1] rod-rank boundaries of the blocks
};

// A block's own rods [r0, r1) and constraints [c0, c1), with their
// shared-memory copies (valid when the block is staged).
template <typename T>
struct Own {
    int r0, r1, c0, c1, q0, q1, cap_c, cap_r, cap_q;
    T* rec;      // [9][cap_c]
    T* gref;     // [cap_c] q + D^T Uref
    T* ds;       // [cap_c] delta (phase B updates it in place, one thread per entry)
    T* grs;      // [cap_c] g (phase B updates it in place, one thread per entry)
    T* gam;      // [cap_c] gamma_ref
    T* ax;       // [3][cap_r]
    T* U;        // [6][cap_r] delta velocity (the reference velocity during a refresh)
    int* cj;     // [cap_c] other end (rank)
    unsigned short* ci;   // [cap_c] owner, local index
    int* rowP;   // [cap_r + 1] owned ranges (global constraint ids)
    int* rowQ;   // [cap_r + 1] other-side ranges (global CSR positions)
    int* qlist;  // [cap_q] other-side constraint ids of the block's rods
    unsigned short* perm;   // [cap_r] the order in which the rod phase's threads take the rods
};

// Shared-memory bytes of a block's share: per owned constraint 13 values
// and 6 bytes of indices, per rod 9 values, two row pointers and a 16-bit
// slot of the rod order, per other-side entry one id (owner indices are
// 16-bit: at most 65535 rods).
__host__ __device__ inline size_t staged_bytes(int esize, size_t cap_c, size_t cap_r, size_t cap_q)
{
    return (13 * cap_c + 9 * cap_r) * (size_t)esize + (cap_c + 2 * cap_r + 2 + cap_q) * sizeof(int) +
           (((cap_c + cap_r) * sizeof(unsigned short) + 3) & ~(size_t)3);
}

template <typename T>
__device__ void carve(Own<T>& o, unsigned char* base)
{
    T* t = reinterpret_cast<T*>(base);
    const size_t C = o.cap_c, R = o.cap_r;
    o.rec = t; t += 9 * C;
    o.gref = t; t += C;
    o.ds = t; t += C;
    o.grs = t; t += C;
    o.gam = t; t += C;
    o.ax = t; t += 3 * R;
    o.U = t; t += 6 * R;
    int* ip = reinterpret_cast<int*>(t);
    o.cj = ip; ip += C;
    o.rowP = ip; ip += R + 1;
    o.rowQ = ip; ip += R + 1;
    o.qlist = ip; ip += o.cap_q;
    o.ci = reinterpret_cast<unsigned short*>(ip);
    o.perm = o.ci + C;
}

// Rod order of the rod phase: ascending (owned, other-side) entry counts,
// so that the 32 rods of a warp run loops of about the same lengths (a warp
// runs each loop as long as its longest rod's).  Rank sort on unique keys
// (count pair, then the block-local index, < 65536) in the scratch key and
// rk ([nr] each); rowP and rowQ point at the block's first rod's row
// pointers.
__device__ void sort_rods(const int* rowP, const int* rowQ, int nr, unsigned* key, int* rk, unsigned short* perm)
{
    for (int li = threadIdx.x; li < nr; li += blockDim.x) {
        const int no = min(rowP[li + 1] - rowP[li], 255), nq = min(rowQ[li + 1] - rowQ[li], 255);
        key[li] = ((unsigned)(no << 8 | nq) << 16) | (unsigned)li;
    }
    __syncthreads();
    for (int li = threadIdx.x; li < nr; li += blockDim.x) {
        const unsigned kk = key[li];
        int r = 0;
        for (int lj = 0; lj < nr; ++lj) r += key[lj] < kk;
        rk[li] = r;
    }
    __syncthreads();
    for (int li = threadIdx.x; li < nr; li += blockDim.x) perm[rk[li]] = (unsigned short)li;
    __syncthreads();
}

template <typename T>
__device__ void stage_in(const SolveArgs<T>& a, Own<T>& o)
{
    const int nr = o.r1 - o.r0, nc = o.c1 - o.c0;
    const size_t mp = a.mp, np = a.np;
    for (int li = threadIdx.x; li <= nr; li += blockDim.x) {
        o.rowP[li] = a.rowP[o.r0 + li];
        o.rowQ[li] = a.rowQ[o.r0 + li];
    }
    for (int li = threadIdx.x; li < nr; li += blockDim.x)
        for (int w = 0; w < 3; ++w) o.ax[w * o.cap_r + li] = a.ax[w * np + o.r0 + li];
#pragma unroll 1
    for (int lc = threadIdx.x; lc < nc; lc += blockDim.x) {
        const int c = o.c0 + lc;
#pragma unroll
        for (int w = 0; w < 9; ++w) o.rec[w * o.cap_c + lc] = a.rec[w * mp + c];
        o.cj[lc] = a.cj[c];
        o.ci[lc] = (unsigned short)(a.ci[c] - o.r0);
        T d, g, gr, gl;
        ld_state(a.gg0, c, d, g, gr, gl);
        o.ds[lc] = d;
        o.gam[lc] = gr;
        o.grs[lc] = T(0);
    }
    for (int k = threadIdx.x; k < o.q1 - o.q0; k += blockDim.x) o.qlist[k] = a.qlist[o.q0 + k];
    // the keys and ranks of the rod order live in the velocity array, which
    // the first rod phase writes before anyone reads it (6 cap_r values hold
    // 2 nr words)
    __syncthreads();
    sort_rods(o.rowP, o.rowQ, nr, reinterpret_cast<unsigned*>(o.U), reinterpret_cast<int*>(o.U) + nr, o.perm);
}

// Rod phase modes: A_STEP forms delta_{k+1} = max(-gamma_ref, delta - alpha g)
// (the owner stores it) and stores dU = M D delta_{k+1}; A_PG sums pi.A.pi
// for the projected gradient pi (returned, nothing stored); A_REF stores the
// reference velocity Uref = M D gamma_ref with compensated sums over the
// split (hi + lo) records, and clears dU.
enum { A_STEP = 0, A_PG = 1, A_REF = 2 };
// Constraint phase modes: B_STEP g_{k+1} = gref + D^T dU and the BB sums;
// B_REF gref = q + D^T Uref (compensated, split records and q), then
// g = gref (delta is 0 there) and pi.pi, max |pi| at gamma_ref.
enum { B_STEP = 0, B_REF = 2 };

// g < 0 ? g : 0, and hi > lo ? hi : lo for values >= 0 (or NaN), on the
// integer pipe: a float64 compare costs the SM's one float64 pipe 19 cycles
// per warp, like any other float64 instruction (measured; 1e5 rods 21.4 ->
// 20.1 ms, 2e4 rods 13.6 -> 12.8, float64).
__device__ __forceinline__ double neg_part(double g)
{
    const int h = __double2hiint(g);   // (-0 stays -0; a NaN gives 0, as the compare does)
    return h < 0 && !((h & 0x7fffffff) > 0x7ff00000 || ((h & 0x7fffffff) == 0x7ff00000 && __double2loint(g) != 0)) ? g : 0.0;
}
__device__ __forceinline__ double max_abs(double lo, double hi)
{
    const long long x = __double_as_longlong(lo), y = __double_as_longlong(hi);
    return y > x && y <= 0x7ff0000000000000ll ? hi : lo;   // (no order with a NaN: lo stays)
}

// bil: a spring (bilateral) constraint, whose force has no sign constraint
// (Eq. linearconstraints b): no projection.
template <int MODE, typename T>
__device__ __forceinline__ T a_value(T d, T g, T gr, T alpha, bool bil)
{
    if (MODE == A_REF) return gr;
    if (MODE == A_STEP) {
        const T v = fma(-alpha, g, d);   // one rounding, the same in both phases that form it
        return (bil || v > -gr) ? v : -gr;
    }
    return (bil || d > -gr) ? g : (g < T(0) ? g : T(0));   // projected gradient at gamma = gr + d
}

template <typename T>
__device__ __forceinline__ T comp_of(const SolveArgs<T>& a, int c)
{
    return a.comp ? __ldg(&a.comp[c]) : T(-1);
}

template <typename T, int MODE, bool ST>
__device__ __forceinline__ T phase_a(const SolveArgs<T>& a, const Own<T>& o, int cur, T alpha)
{
    constexpr bool COMP = MODE == A_REF && sizeof(T) == 4;
    T fmf = T(0);
    const size_t mp = a.mp, np = a.np;
    constexpr int B = Batch<T>::v;
    constexpr int BO = ST ? 1 : B;   // owned entries come from shared memory when staged
    const T* gc = cur ? a.gg1 : a.gg0;
    T* gn = cur ? a.gg0 : a.gg1;
    const T* sdc = o.ds;   // shared copy (staged blocks)
#pragma unroll 1
    for (int t = threadIdx.x; t < o.r1 - o.r0; t += blockDim.x) {
        const int li = o.perm ? (int)o.perm[t] : t, i = o.r0 + li;
        Acc<T, COMP> Fa[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) Fa[w].init(T(0));
        {   // owned constraints: loads of up to BO entries issued together
            const int b = ST ? o.rowP[li] : a.rowP[i], e = ST ? o.rowP[li + 1] : a.rowP[i + 1];
#pragma unroll 1
            for (int c = b; c < e; c += BO) {
                T dv[BO], gv[BO], rv_[BO], gl[BO], rv[BO][6];
#pragma unroll
                for (int u = 0; u < BO; ++u) {
                    if (c + u < e) {
                        if (ST) {
                            const int lc = c + u - o.c0;
                            dv[u] = sdc[lc];
                            gv[u] = o.grs[lc];
                            rv_[u] = o.gam[lc];
                            if (MODE == A_REF && COMP) gl[u] = gc[4 * (size_t)(c + u) + 3];
#pragma unroll
                            for (int w = 0; w < 6; ++w) rv[u][w] = o.rec[w * o.cap_c + lc];
                        } else {
                            ld_state(gc, c + u, dv[u], gv[u], rv_[u], gl[u]);
                            if (sizeof(T) == 4 && a.pe) {   // float64 is bound by its arithmetic instead
                                ld_arm(a.pe, c + u, rv[u]);
                            } else {
#pragma unroll
                                for (int w = 0; w < 6; ++w) rv[u][w] = a.rec[w * mp + c + u];
                            }
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < BO; ++u) {
                    if (c + u < e) {
                        const T cmp = comp_of(a, c + u);
                        const T v = a_value<MODE, T>(dv[u], gv[u], rv_[u], alpha, cmp >= T(0));
                        if (MODE == A_PG && cmp >= T(0)) fmf += cmp * v * v;   // the spring's compliance term
                        // phase B forms delta_{k+1} again from the same values (staged
                        // blocks, float32); float64, bound by its arithmetic, stores it
                        if (MODE == A_STEP && !ST && sizeof(T) == 8) gn[4 * (size_t)(c + u)] = v;
#pragma unroll
                        for (int w = 0; w < 6; ++w) Fa[w].add_prod(v, rv[u][w]);
                        if (MODE == A_REF && COMP) {   // gamma_lo and the records' low parts
#pragma unroll
                            for (int w = 0; w < 6; ++w)
                                Fa[w].add_lo(v * __ldg(&a.rec_lo[w * mp + c + u]) + gl[u] * rv[u][w]);
                        }
                    }
                }
            }
        }
        {   // constraints owned by other rods: ids first, then their state and arms
            // (from shared memory when the owner is one of the block's rods)
            const int b = ST ? o.rowQ[li] : a.rowQ[i], e = ST ? o.rowQ[li + 1] : a.rowQ[i + 1];
#pragma unroll 1
            for (int k = b; k < e; k += B) {
                int cid[B];
#pragma unroll
                for (int u = 0; u < B; ++u)
                    cid[u] = k + u < e ? (ST ? o.qlist[k + u - o.q0] : __ldg(&a.qlist[k + u])) : -1;
                T dv[B], gv[B], rv_[B], gl[B], qv[B][6];
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    if (cid[u] >= 0) {
                        if (ST && cid[u] >= o.c0 && cid[u] < o.c1) {
                            const int lc = cid[u] - o.c0;
                            dv[u] = sdc[lc];
                            gv[u] = o.grs[lc];
                            rv_[u] = o.gam[lc];
                            if (MODE == A_REF && COMP) gl[u] = gc[4 * (size_t)cid[u] + 3];
#pragma unroll
                            for (int w = 0; w < 3; ++w) {
                                qv[u][w] = o.rec[w * o.cap_c + lc];
                                qv[u][3 + w] = o.rec[(6 + w) * o.cap_c + lc];
                            }
                        } else {
                            ld_state(gc, cid[u], dv[u], gv[u], rv_[u], gl[u]);
                            ld_arm(a.qe, k + u, qv[u]);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    if (cid[u] >= 0) {
                        const T v = a_value<MODE, T>(dv[u], gv[u], rv_[u], alpha, comp_of(a, cid[u]) >= T(0));
#pragma unroll
                        for (int w = 0; w < 6; ++w) Fa[w].add_prod(-v, qv[u][w]);
                        if (MODE == A_REF && COMP) {
                            T ql[6];
                            ld_arm(a.qe_lo, k + u, ql);
#pragma unroll
                            for (int w = 0; w < 6; ++w) Fa[w].add_lo(-(v * ql[w] + gl[u] * qv[u][w]));
                        }
                    }
                }
            }
        }
        T F[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) F[w] = Fa[w].value();
        T p0, p1, p2;
        if (ST) {
            p0 = o.ax[li]; p1 = o.ax[o.cap_r + li]; p2 = o.ax[2 * o.cap_r + li];
        } else {
            p0 = a.ax[i]; p1 = a.ax[np + i]; p2 = a.ax[2 * np + i];
        }
        T ip = a.inv_perp, ipa = a.inv_par, ir = a.inv_rot, is = a.inv_spin;
        if (a.mobr) {
            ip = __ldg(&a.mobr[i]); ipa = __ldg(&a.mobr[np + i]);
            ir = __ldg(&a.mobr[2 * np + i]); is = __ldg(&a.mobr[3 * np + i]);
        }
        const T pf = p0 * F[0] + p1 * F[1] + p2 * F[2];
        const T pt = p0 * F[3] + p1 * F[4] + p2 * F[5];
        const T cf = pf * (ipa - ip), ct = pt * (is - ir);
        T Uv[6] = {F[0] * ip + p0 * cf, F[1] * ip + p1 * cf, F[2] * ip + p2 * cf,
                   F[3] * ir + p0 * ct, F[4] * ir + p1 * ct, F[5] * ir + p2 * ct};
        if (MODE == A_PG) {
#pragma unroll
            for (int w = 0; w < 6; ++w) fmf += F[w] * Uv[w];
        } else {
            // staged steps publish dU after the rod loop, coalesced (copy_out_du)
            if (!(ST && MODE == A_STEP)) st_u6(MODE == A_REF ? a.Uref : a.U, i, Uv);
            if (MODE == A_REF) {
                const T z[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
                st_u6(a.U, i, z);   // dU = 0: delta is 0 after a reference pass
            }
            if (ST) {
#pragma unroll
                for (int w = 0; w < 6; ++w) o.U[w * o.cap_r + li] = Uv[w];
            }
        }
    }
    return fmf;
}

// Velocity M F of one rod, three components: a n F + p (p.F)(b - a), the
// translational half (a = 1/zeta_perp, b = 1/zeta_par) or the rotational
// one.  The products' fusing is written out, so that every kernel rounds alike.
template <typename T>
__device__ __forceinline__ void half_mobility(const T p[3], const T F[3], T ia, T ib, T U[3])
{
    const T pf = fma(p[2], F[2], fma(p[0], F[0], p[1] * F[1]));
    const T cf = pf * (ib - ia);
#pragma unroll
    for (int w = 0; w < 3; ++w) U[w] = fma(p[w], cf, F[w] * ia);
}

// Rod phase of a float32 step of the batched solver: one thread per rod over
// its entries, owned then other-side, in one loop; the next entry's state and
// row and the id of the one after are loaded while the current one is summed.
// A cluster's blocks have too few rods to hide the loads of one entry behind
// other warps' (solve, 256 systems 21.5 -> 20.8 ms, 16 small ones 2.52 -> 2.38;
// the single-system solver, whose loads L2 and HBM bound, is 6 to 9 % slower this
// way on the 4e5-rod pack and keeps phase_a's two loops).
__device__ __forceinline__ void rod_step_g(const SolveArgs<float>& a, const Own<float>& o, int cur, float alpha)
{
    const float4* const gc = reinterpret_cast<const float4*>(cur ? a.gg1 : a.gg0);
    const size_t np = a.np;
    const bool has_comp = a.comp != nullptr;
#pragma unroll 1
    for (int i = o.r0 + threadIdx.x; i < o.r1; i += blockDim.x) {
        const int b = a.rowP[i], no = a.rowP[i + 1] - b, k0 = a.rowQ[i] - no, ne = no + a.rowQ[i + 1] - a.rowQ[i];
        float F[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        auto id = [&](int e) { return e < no ? b + e : e < ne ? __ldg(&a.qlist[k0 + e]) : 0; };
        auto row = [&](int e, int c) {
            return reinterpret_cast<const float4*>(e < no ? a.pe : a.qe) + 2 * (size_t)(e < no ? c : k0 + e);
        };
        int c = id(0), c1 = id(1);
        float4 st = make_float4(0.0f, 0.0f, 0.0f, 0.0f), ra = st;
        float2 rb = make_float2(0.0f, 0.0f);
        if (ne > 0) {
            st = gc[c];
            const float4* const p = row(0, c);
            ra = __ldg(p);
            rb = __ldg(reinterpret_cast<const float2*>(p + 1));
        }
#pragma unroll 1
        for (int e = 0; e < ne; ++e) {
            float4 st1 = st, ra1 = ra;
            float2 rb1 = rb;
            if (e + 1 < ne) {
                st1 = gc[c1];
                const float4* const p = row(e + 1, c1);
                ra1 = __ldg(p);
                rb1 = __ldg(reinterpret_cast<const float2*>(p + 1));
            }
            const int c2 = id(e + 2);
            bool bil = false;
            if (has_comp) bil = __ldg(&a.comp[c]) >= 0.0f;
            const float v = a_value<A_STEP, float>(st.x, st.y, st.z, alpha, bil);
            const float w = e < no ? v : -v;
            F[0] = fma(w, ra.x, F[0]);
            F[1] = fma(w, ra.y, F[1]);
            F[2] = fma(w, ra.z, F[2]);
            F[3] = fma(w, ra.w, F[3]);
            F[4] = fma(w, rb.x, F[4]);
            F[5] = fma(w, rb.y, F[5]);
            st = st1;
            ra = ra1;
            rb = rb1;
            c = c1;
            c1 = c2;
        }
        const float p[3] = {a.ax[i], a.ax[np + i], a.ax[2 * np + i]};
        float ip = a.inv_perp, ipa = a.inv_par, ir = a.inv_rot, is = a.inv_spin;
        if (a.mobr) {
            ip = __ldg(&a.mobr[i]); ipa = __ldg(&a.mobr[np + i]);
            ir = __ldg(&a.mobr[2 * np + i]); is = __ldg(&a.mobr[3 * np + i]);
        }
        float U[6];
        half_mobility(p, F, ip, ipa, U);
        half_mobility(p, F + 3, ir, is, U + 3);
        st_u6(a.U, i, U);
    }
}

// A staged step's dU for the other blocks: the block's rods [r0, r1) are
// contiguous in the [n][6] global array, so after the rod loop the block
// copies its shared [6][cap_r] values out with consecutive threads writing
// consecutive pairs.  The rod loop's own stores would be three scattered
// 8-byte stores per rod (its threads take the rods in count order), which
// the grid barrier's release then waits for.
template <typename T>
__device__ __forceinline__ void copy_out_du(const SolveArgs<T>& a, const Own<T>& o)
{
    __syncthreads();
    const int nr = o.r1 - o.r0;
    typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(a.U + 6 * (size_t)o.r0);
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x) {
        const int r = k / 3, w = 2 * (k - 3 * r);
        typename V2<T>::t v;
        v.x = o.U[w * o.cap_r + r];
        v.y = o.U[(w + 1) * o.cap_r + r];
        g[k] = v;
    }
}

// Constraint phase for the block's owned constraints (modes above).  In
// B_STEP the new state (delta_{k+1}, g_{k+1}, gamma_ref) goes to buffer nx,
// and acc0..2 = s.s, s.y, y.y against buffer cur; acc3 = max |pi|.
template <typename T, int MODE, bool ST>
__device__ __forceinline__ void phase_b(const SolveArgs<T>& a, const Own<T>& o, int cur, int nx, T alpha, T acc[4])
{
    constexpr bool COMP = MODE != B_STEP && sizeof(T) == 4;
    const size_t mp = a.mp;
    T* gnew = nx ? a.gg1 : a.gg0;
    const T* gold = cur ? a.gg1 : a.gg0;
    const T* Uu = MODE == B_STEP ? a.U : a.Uref;
    const int nc = o.c1 - o.c0;
#pragma unroll 1
    for (int lc = threadIdx.x; lc < nc; lc += blockDim.x) {
        const int c = o.c0 + lc;
        T Ui[6], Uj[6], r[9], base, dm, gam, dold = T(0), gro = T(0);
        bool xstate = false;
        if (ST) {
            const int il = o.ci[lc], j = o.cj[lc];
            xstate = j >= 0 && (j < o.r0 || j >= o.r1);
#pragma unroll
            for (int w = 0; w < 6; ++w) Ui[w] = o.U[w * o.cap_r + il];
            if (j < 0) {   // a wall: no other side
#pragma unroll
                for (int w = 0; w < 6; ++w) Uj[w] = T(0);
            } else if (j >= o.r0 && j < o.r1) {
#pragma unroll
                for (int w = 0; w < 6; ++w) Uj[w] = o.U[w * o.cap_r + (j - o.r0)];
            } else {
                ld_u6(Uu, j, Uj);
            }
#pragma unroll
            for (int w = 0; w < 9; ++w) r[w] = o.rec[w * o.cap_c + lc];
            base = MODE == B_STEP ? o.gref[lc] : a.q[c];
            gam = o.gam[lc];
            if (MODE == B_STEP) {
                // delta_{k+1} as the rod phase formed it (same inputs, same rounding)
                dold = o.ds[lc];
                gro = o.grs[lc];
                dm = a_value<A_STEP, T>(dold, gro, gam, alpha, comp_of(a, c) >= T(0));
                o.ds[lc] = dm;
            } else {
                dm = o.ds[lc];
            }
        } else {
            ld_u6(Uu, a.ci[c], Ui);
            const int j = a.cj[c];
            if (j < 0) {   // a wall: no other side
#pragma unroll
                for (int w = 0; w < 6; ++w) Uj[w] = T(0);
            } else {
                ld_u6(Uu, j, Uj);
            }
#pragma unroll
            for (int w = 0; w < 9; ++w) r[w] = a.rec[w * mp + c];
            base = MODE == B_STEP ? a.gref[c] : a.q[c];
            T gl;
            if (MODE == B_STEP && sizeof(T) == 4) {
                // delta_{k+1} as the rod phase formed it (same inputs, same rounding)
                ld_state(gold, c, dold, gro, gam, gl);
                dm = a_value<A_STEP, T>(dold, gro, gam, alpha, comp_of(a, c) >= T(0));
            } else {
                T gdummy;
                ld_state(gnew, c, dm, gdummy, gam, gl);
                if (MODE == B_STEP) {
                    T g2, gl2;
                    ld_state(gold, c, dold, gro, g2, gl2);
                }
            }
        }
        Acc<T, COMP> du;
        du.init(base);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            du.add_prod(r[u], Ui[u]);
            du.add_prod(-r[u], Uj[u]);
            du.add_prod(r[3 + u], Ui[3 + u]);
            du.add_prod(-r[6 + u], Uj[3 + u]);
        }
        // springs: + (1/(h kappa)) gamma (Eq. blockdef F); the increment's
        // part in a step, the whole force in a reference pass
        const T cmp = comp_of(a, c);
        const bool bil = cmp >= T(0);
        if (bil) {
            if (MODE == B_STEP) {
                du.add_prod(cmp, dm);
            } else {
                const T glo = gl_of_state(gnew, c);
                du.add_prod(cmp, gam);
                du.add_lo(cmp * glo);
            }
        }
        if (MODE == B_REF && COMP) {
            // low parts of q and of the record
            T rl[9];
#pragma unroll
            for (int w = 0; w < 9; ++w) rl[w] = __ldg(&a.rec_lo[w * mp + c]);
            T t = __ldg(&a.q_lo[c]);
#pragma unroll
            for (int u = 0; u < 3; ++u)
                t += rl[u] * (Ui[u] - Uj[u]) + rl[3 + u] * Ui[3 + u] - rl[6 + u] * Uj[3 + u];
            du.add_lo(t);
        }
        const T gr = du.value();
        if (MODE == B_REF) {
            if (ST) o.gref[lc] = gr;
            else a.gref[c] = gr;
        }
        // g of the new iterate (for B_REF: gamma_ref itself, delta = 0)
        if (ST) {
            o.grs[lc] = gr;
            // the state other blocks read in the next rod phase: in a step,
            // only that of constraints whose other rod is another block's
            if (MODE != B_STEP || xstate) st_dg(gnew, c, dm, gr);
        } else if (MODE == B_STEP && sizeof(T) == 4) {
            st_dg(gnew, c, dm, gr);
        } else {
            gnew[4 * (size_t)c + 1] = gr;
        }
        T pi;
        // the residual is taken on the unscaled projected gradient pi / sigma_c
        if constexpr (sizeof(T) == 8) {
            pi = (bil || dm > -gam) ? gr : neg_part(gr);
            acc[3] = max_abs(acc[3], fabs(pi) * __ldg(&a.isc[c]));
        } else {
            pi = (bil || dm > -gam) ? gr : (gr < T(0) ? gr : T(0));
            const T api = (pi < T(0) ? -pi : pi) * __ldg(&a.isc[c]);
            acc[3] = api > acc[3] ? api : acc[3];
        }
        if (MODE == B_REF) {
            acc[0] += pi * pi;
        } else {
            const T sv = dm - dold, yv = gr - gro;
            acc[0] += sv * sv;
            acc[1] += sv * yv;
            acc[2] += yv * yv;
        }
    }
}

// Refresh, first half: (gamma_ref, gamma_lo) absorbs delta as a
// double-float sum (TwoSum, then renormalised so that |gamma_lo| is at most
// half an ulp of gamma_ref) and delta becomes 0, in shared memory and in
// both global state buffers.  A constraint held at the bound (delta =
// -gamma_ref) gets gamma = 0 exactly.
template <typename T, bool ST>
__device__ __forceinline__ void fold_delta(const SolveArgs<T>& a, const Own<T>& o, int cur)
{
    T* gc = cur ? a.gg1 : a.gg0;
    T* go = cur ? a.gg0 : a.gg1;
    T* sdc = o.ds;
    const int nc = o.c1 - o.c0;
#pragma unroll 1
    for (int lc = threadIdx.x; lc < nc; lc += blockDim.x) {
        const int c = o.c0 + lc;
        T d, g, gr, gl;
        ld_state(gc, c, d, g, gr, gl);
        if (ST) {
            d = sdc[lc]; g = o.grs[lc]; gr = o.gam[lc];
        }
        const bool bil = comp_of(a, c) >= T(0);   // springs: no bound
        T hi = T(0), lo = T(0);
        if (bil || d > -gr) {
            T s, e;
            two_sum(gr, d, s, e);
            const T l = gl + e;
            hi = s + l;
            lo = l - (hi - s);
            if (!bil && (hi < T(0) || (hi == T(0) && lo < T(0)))) { hi = T(0); lo = T(0); }
        }
        if (ST) {
            sdc[lc] = T(0);
            o.gam[lc] = hi;
        }
        st_dg(gc, c, T(0), g);
        st_ref(gc, c, hi, lo);
        st_ref(go, c, hi, lo);
    }
}

// hi > lo ? hi : lo
template <typename T>
__device__ __forceinline__ T max_of(T lo, T hi)
{
    if constexpr (sizeof(T) == 8) return max_abs(lo, hi);   // (magnitudes everywhere: values >= 0)
    else return hi > lo ? hi : lo;
}

// One warp's (sum, sum, sum, max) over its lanes: lane 0, 16, 8 and 24 return
// them.  The four values fold into one register per lane as the tree halves
// (lanes keep one value and pass the other on), so the five levels cost six
// exchanges and adds instead of twenty; every pair of operands is the same as in
// a plain tree per value, and so is every bit.
template <typename T>
__device__ __forceinline__ T warp_sums4(const T v[4])
{
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool h16 = lane & 16, h8 = lane & 8;
    // value 0 (sum) stays in lanes 0-15, value 1 (sum) in lanes 16-31; likewise 2 (sum), 3 (max)
    const T s01 = __shfl_xor_sync(all, h16 ? v[0] : v[1], 16);
    const T s23 = __shfl_xor_sync(all, h16 ? v[2] : v[3], 16);
    const T a = (h16 ? v[1] : v[0]) + s01;
    const T b = h16 ? max_of(s23, v[3]) : v[2] + s23;
    // the maximum ends in lanes 24-31, the sums in lanes 0, 16 and 8
    const bool is_max = h16 && h8;
    T x = h8 ? b : a;
    T y = __shfl_xor_sync(all, h8 ? a : b, 8);
    x = is_max ? max_of(y, x) : x + y;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        y = __shfl_xor_sync(all, x, o);
        const bool up = lane & o;
        x = is_max ? max_of(up ? y : x, up ? x : y) : x + y;
    }
    return x;
}
// The value (0-3) that a lane of warp_sums4 with lane % 8 == 0 returns.
__device__ __forceinline__ int sums4_value(int lane) { return (lane & 8 ? 2 : 0) + (lane & 16 ? 1 : 0); }

// Warp w's share of the block sums into red[w].
template <typename T>
__device__ __forceinline__ void warp_partial(const T v[4], T (*red)[4])
{
    const T x = warp_sums4(v);
    const int lane = threadIdx.x & 31;
    if ((lane & 7) == 0) red[threadIdx.x >> 5][sums4_value(lane)] = x;
}

// Block partial of (sum, sum, sum, max) in the working precision (warp
// shuffles, then warp 0 over the warp results, fixed order); lane 0 stores
// it for the cross-block sum.
template <typename T>
__device__ __forceinline__ void block_partial(T v[4], T (*red)[4], T* dst, int stride)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < 3; ++u) v[u] += __shfl_down_sync(0xffffffffu, v[u], o);
        T mx = __shfl_down_sync(0xffffffffu, v[3], o);
        v[3] = mx > v[3] ? mx : v[3];
    }
    if (lane == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) red[warp][u] = v[u];
    }
    __syncthreads();
    if (warp == 0) {
        T w[4] = {T(0), T(0), T(0), T(0)};
        if (lane < nw) {
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = red[lane][u];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int u = 0; u < 3; ++u) w[u] += __shfl_down_sync(0xffffffffu, w[u], o);
            T mx = __shfl_down_sync(0xffffffffu, w[3], o);
            w[3] = mx > w[3] ? mx : w[3];
        }
        if (lane == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) dst[u * stride] = w[u];
        }
    }
}

// The same in float64 with the folded trees: the plain ones of 24 warps are
// 480 float64 instructions, of 19 cycles each on the SM's one float64 pipe, a
// tenth of an iteration at 2e4 rods (solve_lcp 15.2 -> 14.3 ms).  (In float32
// they cost nothing, and the plain trees are 1 % faster.)
__device__ __forceinline__ void block_partial(double v[4], double (*red)[4], double* dst, int stride)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    warp_partial(v, red);
    __syncthreads();
    if (warp == 0) {
        double w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = lane < nw ? red[lane][u] : 0.0;
        const double x = warp_sums4(w);
        if ((lane & 7) == 0) dst[sums4_value(lane) * stride] = x;
    }
}

// After a barrier: warps 0-3 each reduce one component of the per-block
// partials ([4][nb]: a warp reads one contiguous row) in the working
// precision in a fixed order, the first 12 loads of every lane in flight
// together (one L2 round trip for up to 384 blocks: 304 at 512 threads x 2
// blocks per SM), and the four totals are broadcast through shared memory.
template <typename T>
__device__ __forceinline__ void grid_total(const T* partials, int nb, T* bc, T out[4])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 4) {
        const T* row = partials + (size_t)warp * nb;
        T xs[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int b = lane + 32 * k;
            xs[k] = b < nb ? __ldcg(row + b) : T(0);
        }
        T w = T(0);
        if (warp == 3) {   // max |pi| (every entry >= 0)
#pragma unroll
            for (int k = 0; k < 12; ++k) w = xs[k] > w ? xs[k] : w;
            for (int b = lane + 384; b < nb; b += 32) {
                const T x = __ldcg(row + b);
                w = x > w ? x : w;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const T y = __shfl_down_sync(0xffffffffu, w, o);
                w = y > w ? y : w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 12; ++k) w += xs[k];
            for (int b = lane + 384; b < nb; b += 32) w += __ldcg(row + b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
        }
        if (lane == 0) bc[warp] = w;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = bc[u];
}

// The stopping test's complement: (h/D) max |pi| > tol, decided in float64
// (float64 iterations) or by the equivalent float32 threshold.
__device__ __forceinline__ bool above_tol(const SolveArgs<double>& a, double pimax) { return a.hD * pimax > a.tol; }
__device__ __forceinline__ bool above_tol(const SolveArgs<float>& a, float pimax) { return pimax > a.pi_tol; }

// Step-size bookkeeping, done by thread 0 alone (every other thread only
// reads the broadcast).
// Pass kinds of the loop: a step, a reference pass, the line step of alpha_0.
enum { P_STEP = 0, P_REF = 1, P_PG = 2 };

template <typename T>
struct StepState {
    T alpha0, pimax;   // max |pi| of the last test: the residual is (h/D) pimax
    double pp;         // pi.pi at gamma_0 (for alpha_0)
    T pss, psy, pyy;   // the previous step's s.s, s.y, y.y (the step length lags one iteration)
    int have, hist;    // previous sums held; BB1/BB2 alternation counter
    int iters, cur, done;
    int since;   // iterations since the last reference refresh
    __device__ __forceinline__ double residual(double hD) const { return hD * (double)pimax; }
};

template <typename T>
struct Shared {
    T red[32][4];
    T bc[4];
    T part[4];   // this block's partial (cluster solver: read by the cluster's blocks)
    T alpha;
    int done, ok, kind, cur, sys, pair;
};

// Synchronisation of the blocks that share one problem.
// Grid: all blocks of a cooperative launch, bounded barrier on a global
// counter, partials in global memory.
template <typename T>
struct GridSync {
    unsigned* bar;
    int* flags;
    long long wait_cycles;
    T* partials;   // [4][nb]
    unsigned nb, epoch;
    template <typename SH>
    __device__ __forceinline__ bool barrier(SH& sh)
    {
        return grid_barrier(bar, nb * ++epoch, flags, wait_cycles, &sh.ok);
    }
    template <typename SH>
    __device__ __forceinline__ T* slot(SH&) { return partials + blockIdx.x; }
    __device__ __forceinline__ int stride() const { return (int)nb; }
    template <typename SH>
    __device__ __forceinline__ void total(SH& sh, T tot[4]) { grid_total(partials, nb, sh.bc, tot); }
};

// Cluster: the blocks of one thread-block cluster, hardware cluster barrier,
// partials in each block's shared memory read through distributed shared
// memory (every block sums them in the same order: identical decisions).
struct ClusterSync {
    template <typename SH>
    __device__ __forceinline__ bool barrier(SH&)
    {
        cg::this_cluster().sync();
        return true;
    }
    template <typename SH>
    __device__ __forceinline__ auto slot(SH& sh) { return sh.part; }
    __device__ __forceinline__ int stride() const { return 1; }
    template <typename SH, typename T>
    __device__ __forceinline__ void total(SH& sh, T tot[4])
    {
        cg::cluster_group cl = cg::this_cluster();
        if (threadIdx.x < 4) {
            const int u = threadIdx.x;
            const unsigned cs = cl.num_blocks();
            T w = T(0);
            for (unsigned r = 0; r < cs; ++r) {
                const T x = cl.map_shared_rank(sh.part, r)[u];
                w = u == 3 ? (x > w ? x : w) : w + x;
            }
            sh.bc[u] = w;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) tot[u] = sh.bc[u];
    }
};

// Batches: a cluster alone, or two clusters on one system (a pair).  A pair
// synchronises its blocks like the grid solver, on a bounded barrier over a
// counter of its own, with the block sums in global memory; a cluster alone
// uses the hardware cluster barrier and distributed shared memory.
template <typename T>
struct BatchSync {
    unsigned* bar;       // the pair's arrival counter (null: a cluster alone)
    int* flags;
    long long wait_cycles;
    T* partials;         // the pair's [4][nb] block sums
    unsigned nb, epoch;  // the pair's blocks, barriers passed
    int rank;            // this block's rank in the pair
    template <typename SH>
    __device__ __forceinline__ bool barrier(SH& sh)
    {
        if (bar) return grid_barrier(bar, nb * ++epoch, flags, wait_cycles, &sh.ok);
        cg::this_cluster().sync();
        return true;
    }
    template <typename SH>
    __device__ __forceinline__ T* slot(SH& sh) { return bar ? partials + rank : sh.part; }
    __device__ __forceinline__ int stride() const { return bar ? (int)nb : 1; }
    template <typename SH>
    __device__ __forceinline__ void total(SH& sh, T tot[4])
    {
        if (bar) grid_total(partials, (int)nb, sh.bc, tot);
        else ClusterSync().total(sh, tot);
    }
};

// Smallest rank r in [lo, hi] whose cumulative work W(r) = kOwnWork *
// rowP[r] + kOtherWork * rowQ[r] + kRodWork * r reaches target (an
// other-side entry, gathered from another block, costs about twice an owned
// one in the two-barrier kernels); W is strictly increasing and W(hi) >=
// target.  One warp: 32 probes per round, then a final scan of at most 32
// ranks.  The one-barrier kernel's blocks were timed under other weights
// (owned : other-side : rod = 4:1:4, 4:1:2, 3:1:3, 2:1:2; four seeds at 1e5
// rods): the first two push some shares past the shared-memory budget, the
// others cost 0.5-1.7 % more per iteration than 1:2:2.
constexpr int kOwnWork = 1;
constexpr int kRodWork = 2;
constexpr int kOtherWork = 2;
__device__ __forceinline__ long long rank_work(const int* rowP, const int* rowQ, int r)
{
    return (long long)kOwnWork * rowP[r] + (long long)kOtherWork * rowQ[r] + (long long)kRodWork * r;
}
__device__ __forceinline__ int find_rank(const int* rowP, const int* rowQ, int lo, int hi, long long target)
{
    const int lane = threadIdx.x & 31;
    while (hi - lo >= 32) {
        const long long span = hi - lo;
        const int p = lo + (int)(span * (lane + 1) / 33);
        const long long w = rank_work(rowP, rowQ, p);
        const unsigned ge = __ballot_sync(0xffffffffu, w >= target);
        if (ge == 0) {
            lo = __shfl_sync(0xffffffffu, p, 31) + 1;
        } else {
            const int f = __ffs(ge) - 1;
            const int pf = __shfl_sync(0xffffffffu, p, f);
            const int pb = __shfl_sync(0xffffffffu, p, f > 0 ? f - 1 : 0);
            if (f > 0) lo = pb + 1;
            hi = pf;
        }
    }
    const int p = lo + lane;
    bool ge = false;
    if (p <= hi) ge = rank_work(rowP, rowQ, p) >= target;
    const unsigned m = __ballot_sync(0xffffffffu, ge);
    return m ? lo + __ffs(m) - 1 : hi;
}

// The BBPGD loop over the problem shared by the blocks that SY synchronises.
// On return thread 0 holds the step state; sh.cur is the final buffer.
template <typename T, bool ST, typename SY>
__device__ __forceinline__ void solve_loop(const SolveArgs<T>& a, const Own<T>& o, Shared<T>& sh, SY& sy,
                                           StepState<T>& st)
{
    T* mine = sy.slot(sh);
    T tot[4];
    T v[4];
    st.alpha0 = T(1);
    st.pimax = T(0);
    st.pp = 0.0;
    st.pss = st.psy = st.pyy = T(0);
    st.have = 0;
    st.hist = 0;
    st.cur = 0;
    st.since = 0;
    st.iters = 0;
    if (threadIdx.x == 0) {
        sh.cur = 0;
        sh.kind = P_REF;
    }
    __syncthreads();
    int cur = 0, k = 0;           // k: steps taken
    bool first = true;            // the first pass: the reference is gamma_0 (delta = 0)
    // Every pass ends in the same reduction and decision code, and each
    // pass's code appears once: the persistent kernel's code must stay
    // within the instruction cache (inlined copies made every warp stall on
    // instruction fetch after each barrier).
    for (;;) {
        const int kind = sh.kind;
        const bool initial = first;   // this pass is the reference pass at gamma_0
        const int nx = cur ^ 1;
        v[0] = v[1] = v[2] = v[3] = T(0);
        if (kind == P_STEP) {
            if constexpr (!ST && sizeof(T) == 4 && std::is_same<SY, BatchSync<T>>::value) {
                rod_step_g(a, o, cur, sh.alpha);
            } else {
                phase_a<T, A_STEP, ST>(a, o, cur, sh.alpha);
            }
            if (ST) copy_out_du(a, o);
            if (!sy.barrier(sh)) return;
            phase_b<T, B_STEP, ST>(a, o, cur, nx, sh.alpha, v);
        } else if (kind == P_REF) {
            // the reference takes the iterate; Uref = M D gamma_ref, gref =
            // q + D^T Uref and g are recomputed from the split records with
            // compensated sums, and pi.pi and max |pi| with them
            if (!first) {
                fold_delta<T, ST>(a, o, cur);
                if (!sy.barrier(sh)) return;
            }
            first = false;
            phase_a<T, A_REF, ST>(a, o, cur, T(0));
            if (!sy.barrier(sh)) return;
            phase_b<T, B_REF, ST>(a, o, cur, cur, T(0), v);
        } else {
            // pi.A.pi for alpha_0 = pi.pi / pi.A.pi (exact line step along
            // the projected gradient at gamma_0)
            v[0] = phase_a<T, A_PG, ST>(a, o, cur, T(0));
            // every block has read the partials (grid_total) before any rewrites them
            if (!sy.barrier(sh)) return;
        }
        block_partial(v, sh.red, mine, sy.stride());
        if (!sy.barrier(sh)) return;
        sy.total(sh, tot);
        if (kind == P_STEP) cur = nx;
        if (threadIdx.x == 0) {
            int next = P_STEP;
            if (kind == P_STEP) {
                const T ss = tot[0], sy = tot[1], yy = tot[2];
                st.pimax = tot[3];
                st.cur = cur;
                st.iters = k + 1;
                const bool below = !above_tol(a, tot[3]);
                // the step length of step k + 1 from (s_{k-1}, y_{k-1}): the
                // same one-iteration lag as the one-barrier solver, so every
                // solver kernel runs one method (alpha_0 until a pair is held)
                T an = st.alpha0;
                if (st.have) {
                    an = (st.hist & 1) == 0 ? st.pss / st.psy : st.psy / st.pyy;
                    if (!(st.psy > T(0)) || !isfinite(an) || !(an > T(0))) an = st.alpha0;
                    ++st.hist;
                }
                st.pss = ss;
                st.psy = sy;
                st.pyy = yy;
                st.have = 1;
                sh.alpha = an;
                // float32: a residual below tol is confirmed on a fresh
                // reference before the loop stops (the increments since the
                // last refresh carry float32 rounding); after a refresh that
                // did not confirm it, the next try waits two iterations
                st.done = below && a.refresh == 0;
                ++st.since;
                const bool refresh = a.refresh > 0 && ((below && st.since >= 3) || st.since >= a.refresh);
                if (refresh) {
                    st.since = 0;
                    next = P_REF;
                } else if (k + 1 >= a.max_iter) {
                    st.done = 1;
                }
            } else if (kind == P_REF) {
                st.pimax = tot[3];
                st.done = !above_tol(a, tot[3]) || k >= a.max_iter;
                if (initial) {   // gamma_0: the line step comes next
                    st.pp = (double)tot[0];
                    next = P_PG;
                }
            } else {
                const double pap = (double)tot[0];
                double alpha0 = st.pp / pap;
                if (!(pap > 0.0) || !isfinite(alpha0) || !(alpha0 > 0.0) || !isfinite((T)alpha0)) alpha0 = 1.0;
                st.alpha0 = (T)alpha0;
                sh.alpha = (T)alpha0;
                st.done = 0;
            }
            sh.kind = next;
            sh.done = st.done;
        }
        __syncthreads();
        if (kind == P_STEP) ++k;
        if (sh.done) break;
    }
    if (ST) {
        // the final state of every owned constraint (a step stores only the
        // state that other blocks read)
        T* gf = cur ? a.gg1 : a.gg0;
        for (int lc = threadIdx.x; lc < o.c1 - o.c0; lc += blockDim.x) st_dg(gf, o.c0 + lc, o.ds[lc], o.grs[lc]);
    }
    if (threadIdx.x == 0) sh.cur = st.cur;
    __syncthreads();
}

// MAXT: the most threads of a launch (768: the default shape in float64, with
// 80 registers a thread where 1024 leave 64 and spill: 1e5 rods 21.9 -> 21.4 ms,
// 2e4 rods 14.3 -> 13.6; float32 does not spill and is 3 % slower with more
// registers on the 4e5-rod pack).
template <typename T, bool ST, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_bbpgd(SolveArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ Shared<T> sh;
    if (a.fault == 1 && blockIdx.x == 0) return;   // test hook: this block never arrives
    Own<T> o;
    o.r0 = a.bstart[blockIdx.x];
    o.r1 = a.bstart[blockIdx.x + 1];
    o.c0 = a.rowP[o.r0];
    o.c1 = a.rowP[o.r1];
    o.q0 = a.rowQ[o.r0];
    o.q1 = a.rowQ[o.r1];
    // the carve uses the block's own counts (all of them fit: checked on launch)
    o.cap_c = o.c1 - o.c0;
    o.cap_r = o.r1 - o.r0;
    o.cap_q = o.q1 - o.q0;
    o.perm = nullptr;
    if (ST) {
        carve(o, dyn);
        stage_in(a, o);
    } else if (a.sort_ns) {
        // global-memory blocks: the rod order alone in shared memory
        const int nr = o.r1 - o.r0;
        unsigned* key = reinterpret_cast<unsigned*>(dyn);
        int* rk = reinterpret_cast<int*>(key + nr);
        o.perm = reinterpret_cast<unsigned short*>(rk + nr);
        sort_rods(a.rowP + o.r0, a.rowQ + o.r0, nr, key, rk, o.perm);
    }
    GridSync<T> sy;
    sy.bar = a.bar; sy.flags = a.flags; sy.wait_cycles = a.wait_cycles;
    sy.partials = reinterpret_cast<T*>(a.partials);
    sy.nb = gridDim.x; sy.epoch = 0;
    StepState<T> st;   // meaningful in thread 0 only
    solve_loop<T, ST>(a, o, sh, sy, st);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[1] = (double)st.alpha0;
        a.flags[F_FINAL] = st.cur;
        a.flags[F_ITERS] = st.iters;
        a.out[0] = st.residual(a.hD);
    }
}

// ---------------------------------------------------------------------
// No grid barrier in an iteration (staged blocks).
//
// The loop above exchanges two things between blocks in every iteration:
// the velocities dU, which the constraint phase gathers, and the state of
// constraints whose ends lie in different blocks, which the rod phase
// gathers; each needs its own grid barrier, and the step-length sums ride
// on the second.  Here a block also keeps a copy ("ghost") of every
// constraint that another block owns but whose other end is one of its
// rods, and updates it with the owner's arithmetic on the same inputs
// (the same delta, g and alpha, the same two velocities, the same order of
// operations), so that owner and ghost stay equal bit for bit and the rod
// phase reads nothing but shared memory.  Only dU and the block sums cross
// blocks, and both travel as tagged words (below), so that no iteration
// waits on a grid barrier:
//   constraint phase k (every owned and ghost constraint):
//       g_k = gref + D^T dU_k, for owned constraints the sums of s.s, s.y,
//       y.y (s = delta_k - delta_{k-1}, y = g_k - g_{k-1}) and max |pi_k|,
//       and delta_{k+1} = max(-gamma_ref, delta_k - alpha_k g_k);
//   rod phase k: dU_{k+1} = M D delta_{k+1}, published rod by rod;
//   step decision, by a warp of its own while the others run the rod phase,
//       from the sums of constraint phase k: alpha_{k+1} =
//       BB(s_{k-1}, y_{k-1}), i.e. the Barzilai-Borwein step of the
//       published method taken one iteration late (a gradient method with
//       retards: Friedlander, Martinez, Molina & Raydan, SIAM J. Numer.
//       Anal. 36, 1999), which leaves the sums the rod phase to arrive in.
// A residual below tol, 64 float32 iterations, or max_iter start a
// reference refresh of the iterate the slots hold (the same compensated
// passes as above, with one grid barrier); the loop stops only on the
// residual of a fresh reference, so the returned gamma (delta = 0 there)
// carries the residual it reports, in float64 and float32 alike.
//
// Tagged words: 12 bytes of values and a 32-bit exchange number in one
// 16-byte word, stored and loaded whole (ld/st .b128, relaxed).  A reader
// polls the word it needs until its number is the iteration's, so a
// velocity costs one store and one load across L2, where a grid barrier
// costs the fence over the block's stores, the arrival, the poll and then
// the load.  A word is rewritten two exchanges (velocities) or kSumSlots
// exchanges (sums) later: a block writes dU_{k+2} after decision k+1, which
// took every block's sums of constraint phase k, and a block publishes those
// once all its threads have read dU_k; likewise it publishes sums k + 2
// after decision k + 2, which took every block's sums k + 1, and a block
// publishes those after decision k + 1, when it has read all the sums k.
//
// What bounds it: two messages across L2 an iteration (velocities, sums; one
// way 700-1080 cycles, all blocks' words at every block about 2500) and the
// latency of the two phases; the data sit in shared memory.  Solve times
// before (one grid barrier an iteration) and after, the same bits: 1e3 rods
// float64 5.09 -> 2.01 ms (219 iterations), 1e3 rods with walls 0.71 -> 0.43
// ms a step, 5e3 rods 0.86 -> 0.66, 2e4 rods 1.98 -> 1.45, 5e4 rods 1.43 ->
// 1.25, 1e5 rods 3.90 -> 3.60 (366 iterations), 1e4 rods float64 2.17 -> 1.56.
// Where the rods come in no spatial order (a large solve_lcp) nearly every
// slot's other end is in the halo and the polls cost more than they save, and
// where a launch leaves no L1 for what this kernel spills: those keep the
// barrier (k_bbpgd1_meet, variant1).

// A block's share: rods [r0, r1), owned constraints [c0, c1) in slots
// [0, nc), ghosts in slots [nc, nt).
//
// A slot is three rows of four values, so that one rod's entry is two
// 16-byte loads of shared memory (float32) instead of eight 4-byte gathers:
//   row 0  e_x e_y e_z, the increment delta
//   row 1  y_P x e,     gamma_ref
//   row 2  y_Q x e,     gref = q + D^T Uref (gamma_lo during a refresh)
// Slot nt is all zero.  The constraint phase leaves delta_{k+1}, the rod
// phase's input, in row 0.  A rod's entries, owned then other-side, are
// 16-bit slot numbers (kOther: the rod is the slot's Q side), padded to a
// multiple of four with the zero slot, so that four come in one load and the
// loop has no tail.
//
// Velocities are rows too: the block's rods, one zero row (the other end of a
// wall contact) and the halo, every rod of another block that a slot touches,
// fetched once per iteration however many slots read it.  A slot knows the rows
// of its P and Q ends.
//
// The share's description lives in shared memory, its arrays as offsets into
// the block's dynamic shared memory: held in registers it pushed the kernel
// past the 72 a thread has, and what spilled went to L2, since shared memory
// leaves little L1.
template <typename X>
__device__ __forceinline__ X* smem_at(int off)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    return reinterpret_cast<X*>(dyn + off);
}
template <typename T>
struct Own1 {
    int r0, r1, c0, c1, q0, q1, nc, ng, nt, cap_r;
    int ne;      // entries, padding included
    int nh;      // halo rods
    int halo;    // their rows fit (else every slot polls for itself)
    T* ds;       // [nc] delta before the last step (owned slots: the step's s)
    T* gs;       // [nc] g of the last step (owned slots: the step's y)
    int* gid;    // [ng] constraint id of ghost slot nc + g (global memory)
    int* hrank;  // [nh] rank of each halo rod (global memory)
    int off_ax, off_ij, off_ent, off_rowE, off_perm, off_U;
    using u16 = unsigned short;
    __device__ __forceinline__ T* row() const { return smem_at<T>(0); }             // [3][nt + 1][4]
    __device__ __forceinline__ T* ax() const { return smem_at<T>(off_ax); }         // [3][cap_r]
    __device__ __forceinline__ T* U() const { return smem_at<T>(off_U); }           // [cap_r + 1 + nh][6] this iteration's dU (Uref in a refresh)
    __device__ __forceinline__ unsigned* ij() const { return smem_at<unsigned>(off_ij); }   // [nt] velocity rows of P (low half) and Q
    __device__ __forceinline__ u16* ent() const { return smem_at<u16>(off_ent); }   // [ne]
    __device__ __forceinline__ u16* rowE() const { return smem_at<u16>(off_rowE); } // [cap_r + 1] first entry of each rod, in fours
    __device__ __forceinline__ u16* perm() const { return smem_at<u16>(off_perm); } // [cap_r] rod order of the rod phase
};
constexpr unsigned kOther = 0x8000u;
constexpr int kMaxSlots = 0x7ffe;

__host__ __device__ inline size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

// Whether a share (nt slots of which ng ghosts, nr rods, nq other-side
// entries, nb blocks) is the one-barrier kernel's: 13 values a slot, 9 a rod
// and the indices within the shared-memory budget.  The bound decides which
// kernel solves a system, and with it every bit of the result, so it stays
// where it was drawn; carve1 needs about as much (and leaves ds and gs to
// global memory where a share would not fit).
__host__ __device__ inline size_t staged1_bytes(int esize, size_t nt, size_t ng, size_t nr, size_t nq, size_t nb)
{
    const size_t nbp = (nb + 3) & ~(size_t)3;
    return align16(4 * nbp * esize) + align16((13 * nt + 9 * nr) * esize) +
           align16((nt + ng + 2 * nr + 2) * sizeof(int)) + align16((nt + nq + nr) * sizeof(unsigned short));
}

// Carves the share out of the block's dynamic shared memory.  12 (nt + 1) +
// 9 nr + 6 values, nt words and at most nt + nq + 5 nr + 1 16-bit words are
// no more than staged1_bytes, so they always fit; the halo and then ds and gs
// take what is left of cap bytes (carve_rest, once the halo is counted).
template <typename T>
__device__ void carve1(Own1<T>& o)
{
    const int nt = o.nt, R = o.cap_r;
    int at = 12 * (nt + 1) * (int)sizeof(T);
    o.off_ij = at; at += 4 * nt;
    o.off_ax = (int)(((size_t)at + sizeof(T) - 1) & ~(sizeof(T) - 1)); at = o.off_ax + 3 * R * (int)sizeof(T);
    o.off_ent = (at + 7) & ~7; at = o.off_ent + 2 * o.ne;   // (fours of entries on 8-byte boundaries)
    o.off_rowE = at; at += 2 * (R + 1);
    o.off_perm = at; at += 2 * R;
    o.off_U = (int)align16((size_t)at);   // (vector loads)
}

template <typename T>
__device__ void carve_rest(Own1<T>& o, size_t cap, T* priv, size_t mp)
{
    size_t used = o.off_U + 6 * (size_t)(o.cap_r + 1) * sizeof(T);
    const size_t h = 6 * (size_t)o.nh * sizeof(T), d = 2 * (size_t)o.nc * sizeof(T);
    o.halo = used + h <= cap;
    if (o.halo) used += h;
    if (used + d <= cap) {
        o.ds = smem_at<T>((int)used);
        o.gs = o.ds + o.nc;
    } else {
        o.ds = priv + o.c0;
        o.gs = priv + mp + o.c0;
    }
}

// ------------------------------------------------- tagged 16-byte words
__device__ __forceinline__ void st_word(uint4* p, unsigned x, unsigned y, unsigned z, unsigned tag)
{
    asm volatile("{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\t"
                 "mov.b128 v, {lo, hi};\n\tst.relaxed.gpu.global.b128 [%0], v;\n\t}"
                 ::"l"(p), "r"(x), "r"(y), "r"(z), "r"(tag) : "memory");
}
__device__ __forceinline__ uint4 ld_word(const uint4* p)
{
    uint4 r;
    asm volatile("{\n\t.reg .b64 lo, hi;\n\t.reg .b128 v;\n\tld.relaxed.gpu.global.b128 v, [%4];\n\t"
                 "mov.b128 {lo, hi}, v;\n\tmov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
    return r;
}

// K values of T in ceil(K sizeof(T) / 12) tagged words; get returns whether
// all of them carry the tag.
template <typename T, int K> struct Tagged;
template <int K>
struct Tagged<float, K> {
    static constexpr int kWords = (K + 2) / 3;
    static __device__ __forceinline__ void put(uint4* p, const float* v, unsigned tag)
    {
#pragma unroll
        for (int w = 0; w < kWords; ++w)
            st_word(p + w, __float_as_uint(v[3 * w]), 3 * w + 1 < K ? __float_as_uint(v[3 * w + 1]) : 0u,
                    3 * w + 2 < K ? __float_as_uint(v[3 * w + 2]) : 0u, tag);
    }
    static __device__ __forceinline__ bool get(const uint4* p, unsigned tag, float* v)
    {
        uint4 r[kWords];
        bool ok = true;
#pragma unroll
        for (int w = 0; w < kWords; ++w) r[w] = ld_word(p + w);
#pragma unroll
        for (int w = 0; w < kWords; ++w) {
            ok = ok && r[w].w == tag;
            v[3 * w] = __uint_as_float(r[w].x);
            if (3 * w + 1 < K) v[3 * w + 1] = __uint_as_float(r[w].y);
            if (3 * w + 2 < K) v[3 * w + 2] = __uint_as_float(r[w].z);
        }
        return ok;
    }
};
template <int K>
struct Tagged<double, K> {   // two words hold three values
    static constexpr int kWords = (2 * K + 2) / 3;
    static __device__ __forceinline__ void put(uint4* p, const double* v, unsigned tag)
    {
        unsigned h[3 * kWords] = {};
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(v[k]);
            h[2 * k] = (unsigned)b;
            h[2 * k + 1] = (unsigned)(b >> 32);
        }
#pragma unroll
        for (int w = 0; w < kWords; ++w) st_word(p + w, h[3 * w], h[3 * w + 1], h[3 * w + 2], tag);
    }
    static __device__ __forceinline__ bool get(const uint4* p, unsigned tag, double* v)
    {
        unsigned h[3 * kWords];
        uint4 r[kWords];
        bool ok = true;
#pragma unroll
        for (int w = 0; w < kWords; ++w) r[w] = ld_word(p + w);
#pragma unroll
        for (int w = 0; w < kWords; ++w) {
            ok = ok && r[w].w == tag;
            h[3 * w] = r[w].x; h[3 * w + 1] = r[w].y; h[3 * w + 2] = r[w].z;
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
            v[k] = __longlong_as_double((long long)((unsigned long long)h[2 * k] | (unsigned long long)h[2 * k + 1] << 32));
        return ok;
    }
};
template <typename T> using Xch = Tagged<T, 6>;      // a rod's velocity
template <typename T> using XchSum = Tagged<T, 4>;   // a block's sums
static_assert(Xch<double>::kWords <= kXchRodWords && XchSum<double>::kWords <= kSumWords, "xch_bytes");
// K values at p, polled until all their words carry the tag.  Bounded like
// grid_barrier: after wait_cycles, or when any block has recorded an error,
// it records ALENS_ERR_TIMEOUT, sets *bad and returns what it read last.
template <typename T, int K>
__device__ __forceinline__ void get_tagged(int* flags, long long wait_cycles, const uint4* p, unsigned tag, int* bad, T* v)
{
    if (Tagged<T, K>::get(p, tag, v)) return;
    const long long t0 = clock64();
    for (unsigned polls = 1; !Tagged<T, K>::get(p, tag, v); ++polls) {
        if ((polls & 15u) == 0) {
            const bool late = clock64() - t0 > wait_cycles || polls > (1u << 28);
            if (late) atomicCAS(&flags[F_SOLVE_ERR], 0, ALENS_ERR_TIMEOUT);
            if (late || ld_volatile_i32(&flags[F_SOLVE_ERR]) != 0) {
                *(volatile int*)bad = 1;
                return;
            }
        }
    }
}

// The slots' and rods' first item of this thread (none for the warp beyond the workers).
template <typename T>
__device__ __forceinline__ int first_item(const SolveArgs<T>& a)
{
    return (int)threadIdx.x < a.workers ? (int)threadIdx.x : 0x40000000;
}

template <typename T>
struct Shared1 {
    Own1<T> o;
    T red[32][4];           // (sort_rods_total's counters before the first iteration)
    T alpha;
    T alpha0, pimax;        // step state, kept by the duty warp's lane 0
    int k, since, hist;
    int kind, ng, nh, ne;
    int nref;               // refreshes taken: the reference lives in state buffer nref & 1
    unsigned epoch;         // grid barriers passed (thread 0's)
    // a wait ran out (or another block's did): the block leaves.  One word for the waits
    // of the constraint phase and one for those after it, each read by every
    // thread between block barriers that no write to it crosses.
    int bad[2];
};

template <typename T> struct Row { T x, y, z, w; };
__device__ __forceinline__ Row<float> ld_row(const float* p)
{
    const float4 v = *reinterpret_cast<const float4*>(p);
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Row<double> ld_row(const double* p)
{
    const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
    return {a.x, a.y, b.x, b.y};
}
template <typename T>
__device__ __forceinline__ T* slot_row(const Own1<T>& o, int plane, int t)
{
    return o.row() + 4 * (plane * (o.nt + 1) + t);
}
template <typename T> __device__ __forceinline__ T& slot_delta(const Own1<T>& o, int t) { return slot_row(o, 0, t)[3]; }
template <typename T> __device__ __forceinline__ T& slot_gam(const Own1<T>& o, int t) { return slot_row(o, 1, t)[3]; }
template <typename T> __device__ __forceinline__ T& slot_gref(const Own1<T>& o, int t) { return slot_row(o, 2, t)[3]; }

template <typename T>
__device__ __forceinline__ int slot_gid(const Own1<T>& o, int t)
{
    return t < o.nc ? o.c0 + t : o.gid[t - o.nc];
}

// Stage one slot (owned or ghost) of constraint c from the global arrays.
template <typename T>
__device__ __forceinline__ void stage_slot(const SolveArgs<T>& a, const Own1<T>& o, int t)
{
    const size_t mp = a.mp;
    const int c = slot_gid(o, t);
#pragma unroll
    for (int w = 0; w < 9; ++w) slot_row(o, w / 3, t)[w % 3] = a.rec[w * mp + c];
    T d, g, gr, gl;
    ld_state(a.gg0, c, d, g, gr, gl);
    slot_delta(o, t) = d;
    slot_gam(o, t) = gr;
    slot_gref(o, t) = gl;   // gamma_lo until the first reference pass replaces it
}

// Hash set of the halo's ranks while the share is staged, in the rows' space
// (linear probing, at most half full: size is a power of two >= 2 nt).
struct RankSet {
    int* key;
    int* val;
    int size, shift;
    __device__ __forceinline__ int first(int r) const { return (int)((unsigned)r * 2654435761u >> shift); }
    __device__ __forceinline__ void insert(int r)
    {
        for (int h = first(r);; h = (h + 1) & (size - 1)) {
            const int was = atomicCAS(&key[h], -1, r);
            if (was == -1 || was == r) return;
        }
    }
    __device__ __forceinline__ int find(int r) const
    {
        int h = first(r);
        while (key[h] != r) h = (h + 1) & (size - 1);
        return val[h];
    }
};

template <typename T>
__device__ __noinline__ void stage_in1(const SolveArgs<T>& a, Shared1<T>& sh)
{
    Own1<T>& o = sh.o;
    const int nr = o.r1 - o.r0, nq = o.q1 - o.q0;
    // ghosts: other-side entries of the block's rods that another block owns
    if (threadIdx.x == 0) sh.ng = sh.ne = sh.nh = 0;
    __syncthreads();
    int cnt = 0, fours = 0;
    for (int k = threadIdx.x; k < nq; k += blockDim.x) {
        const int c = a.qlist[o.q0 + k];
        cnt += c < o.c0 || c >= o.c1;
    }
    for (int i = o.r0 + threadIdx.x; i < o.r1; i += blockDim.x)
        fours += (a.rowP[i + 1] - a.rowP[i] + a.rowQ[i + 1] - a.rowQ[i] + 3) >> 2;
    if (cnt) atomicAdd(&sh.ng, cnt);
    if (fours) atomicAdd(&sh.ne, 4 * fours);
    __syncthreads();
    if (threadIdx.x == 0) {
        o.ng = sh.ng;
        o.nt = o.nc + o.ng;
        o.ne = sh.ne;
        carve1(o);
        o.gid = reinterpret_cast<int*>(a.gref) + o.q0;   // gref itself lives in the slots
        o.hrank = a.hrank + o.c0 + o.q0;
        sh.ng = 0;
    }
    __syncthreads();
    RankSet set;
    set.size = 2;
    set.shift = 31;
    while (set.size < 2 * o.nt) { set.size *= 2; --set.shift; }
    set.key = reinterpret_cast<int*>(o.row());
    set.val = set.key + set.size;   // 2 size <= 8 nt words (or 4) of the rows' 12 (nt + 1)
    for (int h = threadIdx.x; h < set.size; h += blockDim.x) set.key[h] = -1;
    // rod order by (owned, other-side) counts for the initial pass, whose
    // per-thread sums depend on it; the keys and ranks live in the velocities'
    // space, which the first pass fills
    {
        unsigned* key = reinterpret_cast<unsigned*>(o.U());
        sort_rods(a.rowP + o.r0, a.rowQ + o.r0, nr, key, reinterpret_cast<int*>(key) + nr, o.perm());
    }
    if (threadIdx.x < 32) {   // first entry of every rod
        int base = 0;
        for (int l0 = 0; l0 <= nr; l0 += 32) {
            const int li = l0 + (int)threadIdx.x, i = o.r0 + li;
            const int f = li < nr ? (a.rowP[i + 1] - a.rowP[i] + a.rowQ[i + 1] - a.rowQ[i] + 3) >> 2 : 0;
            int x = f;
#pragma unroll
            for (int s = 1; s < 32; s *= 2) {
                const int y = __shfl_up_sync(0xffffffffu, x, s);
                if ((int)threadIdx.x >= s) x += y;
            }
            if (li <= nr) o.rowE()[li] = (unsigned short)(base + x - f);
            base += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    for (int li = threadIdx.x; li < nr; li += blockDim.x)
        for (int w = 0; w < 3; ++w) o.ax()[w * o.cap_r + li] = a.ax[w * (size_t)a.np + o.r0 + li];
    for (int e = threadIdx.x; e < o.ne; e += blockDim.x) o.ent()[e] = (unsigned short)o.nt;
    // the halo: other ends of owned constraints, owners of ghosts
    for (int t = threadIdx.x; t < o.nc; t += blockDim.x) {
        const int j = a.cj[o.c0 + t];
        if (j >= 0 && (j < o.r0 || j >= o.r1)) set.insert(j);
    }
    for (int k = threadIdx.x; k < nq; k += blockDim.x) {
        const int c = a.qlist[o.q0 + k];
        if (c < o.c0 || c >= o.c1) set.insert(a.ci[c]);
    }
    __syncthreads();
    for (int h = threadIdx.x; h < set.size; h += blockDim.x) {
        if (set.key[h] >= 0) {
            const int x = atomicAdd(&sh.nh, 1);   // (no result depends on the halo's order)
            set.val[h] = x;
            o.hrank[x] = set.key[h];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        o.nh = sh.nh;
        carve_rest(o, a.dyn_bytes, a.priv, (size_t)a.mp);
    }
    const int zero = nr, halo = nr + 1;   // velocity rows: own rods, zero, halo
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nc; t += blockDim.x) {
        const int c = o.c0 + t, i = a.ci[c], j = a.cj[c], li = i - o.r0;
        const int lj = j < 0 ? zero : j >= o.r0 && j < o.r1 ? j - o.r0 : halo + set.find(j);
        o.ij()[t] = (unsigned)li | (unsigned)lj << 16;
        o.ent()[4 * o.rowE()[li] + c - a.rowP[i]] = (unsigned short)t;
    }
    // other-side entries in CSR order
#pragma unroll 1
    for (int k = o.q0 + threadIdx.x; k < o.q1; k += blockDim.x) {
        const int c = a.qlist[k], j = a.cj[c], li = j - o.r0;   // the block's rod is c's Q side
        int t = c - o.c0;
        if (c < o.c0 || c >= o.c1) {
            // the slot order of ghosts does not enter any result
            const int g = atomicAdd(&sh.ng, 1);
            t = o.nc + g;
            o.gid[g] = c;
            o.ij()[t] = (unsigned)(halo + set.find(a.ci[c])) | (unsigned)li << 16;
        }
        o.ent()[4 * o.rowE()[li] + a.rowP[j + 1] - a.rowP[j] + k - a.rowQ[j]] = (unsigned short)(t | kOther);
    }
    __syncthreads();   // the rows take the place of the set
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) stage_slot(a, o, t);
    if (threadIdx.x < 12) slot_row(o, threadIdx.x / 4, o.nt)[threadIdx.x % 4] = T(0);
    if (threadIdx.x < 6) o.U()[6 * zero + threadIdx.x] = T(0);
    __syncthreads();
}

// Orders the block's rods by the length of their entry loops, so that the
// rods of a warp run about equally long: a counting sort (no result depends
// on the order within one length) over kLens counters.
constexpr int kLens = 64;
template <typename T>
__device__ __noinline__ void sort_rods_total(const Own1<T>& o, int* count)
{
    const int nr = o.r1 - o.r0, lane = threadIdx.x & 31;
    if (threadIdx.x < kLens) count[threadIdx.x] = 0;
    __syncthreads();
    for (int li = threadIdx.x; li < nr; li += blockDim.x)
        atomicAdd(&count[min(o.rowE()[li + 1] - o.rowE()[li], kLens - 1)], 1);
    __syncthreads();
    if (threadIdx.x < 32) {   // starts of the lengths
        const int c0 = count[2 * lane], c1 = count[2 * lane + 1];
        int x = c0 + c1;
#pragma unroll
        for (int s = 1; s < 32; s *= 2) {
            const int y = __shfl_up_sync(0xffffffffu, x, s);
            if (lane >= s) x += y;
        }
        count[2 * lane] = x - c0 - c1;
        count[2 * lane + 1] = x - c1;
    }
    __syncthreads();
    for (int li = threadIdx.x; li < nr; li += blockDim.x)
        o.perm()[atomicAdd(&count[min(o.rowE()[li + 1] - o.rowE()[li], kLens - 1)], 1)] = (unsigned short)li;
    __syncthreads();
}

// The six low parts of one side of constraint c: e's, then the arm's (rec_lo
// rows 0-2 and 3-5 for the owner, 0-2 and 6-8 for the other side, arm0 = 3
// or 6), from the side's 32-byte row when there is one.
template <typename T>
__device__ __forceinline__ void lo_side(const T* rows, const T* rec_lo, size_t mp, int c, int arm0, T out[6])
{
    if (sizeof(T) == 4 && rows) {
        const float4* r = reinterpret_cast<const float4*>(rows + 8 * (size_t)c);
        const float4 x = __ldg(r), y = __ldg(r + 1);
        out[0] = (T)x.x; out[1] = (T)x.y; out[2] = (T)x.z;
        out[3] = (T)x.w; out[4] = (T)y.x; out[5] = (T)y.y;
        return;
    }
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        out[w] = __ldg(&rec_lo[w * mp + c]);
        out[3 + w] = __ldg(&rec_lo[(arm0 + w) * mp + c]);
    }
}

// Rod pass of the reference (one thread per rod): A_REF leaves Uref = M D
// gamma_ref (compensated in float32) in shared memory and in the global
// Uref; A_PG returns this thread's share of pi.A.pi.
template <typename T, int MODE>
__device__ __noinline__ T rod_pass1(const SolveArgs<T>& a, const Own1<T>& o)
{
    constexpr bool COMP = MODE == A_REF && sizeof(T) == 4;
    const bool has_comp = a.comp != nullptr;
    const size_t mp = a.mp, np = a.np;
    T fmf = T(0);
#pragma unroll 1
    for (int tt = first_item(a); tt < o.r1 - o.r0; tt += a.workers) {
        const int li = (int)o.perm()[tt], i = o.r0 + li;
        Acc<T, COMP> Fa[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) Fa[w].init(T(0));
        const int e1 = 4 * o.rowE()[li + 1];
#pragma unroll 1
        for (int e = 4 * o.rowE()[li]; e < e1; ++e) {   // owned constraints, then those other rods own
            const unsigned x = o.ent()[e];
            const int t = (int)(x & ~kOther);
            if (t == o.nt) break;   // padding
            const bool own = !(x & kOther);
            const Row<T> re = ld_row(slot_row(o, 0, t)), rp = ld_row(slot_row(o, 1, t)), rq = ld_row(slot_row(o, 2, t));
            const T r[6] = {re.x, re.y, re.z, own ? rp.x : rq.x, own ? rp.y : rq.y, own ? rp.z : rq.z};
            const T g = rq.w;   // gref; gamma_lo during a refresh
            const int c = slot_gid(o, t);
            const T cmp = has_comp ? __ldg(&a.comp[c]) : T(-1);
            const bool bil = cmp >= T(0);
            const T v = a_value<MODE, T>(re.w, g, rp.w, T(0), bil);
            if (MODE == A_PG && own && bil) fmf += cmp * v * v;   // the spring's compliance term
            const T sv = own ? v : -v;
#pragma unroll
            for (int w = 0; w < 6; ++w) Fa[w].add_prod(sv, r[w]);
            if (COMP) {   // gamma_lo and the records' low parts
                T rl[6];
                lo_side(own ? a.lop : a.loq, a.rec_lo, mp, c, own ? 3 : 6, rl);
#pragma unroll
                for (int w = 0; w < 6; ++w) {
                    const T lo = fma(v, rl[w], g * r[w]);
                    Fa[w].add_lo(own ? lo : -lo);
                }
            }
        }
        T F[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) F[w] = Fa[w].value();
        const T p[3] = {o.ax()[li], o.ax()[o.cap_r + li], o.ax()[2 * o.cap_r + li]};
        T ip = a.inv_perp, ipa = a.inv_par, ir = a.inv_rot, is = a.inv_spin;
        if (a.mobr) {
            ip = __ldg(&a.mobr[i]); ipa = __ldg(&a.mobr[np + i]);
            ir = __ldg(&a.mobr[2 * np + i]); is = __ldg(&a.mobr[3 * np + i]);
        }
        T Uv[6];
        half_mobility(p, F, ip, ipa, Uv);
        half_mobility(p, F + 3, ir, is, Uv + 3);
        if (MODE == A_PG) {
#pragma unroll
            for (int w = 0; w < 6; ++w) fmf += F[w] * Uv[w];
        } else {
#pragma unroll
            for (int w = 0; w < 6; ++w) o.U()[6 * li + w] = Uv[w];
            st_u6(a.Uref, i, Uv);
        }
    }
    return fmf;
}

// The sign of v flipped for an other-side entry.
__device__ __forceinline__ float signed_by(float v, unsigned x)
{
    return __uint_as_float(__float_as_uint(v) ^ (x & kOther) << 16);
}
__device__ __forceinline__ double signed_by(double v, unsigned x)
{
    return __hiloint2double(__double2hiint(v) ^ (int)((x & kOther) << 16), __double2loint(v));
}

// Rod phase of a step: dU = M D delta_{k+1}, two lanes per rod (force and
// torque halves, which only meet in the slots), every entry from shared
// memory: the slot's number, its delta, and one row.  The loads of four
// entries are in flight together (the sums stay in entry order); dU goes to
// shared memory and, tagged, to the other blocks.
template <typename T>
__device__ __forceinline__ void rod_step2(const SolveArgs<T>& a, const Own1<T>& o, uint4* xb, unsigned tag)
{
    const int n2 = 2 * (o.r1 - o.r0), r0 = o.r0, R = o.cap_r, plane = 4 * (o.nt + 1);
    const T* const row = o.row();
    const T* const ax = o.ax();
    T* const Us = o.U();
    const unsigned short *const perm = o.perm(), *const rowE = o.rowE();
    const ushort4* const ent = reinterpret_cast<const ushort4*>(o.ent());
#pragma unroll 1
    for (int tt = first_item(a); tt < n2; tt += a.workers) {
        const int li = (int)perm[tt >> 1], half = tt & 1;
        const int e1 = rowE[li + 1];
        const int own_plane = half ? plane : 0, oth_plane = half ? 2 * plane : 0;
        T F[3] = {T(0), T(0), T(0)};
#pragma unroll 1
        for (int e = rowE[li]; e < e1; ++e) {
            const ushort4 q = ent[e];
            const unsigned x[4] = {q.x, q.y, q.z, q.w};
            T v[4];
            Row<T> r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const T* p = row + 4 * (int)(x[u] & ~kOther);
                v[u] = signed_by(p[3], x[u]);
                r[u] = ld_row(p + (x[u] & kOther ? oth_plane : own_plane));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                F[0] = fma(v[u], r[u].x, F[0]);
                F[1] = fma(v[u], r[u].y, F[1]);
                F[2] = fma(v[u], r[u].z, F[2]);
            }
        }
        const int i = r0 + li;
        const T p[3] = {ax[li], ax[R + li], ax[2 * R + li]};
        T ia = half ? a.inv_rot : a.inv_perp, ib = half ? a.inv_spin : a.inv_par;
        if (a.mobr) {
            ia = __ldg(&a.mobr[(half ? 2 * (size_t)a.np : 0) + i]);
            ib = __ldg(&a.mobr[(half ? 3 * (size_t)a.np : (size_t)a.np) + i]);
        }
        T U[3];
        half_mobility(p, F, ia, ib, U);
        Tagged<T, 3>::put(xb + Xch<T>::kWords * (size_t)i + half * Tagged<T, 3>::kWords, U, tag);
#pragma unroll
        for (int w = 0; w < 3; ++w) Us[6 * li + 3 * half + w] = U[w];
    }
}

// The same with eight lanes per rod, one component each (two idle), for
// shares of few rods, whose entry loops would otherwise leave most of the
// block waiting for a warp or two.
template <typename T>
__device__ __forceinline__ void rod_step8(const SolveArgs<T>& a, const Own1<T>& o, uint4* xb, unsigned tag)
{
    const int nr = o.r1 - o.r0, r0 = o.r0, R = o.cap_r, plane = 4 * (o.nt + 1);
    const T* const row = o.row();
    const ushort4* const ent = reinterpret_cast<const ushort4*>(o.ent());
    const int lane = threadIdx.x & 31, sub = lane & 7, half = sub >= 3, w = half ? (sub < 6 ? sub - 3 : 0) : sub;
    const int own_off = (half ? plane : 0) + w, oth_off = (half ? 2 * plane : 0) + w;
#pragma unroll 1
    for (int tt = first_item(a) >> 3; (tt & ~3) < nr; tt += a.workers >> 3) {   // (uniform per warp)
        const int li = (int)o.perm()[min(tt, nr - 1)];
        const int e1 = tt < nr ? (int)o.rowE()[li + 1] : 0;
        T F = T(0);
#pragma unroll 1
        for (int e = o.rowE()[li]; e < e1; ++e) {
            const ushort4 q = ent[e];
            const unsigned x[4] = {q.x, q.y, q.z, q.w};
            T v[4], r[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const T* p = row + 4 * (int)(x[u] & ~kOther);
                v[u] = signed_by(p[3], x[u]);
                r[u] = p[x[u] & kOther ? oth_off : own_off];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) F = fma(v[u], r[u], F);
        }
        __syncwarp();
        const int i = r0 + li, g0 = (lane & 24) + (half ? 3 : 0);
        const T* const ax = o.ax();
        const T p[3] = {ax[li], ax[R + li], ax[2 * R + li]};
        T Fh[3], U[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) Fh[c] = __shfl_sync(0xffffffffu, F, g0 + c);
        T ia = half ? a.inv_rot : a.inv_perp, ib = half ? a.inv_spin : a.inv_par;
        if (a.mobr) {
            ia = __ldg(&a.mobr[(half ? 2 * (size_t)a.np : 0) + i]);
            ib = __ldg(&a.mobr[(half ? 3 * (size_t)a.np : (size_t)a.np) + i]);
        }
        half_mobility(p, Fh, ia, ib, U);
        if (tt < nr && (sub == 0 || sub == 3)) {
            Tagged<T, 3>::put(xb + Xch<T>::kWords * (size_t)i + half * Tagged<T, 3>::kWords, U, tag);
#pragma unroll
            for (int c = 0; c < 3; ++c) o.U()[6 * li + 3 * half + c] = U[c];
        }
    }
}

// Uref = 0 for the block's rods: shared memory and its rows of the global
// Uref (the velocity the step reports if gamma_0 already meets the tolerance).
template <typename T>
__device__ __forceinline__ void zero_uref1(const SolveArgs<T>& a, const Own1<T>& o)
{
    const int nr = o.r1 - o.r0;
    for (int k = threadIdx.x; k < 6 * o.cap_r; k += blockDim.x) o.U()[k] = T(0);
    typename V2<T>::t z;
    z.x = T(0);
    z.y = T(0);
    typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(a.Uref + 6 * (size_t)o.r0);
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x) g[k] = z;
}

// A halo rod's velocity of exchange tag, polled.
template <typename T>
__device__ __forceinline__ void get_halo(const SolveArgs<T>& a, const Own1<T>& o, int h, const uint4* xb, unsigned tag,
                                         int* bad, T U[6])
{
    get_tagged<T, 6>(a.flags, a.wait_cycles, xb + Xch<T>::kWords * (size_t)o.hrank[h], tag, bad, U);
}

// The halo's velocities of exchange tag into their rows, by the threads with
// the fewest rods first, one rod polled at a time (polling two held the
// publishers up: 2e4 rods 1.46 -> 1.71 ms).
template <typename T>
__device__ __forceinline__ void fetch_halo(const SolveArgs<T>& a, const Own1<T>& o, const uint4* xb, unsigned tag, int* bad)
{
    if (!o.halo || (int)threadIdx.x >= a.workers) return;
    T* const Uh = o.U() + 6 * (o.cap_r + 1);
#pragma unroll 1
    for (int h = a.workers - 1 - (int)threadIdx.x; h < o.nh; h += a.workers) {
        T U[6];
        get_halo(a, o, h, xb, tag, bad, U);
        st_u6(Uh, h, U);
    }
}

// Constraint phase of step k over every slot: from delta_k (which the rod
// phase used), g_k = gref + D^T dU_k (+ the spring's compliance term), for
// owned slots acc = (s.s, s.y, y.y, max |pi|), and delta_{k+1} =
// max(-gamma_ref, delta_k - alpha_k g_k) for the rod phase.  POLL: the halo
// has no rows, its velocities are polled here.
template <typename T, bool POLL>
__device__ __forceinline__ void con_pass_step1(const SolveArgs<T>& a, const Own1<T>& o, T alpha, const uint4* xb,
                                               unsigned tag, int* bad, T acc[4])
{
    const bool has_comp = a.comp != nullptr;
    const int nt = o.nt, nc = o.nc, plane = 4 * (nt + 1), halo = o.cap_r + 1;
    T* const row = o.row();
    const T* const Us = o.U();
    const unsigned* const ij = o.ij();
    T *const ds = o.ds, *const gs = o.gs;
    const T* const isc = a.isc + o.c0;
#pragma unroll 1
    for (int t = first_item(a); t < nt; t += a.workers) {
        const unsigned x = ij[t];
        const int i = (int)(x & 0xffffu), j = (int)(x >> 16);
        T Ui[6], Uj[6];
        T dold = T(0), gold = T(0), is = T(0);
        if (t < nc) { dold = ds[t]; gold = gs[t]; is = __ldg(&isc[t]); }
        if (POLL && i >= halo) get_halo(a, o, i - halo, xb, tag, bad, Ui);
        else ld_u6(Us, i, Ui);
        if (POLL && j >= halo) get_halo(a, o, j - halo, xb, tag, bad, Uj);
        else ld_u6(Us, j, Uj);
        T* const p = row + 4 * t;
        const Row<T> re = ld_row(p), rp = ld_row(p + plane), rq = ld_row(p + 2 * plane);
        const T dm = re.w, gam = rp.w;
        T cmp = T(0);
        bool bil = false;
        if (has_comp) {
            cmp = __ldg(&a.comp[slot_gid(o, t)]);
            bil = cmp >= T(0);
        }
        Acc<T, false> du;
        du.init(rq.w);
        const T r[9] = {re.x, re.y, re.z, rp.x, rp.y, rp.z, rq.x, rq.y, rq.z};
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            du.add_prod(r[u], Ui[u]);
            du.add_prod(-r[u], Uj[u]);
            du.add_prod(r[3 + u], Ui[3 + u]);
            du.add_prod(-r[6 + u], Uj[3 + u]);
        }
        if (bil) du.add_prod(cmp, dm);
        const T gr = du.value();
        p[3] = a_value<A_STEP, T>(dm, gr, gam, alpha, bil);
        if (t < nc) {
            ds[t] = dm;
            gs[t] = gr;
            T pi;
            if constexpr (sizeof(T) == 8) {
                pi = (bil || dm > -gam) ? gr : neg_part(gr);
                acc[3] = max_abs(acc[3], fabs(pi) * is);
            } else {
                pi = (bil || dm > -gam) ? gr : (gr < T(0) ? gr : T(0));
                const T api = (pi < T(0) ? -pi : pi) * is;
                acc[3] = api > acc[3] ? api : acc[3];
            }
            const T sv = dm - dold, yv = gr - gold;
            acc[0] += sv * sv;
            acc[1] += sv * yv;
            acc[2] += yv * yv;
        }
    }
}

// Constraint phase of a refresh over every slot: gref = q + D^T Uref from
// the split records and q with compensated sums (float32), g = gref, and
// for owned slots acc = (pi.pi, 0, 0, max |pi|) at gamma_ref; then, but in
// the initial pass (whose step length is still to come), delta for the step
// from the reference.  ZERO: the initial pass at gamma_0 = 0, where Uref is
// 0, so no velocity is read and the records' products (all zero) are left
// out of the sums.
template <typename T, bool ZERO, bool INITIAL>
__device__ __noinline__ void con_pass_ref1(const SolveArgs<T>& a, const Own1<T>& o, T alpha, T& sum_out, T& max_out)
{
    T acc[4] = {T(0), T(0), T(0), T(0)};
    constexpr bool COMP = sizeof(T) == 4;
    const bool has_comp = a.comp != nullptr;
    const size_t mp = a.mp;
    const int halo = o.cap_r + 1;
#pragma unroll 1
    for (int t = first_item(a); t < o.nt; t += a.workers) {
        T Ui[6], Uj[6], r[9];
        if (!ZERO) {
            const unsigned x = o.ij()[t];
            const int i = (int)(x & 0xffffu), j = (int)(x >> 16);
            if (i >= halo) ld_u6(a.Uref, o.hrank[i - halo], Ui);
            else ld_u6(o.U(), i, Ui);
            if (j >= halo) ld_u6(a.Uref, o.hrank[j - halo], Uj);
            else ld_u6(o.U(), j, Uj);
#pragma unroll
            for (int w = 0; w < 9; ++w) r[w] = slot_row(o, w / 3, t)[w % 3];
        }
        const int c = slot_gid(o, t);
        const T gam = slot_gam(o, t);
        Acc<T, COMP> du;
        du.init(__ldg(&a.q[c]));
        if (!ZERO) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                du.add_prod(r[u], Ui[u]);
                du.add_prod(-r[u], Uj[u]);
                du.add_prod(r[3 + u], Ui[3 + u]);
                du.add_prod(-r[6 + u], Uj[3 + u]);
            }
        }
        const T cmp = has_comp ? __ldg(&a.comp[c]) : T(-1);
        const bool bil = cmp >= T(0);
        if (bil) {
            du.add_prod(cmp, gam);
            du.add_lo(cmp * slot_gref(o, t));   // gamma_lo, before gref takes its place below
        }
        if (COMP) {
            T tl = __ldg(&a.q_lo[c]);
            if (!ZERO) {
                T lp[6], lq[6];   // (e, y_P x e) and (e, y_Q x e) low parts
                lo_side(a.lop, a.rec_lo, mp, c, 3, lp);
                lo_side(a.loq, a.rec_lo, mp, c, 6, lq);
#pragma unroll
                for (int u = 0; u < 3; ++u)
                    tl += fma(-lq[3 + u], Uj[3 + u], fma(lp[u], Ui[u] - Uj[u], lp[3 + u] * Ui[3 + u]));
            }
            du.add_lo(tl);
        }
        const T gr = du.value();
        const T dm = slot_delta(o, t);   // 0 after the fold
        slot_gref(o, t) = gr;
        if (!INITIAL) slot_delta(o, t) = a_value<A_STEP, T>(dm, gr, gam, alpha, bil);
        if (t < o.nc) {
            const T pi = (bil || dm > -gam) ? gr : (gr < T(0) ? gr : T(0));
            const T api = (pi < T(0) ? -pi : pi) * __ldg(&a.isc[c]);
            acc[3] = api > acc[3] ? api : acc[3];
            acc[0] += pi * pi;
            o.ds[t] = dm;
            o.gs[t] = gr;
        }
    }
    sum_out = acc[0];
    max_out = acc[3];
}

// delta_1 of every slot, once alpha_0 is known.
template <typename T>
__device__ __noinline__ void first_step1(const SolveArgs<T>& a, const Own1<T>& o, T alpha)
{
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) {
        const bool bil = a.comp && __ldg(&a.comp[slot_gid(o, t)]) >= T(0);
        slot_delta(o, t) = a_value<A_STEP, T>(slot_delta(o, t), slot_gref(o, t), slot_gam(o, t), alpha, bil);
    }
}

// Refresh, first half: every slot folds delta into (gamma_ref, gamma_lo)
// as fold_delta does, from the previous reference's gamma_lo in gprev;
// ghosts repeat their owner's arithmetic on the same inputs, so both hold
// the same reference without waiting for each other.  gamma_lo goes to the
// place of gref (the reference passes' low part, until the constraint
// pass replaces it), and owned slots publish (gamma_ref, gamma_lo) in
// gnew, the other state buffer (ghosts are still reading gprev).
template <typename T>
__device__ __noinline__ void fold1(const SolveArgs<T>& a, const Own1<T>& o, const T* gprev, T* gnew)
{
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) {
        const int c = slot_gid(o, t);
        const T d = slot_delta(o, t), gr = slot_gam(o, t), gl = gl_of_state(gprev, c);
        const bool bil = a.comp && __ldg(&a.comp[c]) >= T(0);
        T hi = T(0), lo = T(0);
        if (bil || d > -gr) {
            T s, e;
            two_sum(gr, d, s, e);
            const T l = gl + e;
            hi = s + l;
            lo = l - (hi - s);
            if (!bil && (hi < T(0) || (hi == T(0) && lo < T(0)))) { hi = T(0); lo = T(0); }
        }
        slot_gam(o, t) = hi;
        slot_gref(o, t) = lo;
        slot_delta(o, t) = T(0);
        if (t < o.nc) st_ref(gnew, c, hi, lo);
    }
}

// One warp after a block barrier: the block's sums over the workers' red;
// lane 0 holds them.
template <typename T>
__device__ __forceinline__ void block_sums1(T (*red)[4], int nw, T w[4])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < 4; ++u) w[u] = lane < nw ? red[lane][u] : T(0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < 3; ++u) w[u] += __shfl_down_sync(0xffffffffu, w[u], o);
        const T mx = __shfl_down_sync(0xffffffffu, w[3], o);
        w[3] = mx > w[3] ? mx : w[3];
    }
}

// One warp: the grid totals of the tagged block sums at sums ([nb], the
// exchange's slot) in a fixed order, so every block gets the same numbers;
// every lane returns them.  The words of several blocks are in flight
// together.
template <typename T>
__device__ __forceinline__ void grid_sums1(const SolveArgs<T>& a, const uint4* sums, int nb, unsigned tag, int* bad,
                                           T w[4])
{
    constexpr int B = sizeof(T) == 4 ? 5 : 2;
    const int lane = threadIdx.x & 31;
    w[0] = w[1] = w[2] = w[3] = T(0);
    for (int b0 = lane; b0 < nb; b0 += 32 * B) {
        T x[B][4];
        unsigned late = 0;
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (b0 + 32 * u < nb && !XchSum<T>::get(sums + kSumWords * (size_t)(b0 + 32 * u), tag, x[u])) late |= 1u << u;
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (b0 + 32 * u >= nb) break;
            if (late & (1u << u))
                get_tagged<T, 4>(a.flags, a.wait_cycles, sums + kSumWords * (size_t)(b0 + 32 * u), tag, bad, x[u]);
            w[0] += x[u][0];
            w[1] += x[u][1];
            w[2] += x[u][2];
            w[3] = x[u][3] > w[3] ? x[u][3] : w[3];
        }
    }
    __syncwarp();
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
#pragma unroll
        for (int u = 0; u < 3; ++u) w[u] += __shfl_xor_sync(0xffffffffu, w[u], s);
        const T y = __shfl_xor_sync(0xffffffffu, w[3], s);
        w[3] = y > w[3] ? y : w[3];
    }
}

// What an iteration published (its sums decide the next one's step), and
// the decision taken for an iteration.
enum { C_NONE1 = 0, C_STEP1 = 1, C_REF1 = 2 };
enum { K_STEP1 = 0, K_REF1 = 1, K_STOP1 = 2 };

// The decision for the next iteration, by one lane of each block (every
// block decides alike on the same totals); cpub: what the sums are of.
template <typename T>
__device__ __forceinline__ void decide1(const SolveArgs<T>& a, Shared1<T>& sh, int cpub, const T tot[4])
{
    int k = sh.k + 1, next = K_STEP1;
    T an = sh.alpha;
    if (cpub == C_STEP1) {
        // sums of the step before the one just formed, and max |pi| at the iterate before the slots'
        sh.pimax = tot[3];
        const int since = ++sh.since;
        const bool below = !above_tol(a, tot[3]);
        if ((below && since >= 2) || (a.refresh > 0 && since >= a.refresh) || k >= a.max_iter) {
            next = K_REF1;
        } else {
            const T ss = tot[0], sy = tot[1], yy = tot[2];
            an = (sh.hist & 1) == 0 ? ss / sy : sy / yy;
            if (!(sy > T(0)) || !isfinite(an) || !(an > T(0))) an = sh.alpha0;
            ++sh.hist;
        }
    } else if (cpub == C_REF1) {
        // the fresh reference's exact residual: the step formed from it is dropped on a stop
        sh.pimax = tot[3];
        sh.since = 0;
        if (!above_tol(a, tot[3]) || k - 1 >= a.max_iter) {
            next = K_STOP1;
            --k;
        }
    } else if (k >= a.max_iter) {
        next = K_REF1;   // the cap reached before any step's sums came back
    }
    sh.k = k;
    sh.alpha = an;
    sh.kind = next;
}

// MAXT: the most threads of a launch (kThreads1: the default shape and its
// further warp, with 72 registers a thread; 1024: every other shape, with 64).
// Neither holds all it needs: a thread spills 444 bytes (float64; 392 read
// back) or 92 (float32; 252) in the first and 576 or 204 in the second.
constexpr int kThreads1 = 800;
template <typename T, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_bbpgd1(const __grid_constant__ SolveArgs<T> a)
{
    __shared__ Shared1<T> sh;
    if (a.need1_dev) {
        // recorded step: every block reads the same need, so either all run
        // or all leave before their first barrier and ask for an eager step
        const unsigned long long need = *a.need1_dev;
        if (need == 0 || need > (unsigned long long)a.fit_cap) {
            if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[F_SOLVE_ERR] = kSolveRedo;
            return;
        }
    }
    if (a.fault == 1 && blockIdx.x == 0) return;   // test hook: this block never arrives
    Own1<T>& o = sh.o;
    if (threadIdx.x == 0) {
        o.r0 = a.bstart[blockIdx.x];
        o.r1 = a.bstart[blockIdx.x + 1];
        o.c0 = a.rowP[o.r0];
        o.c1 = a.rowP[o.r1];
        o.q0 = a.rowQ[o.r0];
        o.q1 = a.rowQ[o.r1];
        o.nc = o.c1 - o.c0;
        o.cap_r = o.r1 - o.r0;
        sh.bad[0] = sh.bad[1] = 0;
        sh.alpha0 = T(1);
        sh.pimax = T(0);
        sh.k = sh.since = sh.hist = sh.nref = 0;
        sh.epoch = 0;
    }
    __syncthreads();
    // the blocks' tagged sums ([kSumSlots][blocks][kSumWords])
    auto sums = [&](unsigned tag) {
        return a.xch + 2 * Xch<T>::kWords * (size_t)a.n + (size_t)(tag % kSumSlots) * gridDim.x * kSumWords;
    };
    {   // tags of earlier solves away: nobody polls before the first grid barrier
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const size_t w0 = Xch<T>::kWords * (size_t)o.r0, w1 = Xch<T>::kWords * (size_t)o.r1;
        for (size_t w = w0 + threadIdx.x; w < w1; w += blockDim.x) {
            a.xch[w] = z;
            a.xch[Xch<T>::kWords * (size_t)a.n + w] = z;
        }
        for (int w = threadIdx.x; w < kSumSlots * kSumWords; w += blockDim.x)
            sums(w / kSumWords)[blockIdx.x * kSumWords + w % kSumWords] = z;
    }
    stage_in1(a, sh);
    auto barrier = [&]() {
        if (threadIdx.x == 0) ++sh.epoch;
        return grid_barrier(a.bar, gridDim.x * sh.epoch, a.flags, a.wait_cycles, &sh.ng);
    };
    const bool duty = (threadIdx.x >> 5) == (blockDim.x >> 5) - 1;   // sums and decisions

    // initial reference at gamma_0 and the line step alpha_0 = pi.pi / pi.A.pi;
    // from gamma_0 = 0, Uref = M D gamma_0 = 0 needs no rod pass and no
    // other block's velocities
    if (a.zero_start) {
        zero_uref1(a, o);
        __syncthreads();
    } else {
        rod_pass1<T, A_REF>(a, o);
        if (!barrier()) return;
    }
    {
        const int nb = (int)gridDim.x, nbp = (nb + 3) & ~3, lane = threadIdx.x & 31;
        T* const part = reinterpret_cast<T*>(a.partials);   // [4][nbp]
        T v[4] = {T(0), T(0), T(0), T(0)};
        T s0, s3;
        if (a.zero_start) con_pass_ref1<T, true, true>(a, o, T(0), s0, s3);
        else con_pass_ref1<T, false, true>(a, o, T(0), s0, s3);
        v[0] = s0;
        v[3] = s3;
        __syncthreads();   // gref of every slot before the line step reads it
        v[1] = rod_pass1<T, A_PG>(a, o);
        if ((int)threadIdx.x < a.workers) warp_partial(v, sh.red);
        __syncthreads();
        if (duty) {
            T w[4];
            block_sums1(sh.red, a.workers >> 5, w);
            if (lane == 0) {
#pragma unroll
                for (int u = 0; u < 4; ++u) part[u * nbp + blockIdx.x] = w[u];
            }
        }
        __syncthreads();   // red is read
        sort_rods_total(o, reinterpret_cast<int*>(sh.red));
        if (!barrier()) return;
        if (a.fault == 4 && blockIdx.x == 0) return;   // test hook: its words never come
        if (duty) {
            T tot[4] = {T(0), T(0), T(0), T(0)};
            for (int b = lane; b < nb; b += 32) {
#pragma unroll
                for (int u = 0; u < 3; ++u) tot[u] += __ldcg(&part[u * nbp + b]);
                tot[3] = max_of(tot[3], __ldcg(&part[3 * nbp + b]));
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
#pragma unroll
                for (int u = 0; u < 3; ++u) tot[u] += __shfl_xor_sync(0xffffffffu, tot[u], s);
                tot[3] = max_of(tot[3], __shfl_xor_sync(0xffffffffu, tot[3], s));
            }
            if (lane == 0) {
                sh.pimax = tot[3];
                const double pap = (double)tot[1];
                double al = (double)tot[0] / pap;
                if (!(pap > 0.0) || !isfinite(al) || !(al > 0.0) || !isfinite((T)al)) al = 1.0;
                sh.alpha0 = sh.alpha = (T)al;
                sh.kind = (!above_tol(a, tot[3]) || a.max_iter <= 0) ? K_STOP1 : K_STEP1;
            }
        }
        __syncthreads();
    }
    if (sh.kind != K_STOP1) {
        first_step1(a, o, sh.alpha);
        __syncthreads();
    }
    unsigned tag = 0;         // exchanges so far: dU and sums of the last iteration carry it
    while (sh.kind != K_STOP1) {
        const uint4* const xr = a.xch + (tag & 1u) * (Xch<T>::kWords * (size_t)a.n);
        int cpub = C_NONE1;   // what this iteration publishes
        if (tag > 0) {   // the first iteration is the step from gamma_0, already formed
            T v[4] = {T(0), T(0), T(0), T(0)};
            if (sh.kind == K_REF1) {
                fold1(a, o, sh.nref & 1 ? a.gg1 : a.gg0, sh.nref & 1 ? a.gg0 : a.gg1);
                __syncthreads();
                if (threadIdx.x == 0) ++sh.nref;
                rod_pass1<T, A_REF>(a, o);
                if (!barrier()) return;
                T s0, s3;   // (v itself stays in registers)
                con_pass_ref1<T, false, false>(a, o, sh.alpha, s0, s3);
                v[0] = s0;
                v[3] = s3;
                cpub = C_REF1;
            } else {
                if (o.halo) con_pass_step1<T, false>(a, o, sh.alpha, xr, tag, &sh.bad[0], v);
                else con_pass_step1<T, true>(a, o, sh.alpha, xr, tag, &sh.bad[0], v);
                cpub = C_STEP1;
            }
            if ((int)threadIdx.x < a.workers) {
                // (the sums of a warp without owned slots are zero)
                if ((int)(threadIdx.x & ~31u) < o.nc) warp_partial(v, sh.red);
                else if ((threadIdx.x & 31) < 4) sh.red[threadIdx.x >> 5][threadIdx.x & 3] = T(0);
            }
            __syncthreads();
            if (sh.bad[0]) return;
        } else {
            __syncthreads();   // sh.kind is read before the first decision replaces it
        }
        ++tag;
        if (duty && cpub != C_NONE1) {   // this block's sums, while the others run the rod phase
            T w[4];
            block_sums1(sh.red, a.workers >> 5, w);
            if ((threadIdx.x & 31) == 0) XchSum<T>::put(sums(tag) + kSumWords * blockIdx.x, w, tag);
        }
        uint4* const xw = a.xch + (tag & 1u) * (Xch<T>::kWords * (size_t)a.n);
        if (8 * (o.r1 - o.r0) <= a.workers) rod_step8(a, o, xw, tag);
        else rod_step2(a, o, xw, tag);
        fetch_halo(a, o, xw, tag, &sh.bad[1]);
        if (duty) {   // the next iteration's step
            T tot[4];
            if (cpub != C_NONE1) grid_sums1(a, sums(tag), (int)gridDim.x, tag, &sh.bad[1], tot);
            if ((threadIdx.x & 31) == 0) decide1(a, sh, cpub, tot);
        }
        __syncthreads();   // dU and the decision before the next constraint phase
        if (sh.bad[1]) return;
    }
    // every solve ends on a fresh reference: gamma = gamma_ref + gamma_lo
    // (state buffer nref & 1) and delta = 0, so dU = 0
    T* gfin = sh.nref & 1 ? a.gg1 : a.gg0;
    for (int t = threadIdx.x; t < o.nc; t += blockDim.x) st_dg(gfin, o.c0 + t, T(0), slot_gref(o, t));
    {
        typename V2<T>::t z;
        z.x = T(0);
        z.y = T(0);
        typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(a.U + 6 * (size_t)o.r0);
        for (int q = threadIdx.x; q < 3 * (o.r1 - o.r0); q += blockDim.x) g[q] = z;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[1] = (double)sh.alpha0;
        a.flags[F_FINAL] = sh.nref & 1;
        a.flags[F_ITERS] = sh.k;
        a.out[0] = a.hD * (double)sh.pimax;
    }
}

// ---------------------------------------------------------------------
// The same iteration with one grid barrier and without spills, for the
// launches that variant1 names and for large systems whose rods come in no
// spatial order (solve_lcp takes the caller's order): nearly every slot's
// other end then lies in another block, and the halo of tagged words costs more
// to poll than a barrier and plain gathers of the slots' own words (solve, ms,
// barrier / tagged: mixed 8e3 rods 0.70 / 0.56, 1.6e4 0.99 / 0.85, 2e4 1.11 /
// 0.96, 5e4 2.76 / 3.03; float64 1.6e4 5.64 / 4.87, 2e4 5.45 / 4.48: the line
// lies below the crossing).  One thread per rod, a slot's values in columns;
// the sums are the same in the same order, and so is every bit
// (test_barrier_form_repeats_the_tagged_form).
constexpr int kMeetRods = 16000;
namespace meet {

constexpr unsigned kBil = 0x8000u;   // bilateral (spring) constraint: no projection
constexpr int kLocal = 0x7fff;

// A block's share: rods [r0, r1), owned constraints [c0, c1) in slots
// [0, nc), ghosts in slots [nc, nt).
template <typename T>
struct Own1 {
    int r0, r1, c0, c1, q0, q1, nc, ng, nt, cap_r, nbp;
    T* tot;      // [4][nbp] last barrier's block sums (cp.async target)
    T* rec;      // [9][nt]
    T* gref;     // [nt] q + D^T Uref
    T* ds;       // [nt] delta
    T* grs;      // [nt] g
    T* gam;      // [nt] gamma_ref
    T* ax;       // [3][cap_r]
    T* U;        // [6][cap_r] this iteration's dU (the reference velocity during a refresh)
    int* oth;    // [nt] rank of the slot's other end: Q for owned slots, the owner for ghosts (-1: a wall)
    int* gid;    // [ng] constraint id of ghost slot nc + g
    int* rowP;   // [cap_r + 1] owned ranges (constraint ids; slot = id - c0)
    int* rowQ;   // [cap_r + 1] other-side ranges (CSR positions)
    unsigned short* loc;    // [nt] local index of the slot's rod in this block (P owned, Q ghost), | kBil
    unsigned short* qslot;  // [q1 - q0] slot of each other-side entry, | kBil
    unsigned short* perm;   // [cap_r] rod order of the rod phase
};
template <typename T>
__device__ void carve1(Own1<T>& o, unsigned char* base)
{
    const size_t nt = o.nt, R = o.cap_r;
    o.tot = reinterpret_cast<T*>(base);
    base += align16(4 * (size_t)o.nbp * sizeof(T));
    T* t = reinterpret_cast<T*>(base);
    o.rec = t; t += 9 * nt;
    o.gref = t; t += nt;
    o.ds = t; t += nt;
    o.grs = t; t += nt;
    o.gam = t; t += nt;
    o.ax = t; t += 3 * R;
    o.U = t; t += 6 * R;
    base += align16((13 * nt + 9 * R) * sizeof(T));
    int* ip = reinterpret_cast<int*>(base);
    o.oth = ip; ip += nt;
    o.gid = ip; ip += o.ng;
    o.rowP = ip; ip += R + 1;
    o.rowQ = ip; ip += R + 1;
    base += align16((nt + o.ng + 2 * R + 2) * sizeof(int));
    unsigned short* sp = reinterpret_cast<unsigned short*>(base);
    o.loc = sp; sp += nt;
    o.qslot = sp; sp += o.q1 - o.q0;
    o.perm = sp;
}

template <typename T>
struct Shared1 {
    T red[32][4];
    T tot[4];   // grid totals of the last barrier's block sums (warps 1-4, one each)
    T alpha;
    int kind, ng;
};

// Stage one slot (owned or ghost) of constraint c from the global arrays.
template <typename T>
__device__ __forceinline__ void stage_slot(const SolveArgs<T>& a, const Own1<T>& o, int t, int c, int li, int other,
                                           unsigned bil)
{
    const size_t mp = a.mp, nt = o.nt;
#pragma unroll
    for (int w = 0; w < 9; ++w) o.rec[w * nt + t] = a.rec[w * mp + c];
    T d, g, gr, gl;
    ld_state(a.gg0, c, d, g, gr, gl);
    o.ds[t] = d;
    o.gam[t] = gr;
    o.grs[t] = gl;   // gamma_lo until the first reference pass replaces it by g
    o.gref[t] = T(0);
    o.oth[t] = other;
    o.loc[t] = (unsigned short)(li | bil);
}

template <typename T>
__device__ void stage_in1(const SolveArgs<T>& a, Own1<T>& o, unsigned char* dyn, Shared1<T>& sh)
{
    const int nr = o.r1 - o.r0, nq = o.q1 - o.q0;
    // ghosts: other-side entries of the block's rods that another block owns
    if (threadIdx.x == 0) sh.ng = 0;
    __syncthreads();
    int cnt = 0;
    for (int k = threadIdx.x; k < nq; k += blockDim.x) {
        const int c = a.qlist[o.q0 + k];
        cnt += c < o.c0 || c >= o.c1;
    }
    if (cnt) atomicAdd(&sh.ng, cnt);
    __syncthreads();
    o.ng = sh.ng;
    o.nt = o.nc + o.ng;
    carve1(o, dyn);
    __syncthreads();
    if (threadIdx.x == 0) sh.ng = 0;
    for (int li = threadIdx.x; li <= nr; li += blockDim.x) {
        o.rowP[li] = a.rowP[o.r0 + li];
        o.rowQ[li] = a.rowQ[o.r0 + li];
    }
    for (int li = threadIdx.x; li < nr; li += blockDim.x)
        for (int w = 0; w < 3; ++w) o.ax[w * o.cap_r + li] = a.ax[w * (size_t)a.np + o.r0 + li];
    const bool has_comp = a.comp != nullptr;
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nc; t += blockDim.x) {
        const int c = o.c0 + t;
        const unsigned bil = has_comp && a.comp[c] >= T(0) ? kBil : 0u;
        stage_slot(a, o, t, c, a.ci[c] - o.r0, a.cj[c], bil);
    }
    __syncthreads();   // sh.ng is 0 again before the slots are numbered
#pragma unroll 1
    for (int k = threadIdx.x; k < nq; k += blockDim.x) {
        const int c = a.qlist[o.q0 + k];
        const unsigned bil = has_comp && a.comp[c] >= T(0) ? kBil : 0u;
        int t;
        if (c < o.c0 || c >= o.c1) {
            // the slot order of ghosts does not enter any result
            const int g = atomicAdd(&sh.ng, 1);
            t = o.nc + g;
            o.gid[g] = c;
            stage_slot(a, o, t, c, a.cj[c] - o.r0, a.ci[c], bil);
        } else {
            t = c - o.c0;
        }
        o.qslot[k] = (unsigned short)(t | bil);
    }
    __syncthreads();
    sort_rods(o.rowP, o.rowQ, nr, reinterpret_cast<unsigned*>(o.U), reinterpret_cast<int*>(o.U) + nr, o.perm);
}

template <typename T>
__device__ __forceinline__ int slot_gid(const Own1<T>& o, int t)
{
    return t < o.nc ? o.c0 + t : o.gid[t - o.nc];
}

// Rod phase over the block's rods, every entry from shared memory (modes
// as for phase_a: A_STEP forms delta_{k+1} with alpha and leaves dU in
// shared memory; A_PG returns this thread's share of pi.A.pi; A_REF leaves
// Uref = M D gamma_ref (compensated in float32) in shared memory and in
// the global Uref).
template <typename T, int MODE>
__device__ __forceinline__ T rod_pass1(const SolveArgs<T>& a, const Own1<T>& o, T alpha)
{
    constexpr bool COMP = MODE == A_REF && sizeof(T) == 4;
    const bool has_comp = a.comp != nullptr;
    const size_t mp = a.mp, np = a.np, nt = o.nt;
    T fmf = T(0);
#pragma unroll 1
    for (int tt = threadIdx.x; tt < o.r1 - o.r0; tt += blockDim.x) {
        const int li = (int)o.perm[tt], i = o.r0 + li;
        Acc<T, COMP> Fa[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) Fa[w].init(T(0));
        {   // owned constraints: slots [rowP[li] - c0, rowP[li + 1] - c0)
            const int e = o.rowP[li + 1] - o.c0;
#pragma unroll 1
            for (int t = o.rowP[li] - o.c0; t < e; ++t) {
                const T dv = o.ds[t], gv = o.grs[t], gr = o.gam[t];
                T rv[6];
#pragma unroll
                for (int w = 0; w < 6; ++w) rv[w] = o.rec[w * nt + t];
                const bool bil = has_comp && (o.loc[t] & kBil);
                const T v = a_value<MODE, T>(dv, gv, gr, alpha, bil);
                if (MODE == A_PG && bil) fmf += __ldg(&a.comp[o.c0 + t]) * v * v;   // the spring's compliance term
#pragma unroll
                for (int w = 0; w < 6; ++w) Fa[w].add_prod(v, rv[w]);
                if (COMP) {   // gamma_lo (held in grs during a reference pass) and the records' low parts
                    const int c = o.c0 + t;
                    const T gl = gv;
                    T rl[6];
                    lo_side(a.lop, a.rec_lo, mp, c, 3, rl);
#pragma unroll
                    for (int w = 0; w < 6; ++w) Fa[w].add_lo(fma(v, rl[w], gl * rv[w]));
                }
            }
        }
        {   // constraints owned by other rods (owned or ghost slots)
            const int e = o.rowQ[li + 1] - o.q0;
#pragma unroll 1
            for (int k = o.rowQ[li] - o.q0; k < e; ++k) {
                const unsigned qs = o.qslot[k];
                const int t = (int)(qs & kLocal);
                const T dv = o.ds[t], gv = o.grs[t], gr = o.gam[t];
                T qv[6];
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    qv[w] = o.rec[w * nt + t];
                    qv[3 + w] = o.rec[(6 + w) * nt + t];
                }
                const T v = a_value<MODE, T>(dv, gv, gr, alpha, has_comp && (qs & kBil));
#pragma unroll
                for (int w = 0; w < 6; ++w) Fa[w].add_prod(-v, qv[w]);
                if (COMP) {
                    const int c = slot_gid(o, t);
                    const T gl = gv;
                    T ql[6];
                    lo_side(a.loq, a.rec_lo, mp, c, 6, ql);
#pragma unroll
                    for (int w = 0; w < 6; ++w) Fa[w].add_lo(-fma(v, ql[w], gl * qv[w]));
                }
            }
        }
        T F[6];
#pragma unroll
        for (int w = 0; w < 6; ++w) F[w] = Fa[w].value();
        const T p0 = o.ax[li], p1 = o.ax[o.cap_r + li], p2 = o.ax[2 * o.cap_r + li];
        T ip = a.inv_perp, ipa = a.inv_par, ir = a.inv_rot, is = a.inv_spin;
        if (a.mobr) {
            ip = __ldg(&a.mobr[i]); ipa = __ldg(&a.mobr[np + i]);
            ir = __ldg(&a.mobr[2 * np + i]); is = __ldg(&a.mobr[3 * np + i]);
        }
        const T p[3] = {p0, p1, p2};
        T Uv[6];
        half_mobility(p, F, ip, ipa, Uv);
        half_mobility(p, F + 3, ir, is, Uv + 3);
        if (MODE == A_PG) {
#pragma unroll
            for (int w = 0; w < 6; ++w) fmf += F[w] * Uv[w];
        } else {
#pragma unroll
            for (int w = 0; w < 6; ++w) o.U[w * o.cap_r + li] = Uv[w];
            if (MODE == A_REF) st_u6(a.Uref, i, Uv);
        }
    }
    return fmf;
}

// The block's dU (shared [6][cap_r]) into its contiguous range of the
// global [n][6] buffer dst, consecutive threads writing consecutive pairs.
template <typename T>
__device__ __forceinline__ void copy_out1(T* dst, const Own1<T>& o)
{
    __syncthreads();
    const int nr = o.r1 - o.r0;
    typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(dst + 6 * (size_t)o.r0);
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x) {
        const int r = k / 3, w = 2 * (k - 3 * r);
        typename V2<T>::t v;
        v.x = o.U[w * o.cap_r + r];
        v.y = o.U[(w + 1) * o.cap_r + r];
        g[k] = v;
    }
}

// Uref = 0 for the block's rods: shared memory and its rows of the global
// Uref (the velocity the step reports if gamma_0 already meets the tolerance).
template <typename T>
__device__ __forceinline__ void zero_uref1(const SolveArgs<T>& a, const Own1<T>& o)
{
    const int nr = o.r1 - o.r0;
    for (int k = threadIdx.x; k < 6 * o.cap_r; k += blockDim.x) o.U[k] = T(0);
    typename V2<T>::t z;
    z.x = T(0);
    z.y = T(0);
    typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(a.Uref + 6 * (size_t)o.r0);
    for (int k = threadIdx.x; k < 3 * nr; k += blockDim.x) g[k] = z;
}

// The two velocities of slot t, P side first: Ui of the owner, Uj of the
// other end (0 for a wall).  Local rods from shared memory, others from the
// global buffer Ug.
template <typename T>
__device__ __forceinline__ void slot_velocities(const Own1<T>& o, int t, const T* Ug, T Ui[6], T Uj[6])
{
    const int li = (int)(o.loc[t] & kLocal);
    const int ro = o.oth[t];
    T Ul[6], Uo[6];
#pragma unroll
    for (int w = 0; w < 6; ++w) Ul[w] = o.U[w * o.cap_r + li];
    if (ro < 0) {
#pragma unroll
        for (int w = 0; w < 6; ++w) Uo[w] = T(0);
    } else if (ro >= o.r0 && ro < o.r1) {
#pragma unroll
        for (int w = 0; w < 6; ++w) Uo[w] = o.U[w * o.cap_r + (ro - o.r0)];
    } else {
        ld_u6(Ug, ro, Uo);
    }
    const bool own = t < o.nc;
#pragma unroll
    for (int w = 0; w < 6; ++w) {
        Ui[w] = own ? Ul[w] : Uo[w];
        Uj[w] = own ? Uo[w] : Ul[w];
    }
}

// Constraint phase of a step over every slot: delta_k from
// (delta_{k-1}, g_{k-1}, alpha_{k-1}) exactly as the rod phase formed it,
// g_k = gref + D^T dU_k (+ the spring's compliance term), and for owned
// slots acc = (s.s, s.y, y.y, max |pi|).
template <typename T>
__device__ __forceinline__ void con_pass_step1(const SolveArgs<T>& a, const Own1<T>& o, T alpha, const T* Ug, T acc[4])
{
    const bool has_comp = a.comp != nullptr;
    const size_t nt = o.nt;
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) {
        T Ui[6], Uj[6], r[9];
        slot_velocities(o, t, Ug, Ui, Uj);
#pragma unroll
        for (int w = 0; w < 9; ++w) r[w] = o.rec[w * nt + t];
        const T dold = o.ds[t], gro = o.grs[t], gam = o.gam[t];
        const int c = slot_gid(o, t);
        const T cmp = has_comp ? __ldg(&a.comp[c]) : T(-1);
        const bool bil = cmp >= T(0);
        const T dm = a_value<A_STEP, T>(dold, gro, gam, alpha, bil);
        Acc<T, false> du;
        du.init(o.gref[t]);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
            du.add_prod(r[u], Ui[u]);
            du.add_prod(-r[u], Uj[u]);
            du.add_prod(r[3 + u], Ui[3 + u]);
            du.add_prod(-r[6 + u], Uj[3 + u]);
        }
        if (bil) du.add_prod(cmp, dm);
        const T gr = du.value();
        o.ds[t] = dm;
        o.grs[t] = gr;
        if (t < o.nc) {
            const T pi = (bil || dm > -gam) ? gr : (gr < T(0) ? gr : T(0));
            const T api = (pi < T(0) ? -pi : pi) * __ldg(&a.isc[c]);
            acc[3] = api > acc[3] ? api : acc[3];
            const T sv = dm - dold, yv = gr - gro;
            acc[0] += sv * sv;
            acc[1] += sv * yv;
            acc[2] += yv * yv;
        }
    }
}

// Constraint phase of a refresh over every slot: gref = q + D^T Uref from
// the split records and q with compensated sums (float32), g = gref, and
// for owned slots acc = (pi.pi, 0, 0, max |pi|) at gamma_ref.  ZERO: Uref
// is 0 (gamma_ref = 0), so no velocity is read and the records' products
// (all zero) are left out of the sums.
template <typename T, bool ZERO = false>
__device__ __forceinline__ void con_pass_ref1(const SolveArgs<T>& a, const Own1<T>& o, T acc[4])
{
    constexpr bool COMP = sizeof(T) == 4;
    const bool has_comp = a.comp != nullptr;
    const size_t nt = o.nt, mp = a.mp;
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) {
        T Ui[6], Uj[6], r[9];
        if (!ZERO) {
            slot_velocities(o, t, a.Uref, Ui, Uj);
#pragma unroll
            for (int w = 0; w < 9; ++w) r[w] = o.rec[w * nt + t];
        }
        const int c = slot_gid(o, t);
        const T gam = o.gam[t];
        Acc<T, COMP> du;
        du.init(__ldg(&a.q[c]));
        if (!ZERO) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                du.add_prod(r[u], Ui[u]);
                du.add_prod(-r[u], Uj[u]);
                du.add_prod(r[3 + u], Ui[3 + u]);
                du.add_prod(-r[6 + u], Uj[3 + u]);
            }
        }
        const T cmp = has_comp ? __ldg(&a.comp[c]) : T(-1);
        const bool bil = cmp >= T(0);
        if (bil) {
            du.add_prod(cmp, gam);
            du.add_lo(cmp * o.grs[t]);   // gamma_lo, before g takes its place below
        }
        if (COMP) {
            T tl = __ldg(&a.q_lo[c]);
            if (!ZERO) {
                T lp[6], lq[6];   // (e, y_P x e) and (e, y_Q x e) low parts
                lo_side(a.lop, a.rec_lo, mp, c, 3, lp);
                lo_side(a.loq, a.rec_lo, mp, c, 6, lq);
#pragma unroll
                for (int u = 0; u < 3; ++u)
                    tl += fma(-lq[3 + u], Uj[3 + u], fma(lp[u], Ui[u] - Uj[u], lp[3 + u] * Ui[3 + u]));
            }
            du.add_lo(tl);
        }
        const T gr = du.value();
        o.gref[t] = gr;
        o.grs[t] = gr;
        if (t < o.nc) {
            const T dm = o.ds[t];   // 0 after the fold
            const T pi = (bil || dm > -gam) ? gr : (gr < T(0) ? gr : T(0));
            const T api = (pi < T(0) ? -pi : pi) * __ldg(&a.isc[c]);
            acc[3] = api > acc[3] ? api : acc[3];
            acc[0] += pi * pi;
        }
    }
}

// Refresh, first half: every slot folds delta into (gamma_ref, gamma_lo)
// as fold_delta does, from the previous reference's gamma_lo in gprev;
// ghosts repeat their owner's arithmetic on the same inputs, so both hold
// the same reference without waiting for each other.  gamma_ref goes to
// gam, gamma_lo to grs (the reference passes' low part, until the constraint
// pass replaces it by g), and owned slots publish (gamma_ref, gamma_lo) in
// gnew, the other state buffer (ghosts are still reading gprev).
template <typename T>
__device__ __forceinline__ void fold1(const SolveArgs<T>& a, const Own1<T>& o, const T* gprev, T* gnew)
{
    const bool has_comp = a.comp != nullptr;
#pragma unroll 1
    for (int t = threadIdx.x; t < o.nt; t += blockDim.x) {
        const int c = slot_gid(o, t);
        const T d = o.ds[t], gr = o.gam[t], gl = gl_of_state(gprev, c);
        const bool bil = has_comp && (o.loc[t] & kBil);
        T hi = T(0), lo = T(0);
        if (bil || d > -gr) {
            T s, e;
            two_sum(gr, d, s, e);
            const T l = gl + e;
            hi = s + l;
            lo = l - (hi - s);
            if (!bil && (hi < T(0) || (hi == T(0) && lo < T(0)))) { hi = T(0); lo = T(0); }
        }
        o.gam[t] = hi;
        o.grs[t] = lo;
        o.ds[t] = T(0);
        if (t < o.nc) st_ref(gnew, c, hi, lo);
    }
}

// cp.async of the last barrier's block sums ([4][nbp] of buffer src) into
// shared memory; the threads that issue it wait for it in tot_wait.
template <typename T>
__device__ __forceinline__ void tot_fetch(const Own1<T>& o, const T* src)
{
    const int chunks = (int)(4 * (size_t)o.nbp * sizeof(T) / 16);
    if ((int)threadIdx.x < chunks) {
        for (int q = threadIdx.x; q < chunks; q += blockDim.x) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(reinterpret_cast<unsigned char*>(o.tot) + 16 * (size_t)q);
            const unsigned char* s = reinterpret_cast<const unsigned char*>(src) + 16 * (size_t)q;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(s) : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
}
__device__ __forceinline__ void tot_wait() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Warp w's share of the block sums: each warp's (sum, sum, sum, max) into red[w].
template <typename T>
__device__ __forceinline__ void warp_partial(T v[4], T (*red)[4])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < 3; ++u) v[u] += __shfl_down_sync(0xffffffffu, v[u], o);
        const T mx = __shfl_down_sync(0xffffffffu, v[3], o);
        v[3] = mx > v[3] ? mx : v[3];
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) red[threadIdx.x >> 5][u] = v[u];
    }
}

// Warp 0 after a block barrier: the block's sums over red, lane 0 stores
// them in dst ([4][stride]).
template <typename T>
__device__ __forceinline__ void block_store(T (*red)[4], T* dst, int stride)
{
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    T w[4] = {T(0), T(0), T(0), T(0)};
    if (lane < nw) {
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = red[lane][u];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int u = 0; u < 3; ++u) w[u] += __shfl_down_sync(0xffffffffu, w[u], o);
        const T mx = __shfl_down_sync(0xffffffffu, w[3], o);
        w[3] = mx > w[3] ? mx : w[3];
    }
    if (lane == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) dst[u * stride + blockIdx.x] = w[u];
    }
}

// One warp: the grid total of row u of the fetched block sums (sums for
// u < 3, the maximum for u = 3), in a fixed order, so every block gets the
// same numbers; every lane returns it.
template <typename T>
__device__ __forceinline__ T row_total(const Own1<T>& o, int nb, int u)
{
    const int lane = threadIdx.x & 31;
    const T* row = o.tot + (size_t)u * o.nbp;
    T w = T(0);
    for (int b = lane; b < nb; b += 32) {
        const T x = row[b];
        w = u == 3 ? (x > w ? x : w) : w + x;
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const T y = __shfl_xor_sync(0xffffffffu, w, s);
        w = u == 3 ? (y > w ? y : w) : w + y;
    }
    return w;
}

// The four totals, one warp each: warps 1-4 store them in shared memory and
// meet on a named barrier (warp 0 meanwhile stores the block's own sums).
template <typename T>
__device__ __forceinline__ void warps_totals(const Own1<T>& o, int nb, T* tot)
{
    const int u = (int)(threadIdx.x >> 5) - 1;
    const T w = row_total(o, nb, u);
    if ((threadIdx.x & 31) == 0) tot[u] = w;
    asm volatile("bar.sync 1, 128;\n" ::: "memory");
}

template <typename T>
__global__ void __launch_bounds__(1024, 1) k_bbpgd1_meet(SolveArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ Shared1<T> sh;
    if (a.need1_dev) {   // recorded step: as in k_bbpgd1
        const unsigned long long need = *a.need1_dev;
        if (need == 0 || need > (unsigned long long)a.fit_cap) {
            if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[F_SOLVE_ERR] = kSolveRedo;
            return;
        }
    }
    if (a.fault == 1 && blockIdx.x == 0) return;   // test hook: this block never arrives
    Own1<T> o;
    o.r0 = a.bstart[blockIdx.x];
    o.r1 = a.bstart[blockIdx.x + 1];
    o.c0 = a.rowP[o.r0];
    o.c1 = a.rowP[o.r1];
    o.q0 = a.rowQ[o.r0];
    o.q1 = a.rowQ[o.r1];
    o.nc = o.c1 - o.c0;
    o.cap_r = o.r1 - o.r0;
    const int nb = (int)gridDim.x;
    o.nbp = (nb + 3) & ~3;
    stage_in1(a, o, dyn, sh);
    T* const dU2 = reinterpret_cast<T*>(a.xch);   // the second velocity buffer [n][6]
    T* part = reinterpret_cast<T*>(a.partials);   // [2][4][nbp]
    const size_t pstride = 4 * (size_t)o.nbp;
    unsigned epoch = 0;
    int* s_ok = &sh.ng;   // the barrier's broadcast word (ng is not needed after staging)
    auto barrier = [&]() { return grid_barrier(a.bar, (unsigned)nb * ++epoch, a.flags, a.wait_cycles, s_ok); };
    const int warp = threadIdx.x >> 5;
    // step state, kept by thread 32 (warp 1, lane 0)
    T alpha0 = T(1), pimax = T(0);
    int k = 0, since = 0, hist = 0;
    bool ok = true;

    // initial reference at gamma_0 and the line step alpha_0 = pi.pi / pi.A.pi;
    // from gamma_0 = 0, Uref = M D gamma_0 = 0 needs no rod pass and no
    // other block's velocities
    if (a.zero_start) {
        zero_uref1(a, o);
        __syncthreads();
    } else {
        rod_pass1<T, A_REF>(a, o, T(0));
        ok = barrier();
    }
    int pw = 0;   // block-sum buffer the next barrier publishes
    if (ok) {
        T v[4] = {T(0), T(0), T(0), T(0)};
        if (a.zero_start) con_pass_ref1<T, true>(a, o, v);
        else con_pass_ref1(a, o, v);
        __syncthreads();   // gref and g of every slot before the line step reads them
        v[1] = rod_pass1<T, A_PG>(a, o, T(0));
        warp_partial(v, sh.red);
        __syncthreads();
        if (warp == 0) block_store(sh.red, part + pw * pstride, o.nbp);
        ok = barrier();
    }
    if (ok) {
        tot_fetch(o, part + pw * pstride);
        tot_wait();
        __syncthreads();
        if (warp >= 1 && warp <= 4) {
            warps_totals(o, nb, sh.tot);
            const T* tot = sh.tot;
            if (threadIdx.x == 32) {
                pimax = tot[3];
                const double pap = (double)tot[1];
                double al = (double)tot[0] / pap;
                if (!(pap > 0.0) || !isfinite(al) || !(al > 0.0) || !isfinite((T)al)) al = 1.0;
                alpha0 = (T)al;
                sh.alpha = alpha0;
                sh.kind = (!above_tol(a, pimax) || a.max_iter <= 0) ? K_STOP1 : K_STEP1;
            }
        }
        __syncthreads();
        pw ^= 1;
    }
    int cprev = C_NONE1;      // the constraint phase whose sums the last barrier published
    bool rstep = false;       // the last rod phase formed a step (its delta is still to be stored)
    T alpha_prev = T(0);
    int db = 0;               // dU buffer the next step's rod phase writes
    int nref = 0;             // refreshes taken: the reference lives in state buffer nref & 1
    while (ok && sh.kind != K_STOP1) {
        const int pr = pw ^ 1;   // buffer the last barrier published
        if (cprev != C_NONE1) tot_fetch(o, part + pr * pstride);
        T v[4] = {T(0), T(0), T(0), T(0)};
        if (rstep) con_pass_step1(a, o, alpha_prev, db ? a.U : dU2, v);
        const int ccur = rstep ? C_STEP1 : C_NONE1;
        warp_partial(v, sh.red);
        tot_wait();
        __syncthreads();
        if (warp == 0) {
            block_store(sh.red, part + pw * pstride, o.nbp);
        } else if (warp <= 4) {
            if (cprev != C_NONE1) warps_totals(o, nb, sh.tot);
            const T* tot = sh.tot;
            if (threadIdx.x == 32) {
                if (rstep) ++k;
                int kind = K_STEP1;
                T an = sh.alpha;
                if (cprev == C_STEP1) {
                    // sums of (s_{k-2}, y_{k-2}) and max |pi| at the iterate before the slots'
                    pimax = tot[3];
                    ++since;
                    const bool below = !above_tol(a, pimax);
                    if ((below && since >= 2) || (a.refresh > 0 && since >= a.refresh) || k >= a.max_iter) {
                        kind = K_REF1;
                    } else {
                        const T ss = tot[0], sy = tot[1], yy = tot[2];
                        an = (hist & 1) == 0 ? ss / sy : sy / yy;
                        if (!(sy > T(0)) || !isfinite(an) || !(an > T(0))) an = alpha0;
                        ++hist;
                    }
                } else if (cprev == C_REF1) {
                    // the fresh reference's exact residual: the slots' step from it is dropped on a stop
                    pimax = tot[3];
                    since = 0;
                    if (!above_tol(a, pimax) || k - 1 >= a.max_iter) {
                        kind = K_STOP1;
                        --k;
                    }
                } else if (k >= a.max_iter) {
                    kind = K_REF1;   // the cap reached before any step's sums came back
                }
                sh.alpha = an;
                sh.kind = kind;
            }
        }
        __syncthreads();
        const int kind = sh.kind;
        if (kind == K_STOP1) break;
        int cpub = ccur;
        if (kind == K_REF1) {
            fold1(a, o, nref & 1 ? a.gg1 : a.gg0, nref & 1 ? a.gg0 : a.gg1);
            ++nref;
            __syncthreads();
            rod_pass1<T, A_REF>(a, o, T(0));
            if (!(ok = barrier())) break;
            T w[4] = {T(0), T(0), T(0), T(0)};
            con_pass_ref1(a, o, w);
            warp_partial(w, sh.red);
            __syncthreads();
            if (warp == 0) block_store(sh.red, part + pw * pstride, o.nbp);
            cpub = C_REF1;
        }
        const T al = sh.alpha;
        rod_pass1<T, A_STEP>(a, o, al);
        copy_out1(db ? dU2 : a.U, o);
        alpha_prev = al;
        rstep = true;
        db ^= 1;
        if (!(ok = barrier())) break;
        pw ^= 1;
        cprev = cpub;
    }
    if (!ok) return;
    // every solve ends on a fresh reference: gamma = gamma_ref + gamma_lo
    // (state buffer nref & 1) and delta = 0, so dU = 0
    T* gfin = nref & 1 ? a.gg1 : a.gg0;
    for (int t = threadIdx.x; t < o.nc; t += blockDim.x) st_dg(gfin, o.c0 + t, T(0), o.gref[t]);
    {
        typename V2<T>::t z;
        z.x = T(0);
        z.y = T(0);
        typename V2<T>::t* g = reinterpret_cast<typename V2<T>::t*>(a.U + 6 * (size_t)o.r0);
        for (int q = threadIdx.x; q < 3 * (o.r1 - o.r0); q += blockDim.x) g[q] = z;
    }
    if (blockIdx.x == 0 && threadIdx.x == 32) {
        a.out[1] = (double)alpha0;
        a.flags[F_FINAL] = nref & 1;
        a.flags[F_ITERS] = k;
        a.out[0] = a.hD * (double)pimax;
    }
}

}  // namespace meet

// The work-balanced split and what its shares need, one thread block per solver block b
// in one launch: the share's two boundaries (bstart; a warp
// each), the two-barrier kernel's largest shared-memory share and rod count
// over the blocks (need, maxrods), and the one-barrier kernel's (need1; ghosts
// counted from the block's other-side entries; a share whose slot or rod
// count exceeds the 15-bit local indices does not fit).  Also zeroes the
// solver's barrier words.  The three counters are zero before (reset with the step's).
constexpr int kNeedThreads = 256;
__global__ void __launch_bounds__(kNeedThreads)
k_shares(int n, int nb, int esize, const int* __restrict__ rowP, const int* __restrict__ rowQ,
         const int* __restrict__ qlist, int* __restrict__ bstart, unsigned* __restrict__ bar,
         unsigned long long* __restrict__ need, unsigned long long* __restrict__ maxrods,
         unsigned long long* __restrict__ need1)
{
    __shared__ int wsum[kNeedThreads / 32], bound[2];
    const int b = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 2) {
        const int k = b + warp;
        const long long total = rank_work(rowP, rowQ, n);
        const int r = k == nb ? n : find_rank(rowP, rowQ, 0, n, total * k / nb);
        if (lane == 0) {
            bound[warp] = r;
            if (warp == 0 || k == nb) bstart[k] = r;
        }
    }
    if (b == 0 && threadIdx.x < 4) bar[threadIdx.x] = 0u;
    __syncthreads();
    const int r0 = bound[0], r1 = bound[1];
    const int c0 = rowP[r0], c1 = rowP[r1], q0 = rowQ[r0], q1 = rowQ[r1];
    int ng = 0;
    for (int k = q0 + (int)threadIdx.x; k < q1; k += kNeedThreads) {
        const int c = qlist[k];
        ng += c < c0 || c >= c1;
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) ng += __shfl_down_sync(0xffffffffu, ng, s);
    if (lane == 0) wsum[warp] = ng;
    __syncthreads();
    if (threadIdx.x == 0) {
        ng = 0;
        for (int w = 0; w < kNeedThreads / 32; ++w) ng += wsum[w];
        const size_t nc = (size_t)(c1 - c0), nt = nc + ng, nr = r1 - r0, nq = q1 - q0;
        atomicMax(need, (unsigned long long)staged_bytes(esize, nc, nr, nq));
        atomicMax(maxrods, (unsigned long long)nr);
        unsigned long long bytes = staged1_bytes(esize, nt, ng, nr, nq, nb);
        if (nt > (size_t)kMaxSlots || nr > (size_t)kMaxSlots) bytes = ~0ull;
        atomicMax(need1, bytes);
    }
}

// Batches: every cluster takes whole systems from a queue (largest first)
// and runs the BBPGD of each on its own, with the system's own step sizes,
// residual and stopping test.  A system's rods are the contiguous ranks
// [sysoff[s], sysoff[s+1]) and its constraints the contiguous owner-major
// range they own, so each block of the cluster takes a work-balanced share
// of them exactly as the grid solver does.  The queue's entries (qent:
// system, pair code) list the largest systems twice: the two clusters that
// take them solve the system together as one group of twice the blocks (a
// pair; code = 2 * pair + member), so that no single system's solve outlasts
// the rest of the queue.  Which systems are paired depends only on the
// systems and the launch, so every step computes the same numbers.  The
// final state is left in buffer 0; per-system iterations and residuals are
// written out, and the largest of each into the step's counters.
template <typename T>
__global__ void __launch_bounds__(1024, 1)
k_bbpgd_sys(SolveArgs<T> a, const long long* __restrict__ sysoff, const int* __restrict__ qent,
            const int* __restrict__ qn, unsigned* __restrict__ pair_bar, unsigned long long* __restrict__ queue,
            int* __restrict__ sys_iters, int* __restrict__ sys_blocks, double* __restrict__ sys_res)
{
    extern __shared__ __align__(16) unsigned char dyn[];   // rod order scratch (when a.sort_ns)
    __shared__ Shared<T> sh;
    __shared__ int bounds[2];
    cg::cluster_group cl = cg::this_cluster();
    const int crank = (int)cl.block_rank(), cs = (int)cl.num_blocks();
    const int nq = *qn;
    for (;;) {
        if (crank == 0 && threadIdx.x == 0) {
            const unsigned long long k = atomicAdd(queue, 1ull);
            sh.sys = k < (unsigned long long)nq ? qent[2 * k] : -1;
            sh.pair = k < (unsigned long long)nq ? qent[2 * k + 1] : -1;
        }
        cl.sync();
        const int s = *cl.map_shared_rank(&sh.sys, 0);
        const int pc = *cl.map_shared_rank(&sh.pair, 0);
        cl.sync();   // every block has the entry before block 0 takes the next one
        if (s < 0) break;
        const int member = pc >= 0 ? (pc & 1) : 0;
        if (a.fault == 1 && member == 1) {   // test hook: a pair's second cluster never arrives
            __syncthreads();
            continue;
        }
        const int gs = pc >= 0 ? 2 * cs : cs, grank = member * cs + crank;   // the group's blocks, this one's rank
        const int R0 = (int)sysoff[s], R1 = (int)sysoff[s + 1];
        if (threadIdx.x < 64) {   // warp w finds end w of this block's share
            const int w = threadIdx.x >> 5, k = grank + w;
            const long long W0 = rank_work(a.rowP, a.rowQ, R0), W1 = rank_work(a.rowP, a.rowQ, R1);
            const int r = k == 0 ? R0 : (k == gs ? R1 : find_rank(a.rowP, a.rowQ, R0, R1, W0 + (W1 - W0) * k / gs));
            if ((threadIdx.x & 31) == 0) bounds[w] = r;
        }
        __syncthreads();
        Own<T> o;
        o.perm = nullptr;
        o.r0 = bounds[0];
        o.r1 = bounds[1];
        if (a.sort_ns && o.r1 - o.r0 <= a.sort_cap) {   // the block's share in entry-count order
            const int nr = o.r1 - o.r0;
            unsigned* key = reinterpret_cast<unsigned*>(dyn);
            int* rk = reinterpret_cast<int*>(key + nr);
            o.perm = reinterpret_cast<unsigned short*>(rk + nr);
            sort_rods(a.rowP + o.r0, a.rowQ + o.r0, nr, key, rk, o.perm);
        }
        o.c0 = a.rowP[o.r0];
        o.c1 = a.rowP[o.r1];
        o.q0 = a.rowQ[o.r0];
        o.q1 = a.rowQ[o.r1];
        o.cap_c = o.c1 - o.c0;
        o.cap_r = o.r1 - o.r0;
        o.cap_q = o.q1 - o.q0;
        BatchSync<T> sy;
        sy.bar = pc >= 0 ? pair_bar + (pc >> 1) : nullptr;
        sy.flags = a.flags;
        sy.wait_cycles = a.wait_cycles;
        sy.partials = reinterpret_cast<T*>(a.partials) + (pc >= 0 ? (size_t)(pc >> 1) * 4 * kPairBlocks : 0);
        sy.nb = (unsigned)gs;
        sy.epoch = 0;
        sy.rank = grank;
        StepState<T> st;
        solve_loop<T, false>(a, o, sh, sy, st);
        if (sh.cur == 1) {
            for (int c = o.c0 + threadIdx.x; c < o.c1; c += blockDim.x) {
                T d, g, gr, gl;
                ld_state(a.gg1, c, d, g, gr, gl);
                st_dg(a.gg0, c, d, g);
                st_ref(a.gg0, c, gr, gl);
            }
        }
        if (grank == 0 && threadIdx.x == 0) {
            sys_iters[s] = st.iters;
            sys_blocks[s] = gs;
            const double res = st.residual(a.hD);
            sys_res[s] = res;
            atomicMax(&a.flags[F_ITERS], st.iters);
            const double r = res < 0.0 ? 0.0 : res;   // a NaN stays NaN (its bits order above every number)
            atomicMax(reinterpret_cast<unsigned long long*>(a.out), (unsigned long long)__double_as_longlong(r));
        }
        __syncthreads();   // bounds and sh are rewritten for the next system
    }
}

// Queue order of the systems: descending constraint count (ties by index).
__global__ void k_sys_order(int ns, const long long* __restrict__ sysoff, const int* __restrict__ rowP,
                            int* __restrict__ order)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const int ms = rowP[sysoff[s + 1]] - rowP[sysoff[s]];
    int pos = 0;
    for (int t = 0; t < ns; ++t) {
        const int mt = rowP[sysoff[t + 1]] - rowP[sysoff[t]];
        pos += mt > ms || (mt == ms && t < s);
    }
    order[pos] = s;
}

// The queue of the per-system solver: the first K systems of the order are
// paired (listed twice), the others listed once.  A system is paired if it
// is among the max_pairs largest, holds at least 4096 constraints per
// block of one cluster (below that the pair's grid-style barriers cost more
// than the extra blocks save) and more than half of one cluster's mean
// share of the batch's constraints.  One block; also zeroes the pairs'
// barrier counters.
__global__ void k_sys_queue(int ns, const long long* __restrict__ sysoff, const int* __restrict__ rowP,
                            const int* __restrict__ order, int nclusters, int cs, int max_pairs,
                            int* __restrict__ qent, int* __restrict__ qn, unsigned* __restrict__ pair_bar)
{
    __shared__ int npair;
    if (threadIdx.x == 0) {
        const long long total = (long long)rowP[sysoff[ns]] - rowP[sysoff[0]];
        const int cap = max_pairs;
        int k = 0;
        while (k < cap && k < ns) {
            const int sy = order[k];
            const long long m = (long long)rowP[sysoff[sy + 1]] - rowP[sysoff[sy]];
            if (m < 4096LL * cs || 2LL * nclusters * m <= total) break;
            ++k;
        }
        npair = k;
        *qn = ns + k;
    }
    __syncthreads();
    const int K = npair;
    for (int t = threadIdx.x; t < kMaxPairs; t += blockDim.x) pair_bar[t] = 0u;
    for (int e = threadIdx.x; e < ns + K; e += blockDim.x) {
        const bool paired = e < 2 * K;   // entry e = 2 * pair + member
        qent[2 * e] = paired ? order[e >> 1] : order[e - K];
        qent[2 * e + 1] = paired ? e : -1;
    }
}

// gamma back in the caller's pair order.
template <typename T>
__global__ void k_gamma_out(int m, const int* __restrict__ flags, const int* __restrict__ perm, const T* gg0,
                            const T* gg1, const double* __restrict__ scale64, double* __restrict__ out,
                            const unsigned long long* __restrict__ mdev)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= count_of(m, mdev)) return;
    if (flags[F_SOLVE_ERR] != 0) return;
    const T* g = flags[F_FINAL] == 0 ? gg0 : gg1;
    // sigma_c (gamma_ref + gamma_lo + delta): the scaled iterate mapped back
    out[perm[c]] = scale64[c] * (((double)g[4 * (size_t)c + 2] + (double)g[4 * (size_t)c + 3]) + (double)g[4 * (size_t)c]);
}

// Largest value f of type T with hD * (double)f <= tol in float64 (the
// float64 product is monotone in f, so max |pi| <= f exactly when the float64
// residual test passes); -1 when no f >= 0 passes.
template <typename T>
static T pi_threshold(double hD, double tol)
{
    if (!(hD * 0.0 <= tol)) return T(-1);
    T f = (T)(tol / hD);
    if (!(f >= T(0))) f = T(0);
    while (f > T(0) && !(hD * (double)f <= tol)) f = std::nextafter(f, T(0));
    for (;;) {
        const T g = std::nextafter(f, std::numeric_limits<T>::infinity());
        if (!(g < std::numeric_limits<T>::infinity()) || !(hD * (double)g <= tol)) break;
        f = g;
    }
    return f;
}

template <typename T>
static SolveArgs<T> make_args(aLENS_ctx* ctx, const SolveBufs<T>& sb, int n, int m)
{
    SolveArgs<T> a;
    a.n = n; a.m = m; a.np = (int)ctx->max_rods; a.mp = (int)ctx->max_pairs;
    a.rowP = ctx->rowP; a.rowQ = ctx->rowQ; a.qlist = ctx->qlist; a.ci = ctx->ci; a.cj = ctx->cj;
    a.rec = sb.rec; a.qe = sb.qe; a.q = sb.q; a.ax = sb.ax;
    a.gg0 = sb.gg[0]; a.gg1 = sb.gg[1]; a.U = sb.U; a.Uref = sb.Uref; a.gref = sb.gref;
    // float32 iterations work on increments over a reference that takes
    // the iterate every kRefresh iterations (and to confirm convergence);
    // float64 needs no refresh
    a.refresh = sizeof(T) == 4 ? kRefresh : 0;
    a.xch = ctx->xch;
    a.priv = sb.priv;
    a.hrank = sb.hrank;
    a.dyn_bytes = 0;
    a.workers = ctx->solve_threads;
    a.partials = ctx->partials; a.bar = ctx->bar; a.flags = ctx->dflags;
    a.out = reinterpret_cast<double*>(ctx->dcount + C_RESID);
    a.inv_perp = (T)ctx->mob.inv_perp; a.inv_par = (T)ctx->mob.inv_par;
    a.inv_rot = (T)ctx->mob.inv_rot; a.inv_spin = (T)ctx->mob.inv_spin;
    a.mobr = ctx->cur_systab ? sb.mobr : nullptr;
    a.rec_lo = sb.rec_lo; a.qe_lo = sb.qe_lo; a.q_lo = sb.q_lo;
    a.lop = sb.lop; a.loq = sb.loq;
    a.pe = sb.pe;
    a.isc = sb.isc;
    a.comp = ctx->cur_comp ? sb.comp : nullptr;
    a.hD = ctx->p.dt / ctx->p.diameter; a.tol = ctx->p.tol; a.max_iter = ctx->p.max_iter;
    a.pi_tol = pi_threshold<T>(a.hD, a.tol);
    a.wait_cycles = (long long)(ctx->wait_s * ctx->clock_khz * 1e3);
    a.fault = 0;
    a.need1_dev = nullptr;
    a.fit_cap = 0;
    a.sort_ns = 0;
    a.sort_cap = 0;
    a.zero_start = ctx->zero_start;
    a.bstart = ctx->bstart;
    return a;
}

// The global-memory solver on data beyond L2 (its records, about 100 bytes
// per constraint, and two 16-byte states stream through L2 every
// iteration): the states, which both phases read and the rod phase gathers
// through the Q-side lists, are kept in L2 by an access-policy window over
// the two state buffers (the first whole, the second up to the last
// constraint) marked persisting, with the context's persisting set-aside
// raised to hold them (as far as the device allows).  Addresses only: the
// kernel and its arithmetic are unchanged.  At 4e5 rods this takes 7 % off
// the solve.  Not while the stream is being captured (the set-aside is not
// a stream operation).
template <typename T>
static bool state_window(aLENS_ctx* ctx, const T* gg0, const T* gg1, int m, cudaAccessPolicyWindow& w)
{
    if (ctx->l2_window_off || ctx->l2_window_max <= 0 || ctx->l2_persist_max <= 0 ||
        (long long)m * 136 <= (long long)ctx->l2_bytes)
        return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(ctx->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    const size_t used = 2 * (size_t)m * 4 * sizeof(T);
    const size_t want = used < (size_t)ctx->l2_persist_max ? used : (size_t)ctx->l2_persist_max;
    size_t cur = 0;
    if (cudaDeviceGetLimit(&cur, cudaLimitPersistingL2CacheSize) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (cur < want) {
        if (cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (!ctx->persist_set) ctx->persist_prev = cur;
        ctx->persist_set = want;
    }
    cudaCtxResetPersistingL2Cache();   // the last solve's persisting lines back to normal
    const char* base = reinterpret_cast<const char*>(gg0);
    size_t bytes = (size_t)(reinterpret_cast<const char*>(gg1 + 4 * (size_t)m) - base);
    if (bytes > (size_t)ctx->l2_window_max) bytes = (size_t)ctx->l2_window_max;
    w.base_ptr = const_cast<char*>(base);
    w.num_bytes = bytes;
    w.hitRatio = 1.0f;
    w.hitProp = cudaAccessPropertyPersisting;
    w.missProp = cudaAccessPropertyStreaming;
    return true;
}

// Threads of a one-barrier block of `workers` threads: a warp more for the
// block sums and the step decision, where the block has room for it (at 1024
// threads, or with several blocks on an SM, the last warp does both).
static int threads1(const aLENS_ctx* ctx)
{
    return ctx->solve_threads <= 992 && ctx->solve_bps <= 1 ? ctx->solve_threads + 32 : ctx->solve_threads;
}

static_assert(sizeof(Shared1<double>) <= sizeof(Shared<double>) + 768 && sizeof(Shared1<float>) <= sizeof(Shared<float>) + 768,
              "the one-barrier kernel's static shared memory and the shares' budget exceed a block's limit");
// Dynamic shared memory that a block may ask for where `blocks` of them share an
// SM that divides its 256 KB into kb KB of shared memory and the rest of L1
// (1 KB a block is the system's, and one is left free).
template <typename T>
static long long dyn_within(int kb, int blocks)
{
    return (long long)(kb / blocks) * 1024 - (long long)sizeof(Shared1<T>) - 2048;
}

// The one-barrier kernel of a launch whose largest share needs `need` bytes.
// With the barrier:
//  - above kMeetRods rods in caller order, or with 1024 workers (no room for a
//    warp of the sums' own: 1e5 rods 10.8 us an iteration against 13.3);
//  - where the other one has 64 registers a thread (every shape but up to 768
//    workers one block an SM) and the share leaves too little L1 for what it
//    spills: 576 bytes a thread in float64, 204 in float32 (solve, ms, barrier /
//    tagged: 4.5e4 rods float64 at 992 x 1 7.90 / 8.81, 4e4 at 512 x 2 6.63 /
//    8.77, 2e4 at 256 x 3 5.96 / 7.31; mixed 5e4 rods at 256 x 4 1.84 / 5.91,
//    1e4 dense ones 5.2 / 7.3);
//  - several blocks an SM, above 10,000 rods in float32: as every block reads
//    every block's sums, and the halo grows with the blocks (1.0e4 rods at 512 x
//    2 and 256 x 4 0.91 / 0.91 and 0.88 / 0.87, 1.2e4 1.18 / 1.18 and 1.02 /
//    1.04, 3e4 1.44 / 1.47 and 1.93 / 2.45).
// Without it elsewhere, in the default shape with 72 registers a thread.
enum { V_MEET = 0, V_WIDE = 1, V_ANY = 2 };
constexpr int kMeetRodsSeveral = 10000;
template <typename T>
static int variant1(const aLENS_ctx* ctx, int n, long long need)
{
    const bool several = ctx->solve_bps > 1;
    if ((ctx->caller_order || (ctx->solve_threads > 992 && !several)) && n > kMeetRods) return V_MEET;
    if (threads1(ctx) <= kThreads1 && !several) return V_WIDE;
    const bool f32 = sizeof(T) == 4;
    if (need > dyn_within<T>(f32 ? 196 : 164, several ? ctx->solve_bps : 1) || (f32 && several && n > kMeetRodsSeveral)) return V_MEET;
    return V_ANY;
}
template <typename T>
static const void* kernel1(int variant)
{
    return variant == V_MEET   ? (const void*)meet::k_bbpgd1_meet<T>
           : variant == V_WIDE ? (const void*)k_bbpgd1<T, kThreads1>
                               : (const void*)k_bbpgd1<T, 1024>;
}
// Its threads, and whether bps blocks of it fit an SM with `budget` bytes of
// dynamic shared memory each (occupancy only falls as shared memory grows: one
// answer per shape; the limit on dynamic shared memory is set once per kernel).
template <typename T>
static cudaError_t ready1(aLENS_ctx* ctx, int variant, size_t budget, int& threads, bool& fits)
{
    const int ti = sizeof(T) == 4 ? 0 : 1, bps = ctx->solve_bps > 0 ? ctx->solve_bps : 1;
    const void* fn = kernel1<T>(variant);
    threads = variant == V_MEET ? ctx->solve_threads : threads1(ctx);
    cudaError_t e;
    if (!(ctx->attr1_set[ti] & 1 << variant)) {
        const long long most = (long long)ctx->smem_optin - (long long)sizeof(Shared1<T>) - 256;
        if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most)) != cudaSuccess) return e;
        ctx->attr1_set[ti] |= 1 << variant;
    }
    const int key = (variant * 2048 + ctx->solve_threads) * 64 + bps;
    if (ctx->occ1_key[ti] != key) {
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, budget)) != cudaSuccess) return e;
        ctx->occ1_ok[ti] = per_sm >= bps;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctx->occ1_regs[ti], fn, threads, 0)) != cudaSuccess) return e;
        ctx->occ1_key[ti] = key;
    }
    fits = ctx->occ1_ok[ti] != 0;
    return cudaSuccess;
}

// Dynamic shared memory of a one-barrier launch whose largest share needs
// `need` bytes: the share proper, with room for ds and gs (2 values for 13)
// and for a halo rod (6 values) per slot, but no more than leaves the L1 that
// the share itself leaves, up to 92 KB of it: the kernel's spilled registers
// live there, and where the largest division leaves 28 KB they go to L2 (the
// steps of the division are the device's).  Solve, ms, with the whole room
// and so: 3e4 rods float64 7.86 / 5.21, 1.6e4 rods float64 in caller order
// 8.16 / 4.85, 2e4 rods float64 at 512 x 2 6.23 / 4.97, 6e4 rods mixed 2.18 /
// 1.88; a halo that finds no room then is polled slot by slot.
// The driver divides an SM for as many blocks as their registers allow
// (by_regs), so a launch of fewer asks for little enough that all those fit
// the division, or for too much for one more than bps (2e4 rods float64 at 256
// x 3 7.28 / 5.62).  Naming the division at the launch instead does not do: it
// can hold fewer blocks than the cooperative grid needs on the SM.
template <typename T>
static long long request1(const aLENS_ctx* ctx, int by_regs, long long need, long long budget)
{
    const int bps = ctx->solve_bps > 0 ? ctx->solve_bps : 1;
    const long long room = need + need * 8 / 13;
    for (int kb : {164, 196}) {
        const long long all = dyn_within<T>(kb, by_regs), most = dyn_within<T>(kb, bps);
        if (need <= all) return room < all ? room : all;
        const long long least = std::max(need, 228ll * 1024 / (bps + 1));
        if (by_regs > bps && least <= most) return std::min(std::max(room, least), most);
    }
    return room < budget ? room : budget;
}

template <typename T>
static cudaError_t solve_typed(aLENS_ctx* ctx, const SolveBufs<T>& sb, int n, int m)
{
    SolveArgs<T> a = make_args(ctx, sb, n, m);
    a.fault = ctx->fault_mode;
    ctx->fault_mode = 0;

    const int threads = ctx->solve_threads;
    const int bps = ctx->solve_bps > 0 ? ctx->solve_bps : 1;
    // enough blocks that each has at least a warp of rods
    long long want = ((long long)n + 31) / 32;
    long long blocks = (long long)bps * ctx->num_sms;
    if (want < blocks) blocks = want < 1 ? 1 : want;
    if (blocks > ctx->max_blocks) blocks = ctx->max_blocks;
    // work-balanced split, then the largest shared-memory share: stage every
    // block's data when all shares fit the opt-in budget (one readback)
    cudaError_t e;
    k_shares<<<(int)blocks, kNeedThreads, 0, ctx->stream>>>(n, (int)blocks, (int)sizeof(T), ctx->rowP, ctx->rowQ, ctx->qlist,
                                                             ctx->bstart, ctx->bar, ctx->dcount + C_SMEM,
                                                             ctx->dcount + C_MAXRODS, ctx->dcount + C_SMEM1);
    ++ctx->launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // one readback of the counters C_SMEM .. C_SMEM1 (into the pinned host status
    // buffer; the allocation-free entry point has none and reads into the stack)
    unsigned long long local[C_SMEM1 - C_SMEM + 1];
    unsigned long long* hb = ctx->hcount ? ctx->hcount + C_SMEM : local;
    if ((e = cudaMemcpyAsync(hb, ctx->dcount + C_SMEM, (C_SMEM1 - C_SMEM + 1) * sizeof(unsigned long long),
                             cudaMemcpyDeviceToHost, ctx->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(ctx->stream)) != cudaSuccess)
        return e;
    const unsigned long long need = hb[0], maxrods = hb[C_MAXRODS - C_SMEM], need1 = hb[C_SMEM1 - C_SMEM];
    ctx->last_need1 = need1;
    const int optin = ctx->smem_optin;
    const long long budget = (long long)optin / bps - (long long)sizeof(Shared<T>) - 1024;
    if (ctx->solve_barriers == 1 && threads >= 256 && need1 > 0 && (long long)need1 <= budget) {
        // at most one grid barrier per iteration: every block's share and its ghosts fit
        const int variant = variant1<T>(ctx, n, (long long)need1);
        int threads = 0;
        bool fits = false;
        if ((e = ready1<T>(ctx, variant, (size_t)budget, threads, fits)) != cudaSuccess) return e;
        if (fits && (long long)bps * ctx->num_sms >= blocks) {
            a.dyn_bytes = (size_t)(variant == V_MEET ? (long long)need1 : request1<T>(ctx, ctx->occ1_regs[sizeof(T) == 4 ? 0 : 1], (long long)need1, budget));
            void* args1[] = {&a};
            ++ctx->launches;
            ctx->last_solver = 1;
            return cudaLaunchCooperativeKernel(kernel1<T>(variant), dim3((unsigned)blocks), dim3(threads), args1, a.dyn_bytes,
                                               ctx->stream);
        }
    }
    if ((e = launch_setup_qe(ctx)) != cudaSuccess) return e;   // the two-barrier kernels read qe
    const bool staged = (long long)need <= budget && (long long)n / blocks < 60000;
    // global-memory blocks still take their rods in count order when the
    // order (10 bytes of scratch per rod) fits
    const long long sort_bytes = 10 * (long long)maxrods;
    a.sort_ns = sizeof(T) == 8 && !staged && maxrods > 0 && maxrods < 65536 && sort_bytes <= budget;
    a.sort_cap = (int)maxrods;
    const size_t smem = staged ? (size_t)need : (a.sort_ns ? (size_t)sort_bytes : 0);
    constexpr int kMaxT = sizeof(T) == 8 ? 768 : 1024;
    // (several blocks on an SM share its registers: 64 a thread there as well)
    const void* fn = threads <= kMaxT && bps <= 1 ? (staged ? (const void*)k_bbpgd<T, true, kMaxT> : (const void*)k_bbpgd<T, false, kMaxT>)
                                                  : (staged ? (const void*)k_bbpgd<T, true, 1024> : (const void*)k_bbpgd<T, false, 1024>);
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem)) != cudaSuccess) return e;
    if ((long long)per_sm * ctx->num_sms < blocks) return cudaErrorCooperativeLaunchTooLarge;
    void* args[] = {&a};
    ++ctx->launches;
    ctx->last_solver = staged ? 2 : 3;
    cudaAccessPolicyWindow win;
    if (!staged && sizeof(T) == 4 && state_window(ctx, sb.gg[0], sb.gg[1], m, win)) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        at[1].id = cudaLaunchAttributeAccessPolicyWindow;
        at[1].val.accessPolicyWindow = win;
        cfg.gridDim = dim3((unsigned)blocks);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = ctx->stream;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        return cudaLaunchKernelExC(&cfg, fn, args);
    }
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)blocks), dim3(threads), args, smem, ctx->stream);
}

// Batches: the per-system solver on thread-block clusters (one launch).
template <typename T>
static cudaError_t solve_batch_typed(aLENS_ctx* ctx, const SolveBufs<T>& sb, int n, int m)
{
    SolveArgs<T> a = make_args(ctx, sb, n, m);
    a.fault = ctx->fault_mode == 1 ? 1 : 0;
    ctx->fault_mode = 0;
    const int ns = ctx->batch_n;
    cudaError_t e;
    if ((e = launch_setup_qe(ctx)) != cudaSuccess) return e;   // the per-system solver reads qe
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ctx->batch_cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // rod order scratch: 10 bytes per rod for twice a cluster block's even
    // share of the largest system (a block with a larger share keeps the
    // rank order); kept small, since this solver reads its data through L1
    long long max_sys = 0;
    for (int s = 0; s < ns; ++s) {
        const long long r = ctx->batch_off_host[s + 1] - ctx->batch_off_host[s];
        if (r > max_sys) max_sys = r;
    }
    const long long cap = 2 * ((max_sys + ctx->batch_cluster - 1) / ctx->batch_cluster);
    a.sort_cap = (int)(cap < 65535 ? cap : 65535);
    const long long sort_bytes = 10 * (long long)a.sort_cap;
    a.sort_ns = sizeof(T) == 8 && cap > 0 && sort_bytes <= 64 * 1024;
    const size_t smem = a.sort_ns ? (size_t)sort_bytes : 0;
    // the attribute is the largest dynamic shared memory a launch may ask
    // for: raised when a batch needs more, never lowered, so that no call is
    // made when nothing changes (a batched step may be recorded as a graph)
    static size_t smem_set[64];
    const int dv = ctx->device >= 0 && ctx->device < 64 ? ctx->device : 0;
    if (smem > smem_set[dv]) {
        if ((e = cudaFuncSetAttribute(k_bbpgd_sys<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
            cudaSuccess)
            return e;
        smem_set[dv] = smem;
    }
    cfg.blockDim = dim3((unsigned)ctx->batch_threads);
    cfg.gridDim = dim3((unsigned)ctx->batch_cluster);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int max_active = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&max_active, k_bbpgd_sys<T>, &cfg)) != cudaSuccess) return e;
    if (max_active < 1) return cudaErrorInvalidConfiguration;
    int* qent = ctx->sys_order + ns;
    int* qn = qent + 2 * ((size_t)ns + kMaxPairs);
    unsigned* pair_bar = reinterpret_cast<unsigned*>(qn + 1);
    k_sys_order<<<(ns + 127) / 128, 128, 0, ctx->stream>>>(ns, ctx->sysoff, ctx->rowP, ctx->sys_order);
    ++ctx->launches;
    // Pairs wait for each other, so they need every cluster resident at
    // once: a cooperative launch (tried by the first batched solve of the
    // context; without it the solver runs without pairs).
    cudaLaunchAttribute attr2[2] = {attr[0], {}};
    attr2[1].id = cudaLaunchAttributeCooperative;
    attr2[1].val.cooperative = 1;
    for (int pass = 0; pass < 2; ++pass) {
        const int cap = max_active / 4 < kMaxPairs ? max_active / 4 : kMaxPairs;
        const int max_pairs = ctx->batch_coop != 0 ? cap : 0;
        // a cluster per queue entry at most (every system, and the pairs' second entries)
        const int nclusters = max_active < ns + max_pairs ? max_active : ns + max_pairs;
        k_sys_queue<<<1, 256, 0, ctx->stream>>>(ns, ctx->sysoff, ctx->rowP, ctx->sys_order, nclusters,
                                                ctx->batch_cluster, max_pairs, qent, qn, pair_bar);
        ++ctx->launches;
        if ((e = cudaMemsetAsync(ctx->dcount + C_QUEUE, 0, sizeof(unsigned long long), ctx->stream)) != cudaSuccess)
            return e;
        cfg.gridDim = dim3((unsigned)(nclusters * ctx->batch_cluster));
        cfg.attrs = max_pairs > 0 ? attr2 : attr;
        cfg.numAttrs = max_pairs > 0 ? 2 : 1;
        e = cudaLaunchKernelEx(&cfg, k_bbpgd_sys<T>, a, (const long long*)ctx->sysoff, (const int*)qent,
                               (const int*)qn, pair_bar, ctx->dcount + C_QUEUE, ctx->sys_iters,
                               ctx->sys_iters + ctx->max_systems, ctx->sys_res);
        if (e == cudaSuccess) {
            if (max_pairs > 0) ctx->batch_coop = 1;
            break;
        }
        // a refused cooperative cluster launch enqueued nothing: queue again without pairs
        if (max_pairs == 0 || ctx->batch_coop == 1) return e;
        cudaGetLastError();
        ctx->batch_coop = 0;
    }
    if (e != cudaSuccess) return e;
    ++ctx->launches;
    ctx->last_solver = 4;
    return cudaSuccess;
}

cudaError_t launch_solve(aLENS_ctx* ctx, int n, int m, int precision)
{
    const bool per_system = ctx->cur_systab != nullptr && ctx->batch_n > 1;
    if (precision == ALENS_MIXED)
        return per_system ? solve_batch_typed<float>(ctx, ctx->sb32, n, m) : solve_typed<float>(ctx, ctx->sb32, n, m);
    return per_system ? solve_batch_typed<double>(ctx, ctx->sb64, n, m) : solve_typed<double>(ctx, ctx->sb64, n, m);
}

// The single-system solve of a step recorded as a CUDA graph: no readback.
// The kernel and its shared memory are chosen for the largest share of the
// eager step of the same key (graph_need), and its blocks check the need of
// the shares (computed on the device by k_shares) against it: a share that
// does not fit makes every block leave before its first barrier with
// kSolveRedo in F_SOLVE_ERR, the update and the outputs then leave everything
// untouched, and the caller runs the step eagerly.  (With all the shared
// memory a block may ask for, little L1 is left for the kernel's spills:
// 2e4 rods float64 4.13 ms against 2.98, 1e4 rods mixed at 256 x 4 1.65
// against 0.87.)
template <typename T>
static cudaError_t plan_graph1(aLENS_ctx* ctx, int n, SolveArgs<T>* a, int& variant, int& threads, bool& ok)
{
    ok = false;
    if (ctx->solve_barriers != 1 || ctx->solve_threads < 256) return cudaSuccess;
    const int bps = ctx->solve_bps > 0 ? ctx->solve_bps : 1;
    const long long budget = (long long)ctx->smem_optin / bps - (long long)sizeof(Shared<T>) - 1024;
    const long long need = (long long)ctx->graph_need;
    variant = variant1<T>(ctx, n, need);
    const cudaError_t e = ready1<T>(ctx, variant, (size_t)budget, threads, ok);
    if (a && e == cudaSuccess) {
        a->dyn_bytes = (size_t)request1<T>(ctx, ctx->occ1_regs[sizeof(T) == 4 ? 0 : 1], need, budget);
        a->fit_cap = (long long)a->dyn_bytes;
        ctx->graph_full = (long long)a->dyn_bytes >= budget;
    }
    return e;
}

template <typename T>
static cudaError_t graph1_check(aLENS_ctx* ctx, int n, bool& ok)
{
    int variant = 0, threads = 0;
    ctx->caller_order = 0;   // (a step's: the layout sets it, which is not yet recorded)
    return plan_graph1<T>(ctx, n, nullptr, variant, threads, ok);
}

template <typename T>
static cudaError_t solve_graph1_typed(aLENS_ctx* ctx, const SolveBufs<T>& sb, int n, int m)
{
    SolveArgs<T> a = make_args(ctx, sb, n, m);
    const bool force_redo = ctx->fault_mode == 2;   // test hook: the recorded need never fits
    ctx->fault_mode = 0;
    const int bps = ctx->solve_bps > 0 ? ctx->solve_bps : 1;
    long long want = ((long long)n + 31) / 32;
    long long blocks = (long long)bps * ctx->num_sms;
    if (want < blocks) blocks = want < 1 ? 1 : want;
    if (blocks > ctx->max_blocks) blocks = ctx->max_blocks;
    int variant = 0, threads = 0;
    bool fits = false;
    cudaError_t e = plan_graph1<T>(ctx, n, &a, variant, threads, fits);
    if (e != cudaSuccess) return e;
    if (!fits) return cudaErrorCooperativeLaunchTooLarge;
    a.need1_dev = ctx->dcount + C_SMEM1;
    if (force_redo) {
        a.fit_cap = 0;
        ctx->graph_full = 1;
    }
    k_shares<<<(int)blocks, kNeedThreads, 0, ctx->stream>>>(n, (int)blocks, (int)sizeof(T), ctx->rowP, ctx->rowQ, ctx->qlist,
                                                             ctx->bstart, ctx->bar, ctx->dcount + C_SMEM,
                                                             ctx->dcount + C_MAXRODS, ctx->dcount + C_SMEM1);
    ++ctx->launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    void* args1[] = {&a};
    ++ctx->launches;
    ctx->last_solver = 1;
    return cudaLaunchCooperativeKernel(kernel1<T>(variant), dim3((unsigned)blocks), dim3(threads), args1, a.dyn_bytes,
                                       ctx->stream);
}

// Whether the launch that would be recorded fits the device at all.
cudaError_t graph1_possible(aLENS_ctx* ctx, int n, int precision, bool& ok)
{
    return precision == ALENS_MIXED ? graph1_check<float>(ctx, n, ok) : graph1_check<double>(ctx, n, ok);
}

cudaError_t launch_solve_graph1(aLENS_ctx* ctx, int n, int m, int precision)
{
    return precision == ALENS_MIXED ? solve_graph1_typed<float>(ctx, ctx->sb32, n, m)
                                    : solve_graph1_typed<double>(ctx, ctx->sb64, n, m);
}

cudaError_t launch_gamma_out(aLENS_ctx* ctx, int m, int precision, double* gamma_out)
{
    if (m <= 0 || !gamma_out) return cudaSuccess;
    int b = (m + 255) / 256;
    if (precision == ALENS_MIXED) {
        k_gamma_out<float><<<b, 256, 0, ctx->stream>>>(m, ctx->dflags, ctx->perm, ctx->sb32.gg[0], ctx->sb32.gg[1],
                                                       ctx->scale64, gamma_out, ctx->mdev);
    } else {
        k_gamma_out<double><<<b, 256, 0, ctx->stream>>>(m, ctx->dflags, ctx->perm, ctx->sb64.gg[0], ctx->sb64.gg[1],
                                                        ctx->scale64, gamma_out, ctx->mdev);
    }
    ++ctx->launches;
    return cudaGetLastError();
}

}  // namespace alens
