// mm_kernels.cu -- FP64 kernels of the multi-morphology stepper (sm_103a).
//
// One time step n -> n+1 is two launches:
//   deliver_kernel: spikes detected round(delay/dt) + 1 steps ago raise the
//                   synaptic conductance of their target sites (the local /
//                   global spike buffers of Sec. 2 become a device ring of
//                   per-step spike lists, expanded through an outgoing CSR);
//   step_fp64:      per work item (a run of whole neurons): HH currents,
//                   assembly of the Hines system for dV (Eq. 2), the Hines
//                   solve (Algorithm 1) path by path in shared memory,
//                   V += dV, exponential-Euler gates, synaptic decay and the
//                   soma threshold test.
// The model is the oracle's (units um, mV, ms, nA, uS, nF); the arithmetic
// here is written independently of it.
#include <cuda_runtime.h>

#include <mutex>

#include "mm_fp64_math.h"
#include "mm_gate_table64.h"
#include "mm_internal.h"
#include "mm_tma.h"

using namespace mmk;

namespace {

constexpr double kPi = 3.141592653589793;

// x / (e^x - 1) and its limit near 0.
__device__ __forceinline__ double xexpm1_ratio(double x)
{
    return fabs(x) < 1e-6 ? 1.0 - 0.5 * x : x / expm1(x);
}

// HH rate constants (1/ms) at v (mV), rest -65 mV.
struct Rates {
    double am, bm, ah, bh, an, bn;
};

__device__ __forceinline__ Rates hh_rates(double v)
{
    Rates r;
    r.am = xexpm1_ratio(-(v + 40.0) * 0.1);
    r.bm = 4.0 * exp(-(v + 65.0) * (1.0 / 18.0));
    r.ah = 0.07 * exp(-(v + 65.0) * 0.05);
    r.bh = 1.0 / (1.0 + exp(-(v + 35.0) * 0.1));
    r.an = 0.1 * xexpm1_ratio(-(v + 55.0) * 0.1);
    r.bn = 0.125 * exp(-(v + 65.0) * 0.0125);
    return r;
}

// Exact relaxation of one gate over dt with frozen rates.
__device__ __forceinline__ double relax(double x, double a, double b, double dt)
{
    double s = a + b;
    double xinf = a / s;
    return xinf + (x - xinf) * exp(-dt * s);
}

__device__ __forceinline__ double half_cyl_resistance(double Ra, double L_um, double d_um)
{
    // MOhm: Ra * (L/2) / (pi d^2 / 4), lengths converted um -> cm
    double rad = 0.5e-4 * d_um;
    return Ra * (0.5e-4 * L_um) / (kPi * rad * rad) * 1e-6;
}

// ------------------------------------------------------------------ init

// Areas, axial conductances (negated at path heads) and the resting state.
__global__ void init_kernel(InitArgs a)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.C;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double L = a.L[i], d = a.diam[i];
        a.area[i] = kPi * d * L * 1e-8;
        const int32_t pd = a.parent_dist[i];
        double g = 0.0;
        if (pd != 0) {
            const int64_t q = i - abs(pd);
            g = 1.0 / (half_cyl_resistance(a.Ra, L, d) + half_cyl_resistance(a.Ra, a.L[q], a.diam[q]));
        }
        a.gax[i] = pd > 0 ? g : -g;
        double v = a.v_init;
        Rates r = hh_rates(v);
        a.V[i] = v;
        a.m[i] = r.am / (r.am + r.bm);
        a.h[i] = r.ah / (r.ah + r.bh);
        a.n[i] = r.an / (r.an + r.bn);
    }
}

// The scaling of each work item's Hines system (see step_fp64_kernel), a block
// per item: down each path s = 1 at its head and then the mantissa of
// 1 / (w g s_parent) (w the implicit share of a coupling), so that the coupling
// w g s s_parent inside a path is a power of two, whose exponent field is
// stored; at a head the coupling to the parent compartment, negative.  A coupling
// below 2^-500 uS, or none (infinite Ra), is taken as 2^-500, which adds nothing
// to any diagonal and whose square keeps exponent fields within 32 bits.  Then the
// constant part of the diagonal: C/dt, the implicit leak and the couplings,
// times s^2 -- as the matrix holds them, s 2^k / s_parent inside a path, the
// rounded coupling times or over s_parent at a head.  It is the same at every
// step, so what its rounding leaves out is kept in FP32: it would add up over the
// steps, as a part of the couplings (18 neurons of 20 to 4,000 compartments with
// couplings up to 1e4 C/dt, 80 steps: 6.4e-14 mV in the mean square without it,
// 7.5e-15 with it; 1.5 % of the step's time).
__global__ void __launch_bounds__(128) scale_kernel(ScaleArgs64 a)
{
    const GroupRec G = a.groups[blockIdx.x];
    const unsigned char *blob = a.meta + G.meta_off;
    const PathQ *paths = (const PathQ *)(blob + G.path_off);
    const KidQ *fold = (const KidQ *)(blob + G.fold_off);
    const double *area = a.area + G.comp0, *gax = a.gax + G.comp0;
    double *sc = a.sc + G.comp0, *s2a = a.s2a + G.comp0, *dcon = a.dcon + G.comp0;
    int32_t *kexp = a.kexp + G.comp0;
    float *drest = a.drest + G.comp0;
    auto scale_of = [&](int i) { return signbit(sc[i]) ? 1.0 : sc[i]; };
    // a value and the rest of it; x y, x / y, and the sum
    struct Two {
        double v, r;
    };
    auto times = [](double x, double y) { const double p = x * y; return Two{p, fma(x, y, -p)}; };
    auto over = [](double x, double y) { const double q = x / y; return Two{q, fma(-q, y, x) / y}; };
    auto plus = [](const Two &x, const Two &y) {
        const double t = x.v + y.v, u = t - x.v;
        return Two{t, ((x.v - (t - u)) + (y.v - u)) + (x.r + y.r)};
    };
    auto scaled = [](const Two &x, int k) { return Two{scale2(x.v, k), scale2(x.r, k)}; };
    auto store = [&](int j, const Two &d) {
        const double v = d.v + d.r;
        dcon[j] = v;
        drest[j] = (float)((d.v - v) + d.r);
    };
    for (int pi = threadIdx.x; pi < G.npath; pi += 128) {
        const PathQ P = paths[pi];
        const int h = P.head;
        double s = 1.0;
        Two own{0.0, 0.0};  // s^2 w g of the link to the parent (a head's is added below)
        for (int j = h; j < P.end; ++j) {
            double sn = 1.0;
            Two link{0.0, 0.0}, next_own{0.0, 0.0};
            if (j + 1 < P.end) {
                const double c = a.gimp * gax[j + 1] * s;
                if (c < 0x1p-500) {
                    kexp[j + 1] = -(500 << 20);
                } else {
                    const double p = 1.0 / c;
                    sn = mantissa(p);
                    const int k = -exponent2(p);
                    kexp[j + 1] = k;
                    link = scaled(over(s, sn), k);
                    next_own = scaled(over(sn, s), k);
                }
            }
            const Two ss = times(s, s);
            Two s2 = times(ss.v, area[j]);
            s2.r = fma(ss.r, area[j], s2.r);
            Two cm = times(s2.v, a.cm_leak);
            cm.r = fma(s2.r, a.cm_leak, cm.r);
            sc[j] = j == h ? -0.0 : s;
            if (j == h) kexp[j] = 0;
            s2a[j] = s2.v;
            store(j, plus(cm, plus(own, link)));
            s = sn;
            own = next_own;
        }
    }
    __syncthreads();
    for (int pi = threadIdx.x; pi < G.npath; pi += 128) {
        const PathQ P = paths[pi];
        if (P.parent < 0) continue;
        const double sp = scale_of(P.parent), g = a.gimp * fabs(gax[P.head]) * sp;
        sc[P.head] = -g;
        store(P.head, plus(Two{dcon[P.head], drest[P.head]}, over(g, sp)));
    }
    __syncthreads();
    for (int e = threadIdx.x; e < G.npath; e += 128) {
        const int att = (int)(fold[e] >> 16);
        if (att >= G.ncomp) continue;  // a path from a soma (no parent)
        if (e > 0 && (int)(fold[e - 1] >> 16) == att) continue;  // not the first path of its parent
        Two d{dcon[att], drest[att]};
        const double s = scale_of(att);
        for (int z = e; z < G.npath && (int)(fold[z] >> 16) == att; ++z)
            d = plus(d, times(-sc[paths[fold[z] & 0xFFFFu].head], s));
        store(att, d);
    }
}

// --------------------------------------------------------------- delivery

constexpr int kMaxDClass = 1024;

__global__ void __launch_bounds__(256) deliver_kernel(DeliverArgs a)
{
    __shared__ int s_pref[kMaxDClass + 1];
    __shared__ int s_slot[kMaxDClass];
    const long long n = (long long)a.ctl->step_base + a.step_offset;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->queue_head = 0u;
        a.ctl->big_head = 0u;
        a.ring_cnt[n % a.R] = 0;
    }
    for (int k = threadIdx.x; k < a.n_dclass; k += blockDim.x) {
        long long src_step = n - 1 - a.dclass[k];
        int cnt = 0, slot = 0;
        if (src_step >= 0) {
            slot = (int)(src_step % a.R);
            cnt = a.ring_cnt[slot];
        }
        s_slot[k] = slot;
        s_pref[k + 1] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        s_pref[0] = 0;
        for (int k = 1; k <= a.n_dclass; ++k) s_pref[k] += s_pref[k - 1];
    }
    __syncthreads();
    const int total = s_pref[a.n_dclass];
    // groups of lanes_per_src lanes take one spike each (see the FP32c kernel)
    const int GL = a.lanes_per_src;
    const int lane = threadIdx.x & (GL - 1);
    const int ngroups = (gridDim.x * blockDim.x) / GL;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) / GL; u < total; u += ngroups) {
        int lo = 0, hi = a.n_dclass;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (s_pref[mid] <= u) lo = mid; else hi = mid;
        }
        const int src = a.ring_nrn[(long long)s_slot[lo] * a.N + (u - s_pref[lo])];
        long long b = a.out_off[src], e = a.out_off[src + 1];
        if (a.n_dclass > 1) {
            const int D = a.dclass[lo];
            long long l = b, r = e;            // first entry with dsteps >= D
            while (l < r) { long long m = (l + r) >> 1; if (a.out_dsteps[m] < D) l = m + 1; else r = m; }
            long long l2 = l, r2 = e;          // first entry with dsteps > D
            while (l2 < r2) { long long m = (l2 + r2) >> 1; if (a.out_dsteps[m] <= D) l2 = m + 1; else r2 = m; }
            b = l; e = l2;
        }
        for (long long q = b + lane; q < e; q += GL) atomicAdd(&a.gsyn[a.out_site[q]], a.out_w[q]);
    }
}

// Deterministic delivery (mm_options.deterministic_delivery): each site adds
// the weights of its synapses whose source fired round(delay/dt) + 1 steps
// ago, in ascending synapse id (the oracle's order), one thread per site;
// also the per-step resets of the work queues, of this step's spike-ring
// count and of this step's slot of the fired bitmasks (last written R steps
// ago, all of whose events are delivered).
__global__ void __launch_bounds__(256) deliver_ordered_kernel(DeliverArgs a)
{
    const long long n = (long long)a.ctl->step_base + a.step_offset;
    const long long gt = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nt = (long long)gridDim.x * blockDim.x;
    if (gt == 0) {
        a.ctl->queue_head = 0u;
        a.ctl->big_head = 0u;
        a.ring_cnt[n % a.R] = 0;
    }
    uint32_t *slot = a.fired + (n % a.R) * a.fired_words;
    for (long long w = gt; w < a.fired_words; w += nt) slot[w] = 0u;
    for (long long st = gt; st < a.nsite; st += nt) {
        const long long e0 = a.in_off[st], e1 = a.in_off[st + 1];
        if (e0 == e1) continue;
        double g = a.gsyn[st];
        bool hit = false;
        for (long long e = e0; e < e1; ++e) {
            const long long m = n - 1 - a.in_dsteps[e];
            if (m < 0) continue;
            const int src = a.in_src[e];
            if ((a.fired[(m % a.R) * a.fired_words + (src >> 5)] >> (src & 31)) & 1u) {
                g += a.in_w[e];
                hit = true;
            }
        }
        if (hit) a.gsyn[st] = g;
    }
}

// ------------------------------------------------------------ FP64 step

// Exponential-Euler gate update at V^{n+1} of one compartment (its V is final
// for this step): from the table, or beyond its range from the rates.
__device__ __forceinline__ void gate_update(const StepArgs &a, int64_t c)
{
    const double v = a.V[c];
    double *const x[3] = {a.m + c, a.h + c, a.n + c};
    if (mmg::in_table(v)) {
        const mmg::Index64 t = mmg::index64(v);
        constexpr int I = mmg::kTab64Intervals;
        const double2 *f = a.gtab + t.i;
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            double XF[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const double2 p = __ldg(f + (6 * g + 3 * k) * I), q = __ldg(f + (6 * g + 3 * k + 1) * I);
                const float4 s = __ldg((const float4 *)(f + (6 * g + 3 * k + 2) * I));
                XF[k] = k == 0 ? mmg::eval64_rest({p.x, p.y}, {q.x, q.y}, {s.x, s.y, s.z, s.w}, t)
                               : mmg::eval64({p.x, p.y}, {q.x, q.y}, {s.x, s.y, s.z, s.w}, t);
            }
            *x[g] = mmg::step64(*x[g], XF[0], XF[1]);
        }
    } else {
        const Rates r = hh_rates(v);
        *x[0] = relax(*x[0], r.am, r.bm, a.dt);
        *x[1] = relax(*x[1], r.ah, r.bh, a.dt);
        *x[2] = relax(*x[2], r.an, r.bn, a.dt);
    }
}

// Gate updates of the compartments pc0 .. pc0 + pn - 1, in chunks of
// kGateChunk claimed by whole warps from the shared counter *next until none
// is left.
constexpr int kGateChunk = 64;

__device__ __forceinline__ void gate_chunks(const StepArgs &a, int64_t pc0, int pn, int *next, int lane)
{
    for (;;) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(next, 1);
        ch = __shfl_sync(0xFFFFFFFFu, ch, 0);
        const int i0 = ch * kGateChunk;
        if (i0 >= pn) break;
        const int i1 = min(i0 + kGateChunk, pn);
        for (int i = i0 + lane; i < i1; i += 32) gate_update(a, pc0 + i);
    }
}

// Compartments per step of a path sweep.
constexpr int kSweepChunk = 4;
// Paths of at least this many compartments are swept by a whole warp.
constexpr int kWarpPath = 96;

template <int NT>
__global__ void __launch_bounds__(NT, NT <= 256 ? 512 / NT : 1) step_fp64_kernel(StepArgs a)
{
    // Bound by the FP64 pipe (two lanes per SM and clock: a warp's FP64
    // instruction takes it for 16 clocks whatever the number of active
    // lanes), so everything here saves FP64 instructions and keeps the
    // rest busy in full warps:
    //   * the gates come from the table (mm_gate_table64.h), with the constant
    //     part of the diagonal stored per compartment;
    //   * the sweeps are the part with few active lanes (one lane per
    //     path), so they hold two instructions a compartment and no division.
    //     The elimination carries d'_j = N_j / M_j and rhs'_j = S_j / M_j,
    //       N_{j-1} = d_{j-1} N_j - gamma_j^2 M_j,  M_{j-1} = N_j,
    //       S_{j-1} = r_{j-1} N_j + gamma_j S_j
    //     (Algorithm 1's row times M) on the system scaled by s on both sides
    //     (scale_kernel; the unknown is y = dV / s) so that gamma is a power of
    //     two inside a path: the products by it, and the powers of two taken
    //     out of N, M and S at each step, are integer additions.  The division
    //     for the substitution's factors f_j = gamma_j M_j / N_j, c_j = S_j / N_j
    //     is a pass of full warps;
    //   * warps without a sweep update the gates of the block's previous item.
    // Work items, teams, bundles, levels and the fold list are the FP32c
    // kernel's (step_fp32c_kernel), with the diagonal and rhs in FP64.
    // Measured per step, items of 4,096 compartments: 2,000 neurons of 50 to
    // 5,000 compartments (2.14 M) 1.81 ms with divisions in the sweeps and the
    // rates evaluated, 0.74 ms with the table and products (five instructions a
    // sweep step), 0.55 ms on the scaled system (two); 64 neurons of 255 370,
    // 159, 121 us; 701 of 50 to 3,000, points and ordered delivery, 808, 262,
    // 185 us.  Three or four blocks per SM (85 or 64 registers) 2 to 10 %.
    //
    // Shared memory: the item's tree blob (one bulk copy), then per
    // compartment the pair (diagonal, rhs) -- after a path's elimination
    // (N, S) for its inside and (-f, c) for its head, whose sign says that the
    // division is done, then (f, c), after substitution (f, y).
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *smeta = smem_raw;
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_item, s_abort;
    __shared__ long long s_pc0;  // pending gate work: the previous item's compartments
    __shared__ int s_pn, s_gchunk;

    const long long n = (long long)a.ctl->step_base + a.step_offset;
    const int tid = threadIdx.x;
    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        s_abort = 0;
        s_pc0 = 0;
        s_pn = 0;
        s_gchunk = 0;
    }
    uint32_t parity = 0;

    for (;;) {
        __syncthreads();
        if (s_abort) break;
        if (tid == 0) {
            const int item = (int)atomicAdd(&a.ctl->queue_head, 1u);
            s_item = item;
            if (item < a.n_groups) {
                const GroupRec *gp = a.groups + item;
                const uint32_t bytes = (uint32_t)gp->meta_bytes;
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(&bar, bytes);
                bulk_copy_g2s(smeta, a.meta + gp->meta_off, bytes, &bar);
            }
        }
        __syncthreads();
        const int gi = s_item;
        if (gi >= a.n_groups) break;
        const GroupRec G = a.groups[gi];
        const int64_t c0 = G.comp0;
        const double *V = a.V + c0;
        const double *gax = a.gax + c0;
        const double *sc = a.sc + c0;
        const int32_t *kexp = a.kexp + c0;
        double2 *sdr = (double2 *)(smem_raw + G.meta_bytes);
        auto scale_of = [&](int i) { const double s = __ldg(sc + i); return signbit(s) ? 1.0 : s; };

        // A. diagonal and rhs at (V^n, gates^n): membrane conductance and
        //    current, and the axial currents of the links inside paths (a
        //    link (i-1, i) is inside a path when gax[i] has no sign bit; its
        //    conductances are in the constant part of the diagonal).
#pragma unroll 2
        for (int i = tid; i < G.ncomp; i += NT) {
            const double v = V[i], mm = a.m[c0 + i], hh = a.h[c0 + i], nn = a.n[c0 + i];
            const double ar = a.area[c0 + i], g = gax[i];
            const double gna = a.gNa * ((mm * mm) * (mm * hh)), n2 = nn * nn, gk = a.gK * (n2 * n2);
            double d = a.dcon[c0 + i];
            if (a.g_implicit) d += fma(a.s2a[c0 + i], gna + gk, mmg::widen(a.drest[c0 + i]));
            double r = -ar * fma(gna, v - a.ENa, fma(gk, v - a.EK, a.gL * (v - a.EL)));
            if (!signbit(g)) r = fma(g, V[i - 1] - v, r);
            if (i + 1 < G.ncomp) {
                const double gc = gax[i + 1];
                if (!signbit(gc)) r = fma(gc, V[i + 1] - v, r);
            }
            const double s = sc[i];
            if (!signbit(s)) r *= s;
            sdr[i] = make_double2(d, r);
        }
        if (!mbar_wait_bounded(&bar, parity)) {
            // give up on this item, but not on the copy in flight: wait for
            // it once more (bounded) so that the block never leaves while
            // the copy could still write into its shared memory
            s_abort = 1;
            mbar_wait_bounded(&bar, parity);
        }
        parity ^= 1u;
        __syncthreads();
        if (s_abort) {  // the whole block leaves at the next item boundary
            if (tid == 0) atomicOr(&a.ctl->err, MMK_ERR_TIMEOUT);
            continue;
        }
        const NrnQ *nrns = (const NrnQ *)smeta;
        const PathQ *paths = (const PathQ *)(smeta + G.path_off);
        const KidQ *fold = (const KidQ *)(smeta + G.fold_off);
        const int16_t *loffs = (const int16_t *)(smeta + G.loffs_off);
        const int16_t *mcnt = (const int16_t *)(smeta + G.mcnt_off);

        // S. synaptic sites (then their decay; sites are distinct
        //    compartments), the current across each path's head link into its
        //    head (for the path from a soma the stimulus), then per parent
        //    compartment the currents of the links to the heads that hang off
        //    it, in fold-list order.
        for (int t = tid; t < G.nsite; t += NT) {
            const int st = G.site0 + t;
            const int c = a.site_comp[st];
            const double g = a.gsyn[st];
            double2 w = sdr[c];
            const double s = scale_of(c), t1 = s * g;
            if (a.g_implicit) w.x = fma(t1, s, w.x);
            w.y = fma(-t1, V[c] - a.e_syn, w.y);
            sdr[c] = w;
            a.gsyn[st] = g * a.decay;
        }
        __syncthreads();
        for (int pi = tid; pi < G.npath; pi += NT) {
            const PathQ P = paths[pi];
            double r = sdr[P.head].y;
            if (P.parent >= 0) r = fma(fabs(gax[P.head]), V[P.parent] - V[P.head], r);
            else r += a.stim[G.neuron0 + (P.nflag & kPathNeuron)];
            sdr[P.head].y = r;
        }
        __syncthreads();
        for (int e = tid; e < G.npath; e += NT) {
            const int att = (int)(fold[e] >> 16);
            if (att >= G.ncomp) continue;  // a path from a soma (no parent)
            if (e > 0 && (int)(fold[e - 1] >> 16) == att) continue;  // not the first path of its parent
            const double vp = V[att];
            double t = 0.0;
            for (int z = e; z < G.npath && (int)(fold[z] >> 16) == att; ++z) {
                const int h = paths[fold[z] & 0xFFFFu].head;
                t = fma(fabs(gax[h]), V[h] - vp, t);
            }
            sdr[att].y = fma(scale_of(att), t, sdr[att].y);
        }
        __syncthreads();

        // Team of each warp: T warps per sweep bundle (T = 1, 2 or 4), the
        // teams taking the item's bundles in turn, each on its own named
        // barrier (1 + team; 0 is the block's).
        const int nwarp = NT / 32;
        int T = nwarp / max(G.nbundle, 1);
        T = T >= 4 ? 4 : (T >= 2 ? 2 : 1);
        const int team = (tid >> 5) / T, nteam = nwarp / T;
        const int tl = tid - team * T * 32;  // lane within the team
        const int TL = T * 32, lane = tid & 31;
        auto team_sync = [&]() {
            if (T == 1) __syncwarp();
            else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(TL) : "memory");
        };

        // The head of a path once its inside is eliminated (N, M, S of the
        // head): for the path from a soma its y, else its factors and, if no
        // other path hangs off the same compartment, its elimination into the
        // parent: d_p -= gamma f, r_p += gamma c.
        auto eliminate_head = [&](const PathQ &P, double N, double M, double S) {
            const int h = P.head;
            const double inv = rcp_nr(N), c = div_nr(S, N, inv);
            if (P.parent < 0) {
                sdr[h] = make_double2(-1.0, c);
                return;
            }
            const double g = -__ldg(sc + h);
            const double f = div_nr(g * M, N, inv);
            sdr[h] = make_double2(-f, c);
            if (P.nflag & kPathAlone) {
                double2 w = sdr[P.parent];
                w.x = fma(-g, f, w.x);
                w.y = fma(g, c, w.y);
                sdr[P.parent] = w;
            }
        };
        // one step: compartment j (its coupling's exponent k) into the one
        // above (its diagonal and rhs w)
        auto step = [](double &N, double &M, double &S, int k, const double2 &w) {
            const int d = exponent2(N);
            const double Nn = __hiloint2double(__double2hiint(N) - d, __double2loint(N));
            N = fma(w.x, Nn, -scale2(M, 2 * k - d));
            S = fma(w.y, Nn, scale2(S, k - d));
            M = Nn;
        };
        // One path by one lane, leaf to head: whole chunks, the couplings of
        // the next loaded (from L2) while the current is eliminated, then the
        // rest (indices past the head clamped, their results dropped).
        auto eliminate_path = [&](int pi) {
            const PathQ P = paths[pi];
            const int h = P.head;
            int j = P.end - 1;
            const double2 v0 = sdr[j];
            double N = v0.x, M = 1.0, S = v0.y;
            int kn[kSweepChunk];
            auto load = [&](int jj) {
#pragma unroll
                for (int z = 0; z < kSweepChunk; ++z) kn[z] = __ldg(kexp + max(jj - z, h));
            };
            load(j);
            for (; j - h >= kSweepChunk; j -= kSweepChunk) {
                int k[kSweepChunk];
                double2 w[kSweepChunk];
#pragma unroll
                for (int z = 0; z < kSweepChunk; ++z) {
                    k[z] = kn[z];
                    w[z] = sdr[j - z - 1];
                }
                load(j - kSweepChunk);
#pragma unroll
                for (int z = 0; z < kSweepChunk; ++z) {
                    step(N, M, S, k[z], w[z]);
                    if (j - z - 1 > h) sdr[j - z - 1] = make_double2(N, S);
                }
            }
            const int cnt = j - h;
            double2 w[kSweepChunk - 1];
#pragma unroll
            for (int z = 0; z < kSweepChunk - 1; ++z) w[z] = sdr[max(j - z - 1, h)];
#pragma unroll
            for (int z = 0; z < kSweepChunk - 1; ++z) {
                if (z < cnt) {
                    step(N, M, S, kn[z], w[z]);
                    if (z < cnt - 1) sdr[j - z - 1] = make_double2(N, S);
                }
            }
            eliminate_head(P, N, M, S);
        };
        // The same by a whole warp.  The pivots' recursion in (N, M) would
        // compose into matrices whose parts cancel, to the square of a chunk's
        // length where the couplings are far above C / dt (pivots off by 1e-9 on
        // a chain of 4,000 wide compartments).  The pivot less the link to the
        // compartment above, X = N / M - L, only adds: with U the link as the
        // compartment above holds it (L U = gamma^2) and d its diagonal,
        //   X_{j-1} = (d_{j-1} - U - L_{j-1}) + U X_j / (L_j + X_j),
        // a quotient of linear forms in X with positive factors.  Each lane
        // composes its chunk's as a 2x2 matrix and a warp scan combines them; with
        // the pivot at its chunk's end a lane runs the steps of its chunk, stores
        // -f and composes the rhs recursion R_{j-1} = f_j R_j + r_{j-1}
        // (R = S / M), which a second scan combines; then c = R M / N.
        // 2,000 neurons of 50 to 5,000 compartments 484 -> 495 us per step, the
        // chain of 4,000 off by 1e-13 mV after a step instead of 8e-10, as with a
        // lane for each path; warps from 128 or 160 compartments 498 and 501 us,
        // none 522 us, and 701 neurons of 50 to 3,000 210, 213 and 282 for 210.
        auto eliminate_path_warp = [&](int pi) {
            const PathQ P = paths[pi];
            const int h = P.head, e = P.end;
            const int m = e - 1 - h;  // steps t = 0 .. m-1: compartment e-1-t into e-2-t
            const int cs = (m + 31) >> 5;
            const int t0 = min(lane * cs, m), t1 = min(t0 + cs, m);
            const unsigned F = 0xFFFFFFFFu;
            const double2 leaf = sdr[e - 1];
            // the matrix's entries by a power of two, the largest then in [1, 2)
            double m00 = 1.0, m01 = 0.0, m10 = 0.0, m11 = 1.0;
            auto normalise = [&]() {
                const int x = max(max(__double2hiint(m00), __double2hiint(m01)), max(__double2hiint(m10), __double2hiint(m11)));
                const int d = 0x3FF00000 - (x & 0x7FF00000);
                m00 = scale2(m00, d);
                m01 = scale2(m01, d);
                m10 = scale2(m10, d);
                m11 = scale2(m11, d);
            };
            // a link as one end (scale x) holds it; r: the reciprocal of the other end's scale
            auto link = [](double x, double r, int k) { return scale2(x * r, k); };
            double2 nb = make_double2(0.0, 0.0);
            double l0 = 0.0;  // L of the chunk's first compartment
            if (t0 < t1) {
                int i = e - 2 - t0, ka = __ldg(kexp + i + 1);
                const double sl = scale_of(i + 1);
                double sb = scale_of(i), ra = rcp_nr(sl), rb = rcp_nr(sb);
                double L = link(sl, rb, ka);
                l0 = L;
                for (int t = t0; t < t1; ++t, --i) {
                    const double2 w = sdr[i];
                    const double U = link(sb, ra, ka);
                    double Lu = 0.0, su = 1.0, ru = 1.0;
                    int ku = 0;
                    if (i > h) {
                        ku = __ldg(kexp + i);
                        su = scale_of(i - 1);
                        ru = rcp_nr(su);
                        Lu = link(sb, ru, ku);
                    }
                    const double A = w.x - Lu, B = (A - U) * L;
                    const double n00 = fma(A, m00, B * m10), n01 = fma(A, m01, B * m11);
                    m10 = fma(L, m10, m00);
                    m11 = fma(L, m11, m01);
                    m00 = n00;
                    m01 = n01;
                    normalise();
                    ra = rb;
                    ka = ku;
                    sb = su;
                    rb = ru;
                    L = Lu;
                    nb = w;
                }
            }
            for (int off = 1; off < 32; off <<= 1) {
                const double a00 = __shfl_up_sync(F, m00, off), a01 = __shfl_up_sync(F, m01, off),
                             a10 = __shfl_up_sync(F, m10, off), a11 = __shfl_up_sync(F, m11, off);
                if (lane >= off) {  // this lane's steps act after the earlier lanes'
                    const double n00 = fma(m00, a00, m01 * a10), n01 = fma(m00, a01, m01 * a11);
                    const double n10 = fma(m10, a00, m11 * a10), n11 = fma(m10, a01, m11 * a11);
                    m00 = n00;
                    m01 = n01;
                    m10 = n10;
                    m11 = n11;
                    normalise();
                }
            }
            // the pivot of the chunk's first compartment
            double N = leaf.x;
            {
                const double b00 = __shfl_up_sync(F, m00, 1), b01 = __shfl_up_sync(F, m01, 1),
                             b10 = __shfl_up_sync(F, m10, 1), b11 = __shfl_up_sync(F, m11, 1);
                const double X = leaf.x - __shfl_sync(F, l0, 0);
                if (lane) N = fma(b00, X, b01) / fma(b10, X, b11) + l0;
            }
            double M = 1.0, A = 1.0, B = 0.0, none = 0.0;
            __syncwarp();  // every lane has read its chunk and the element after it
            for (int t = t0; t < t1; ++t) {
                const int j = e - 1 - t, k = __ldg(kexp + j);
                const double2 w = t + 1 < t1 ? sdr[j - 1] : nb;
                const double f = scale2(div_nr(M, N, rcp_nr(N)), k);
                sdr[j].x = -f;
                A *= f;
                B = fma(f, B, w.y);
                step(N, M, none, k, w);
            }
            for (int off = 1; off < 32; off <<= 1) {
                const double pa = __shfl_up_sync(F, A, off), pb = __shfl_up_sync(F, B, off);
                if (lane >= off) {
                    B = fma(A, pb, B);
                    A *= pa;
                }
            }
            const double ea = __shfl_up_sync(F, A, 1), eb = __shfl_up_sync(F, B, 1);
            double R = lane ? fma(ea, leaf.y, eb) : leaf.y;
            for (int t = t0; t < t1; ++t) {
                const int j = e - 1 - t;
                const double f = -sdr[j].x, r = t + 1 < t1 ? sdr[j - 1].y : nb.y;
                sdr[j].y = R * scale2(f, -__ldg(kexp + j));
                R = fma(f, R, r);
            }
            // the head, from the lane whose chunk ends at it
            const int lastl = (m - 1) / cs;
            N = __shfl_sync(F, N, lastl);
            M = __shfl_sync(F, M, lastl);
            R = __shfl_sync(F, R, lastl);
            __syncwarp();
            if (lane == 0) eliminate_head(P, N, M, R * M);
            __syncwarp();
        };
        // eliminations into the compartments that several paths of the level
        // hang off (fold entries e0 .. e1-1); a lane takes the entries that
        // start a run of equal parents
        auto fold_shared = [&](int e0, int e1) {
            for (int e = e0 + tl; e < e1; e += TL) {
                const int att = (int)(fold[e] >> 16);
                if (e > e0 && (int)(fold[e - 1] >> 16) == att) continue;
                double2 w = sdr[att];
                for (int z = e; z < e1 && (int)(fold[z] >> 16) == att; ++z) {
                    const int h = paths[fold[z] & 0xFFFFu].head;
                    const double g = -__ldg(sc + h);
                    const double2 q = sdr[h];
                    w.x = fma(g, q.x, w.x);
                    w.y = fma(g, q.y, w.y);
                }
                sdr[att] = w;
            }
        };
        // The factors of the compartments b0 .. b1-1 whose division is not
        // done: f = gamma M / N, c = S / N with M the N of the compartment below
        // (its power of two taken out, as the elimination does), 1 at a leaf --
        // a compartment followed by one whose first member is negative, or by
        // the end.
        auto divide = [&](int b0, int b1) {
            for (int i0 = b0; i0 < b1; i0 += TL) {
                const int i = i0 + tl;
                double2 w = make_double2(-1.0, 0.0);
                double M = 1.0;
                if (i < b1) {
                    w = sdr[i];
                    if (i + 1 < b1) {
                        const double x = sdr[i + 1].x;
                        if (!signbit(x)) M = mantissa(x);
                    }
                }
                if (signbit(w.x)) {
                    w.x = -w.x;
                } else {
                    const double inv = rcp_nr(w.x);
                    w = make_double2(scale2(div_nr(M, w.x, inv), __ldg(kexp + i)), div_nr(w.y, w.x, inv));
                }
                team_sync();  // the compartment above has read this one's N
                if (i < b1) sdr[i] = w;
            }
        };

        // F. root-to-leaves substitution; the path from a soma runs the spike
        //    test
        auto substitute_head = [&](const PathQ &P) -> double {
            const double2 w = sdr[P.head];
            if (P.parent >= 0) return fma(w.x, sdr[P.parent].y, w.y);
            const double x = w.y;
            const double v0 = V[P.head], v1 = v0 + x;
            const int nrn = G.neuron0 + (P.nflag & kPathNeuron);
            if (!isfinite(v1)) atomicOr(&a.ctl->err, MMK_ERR_NUMERIC);
            if (v0 < a.threshold && v1 >= a.threshold) {
                const int src = soma_source(a, nrn);
                if (src >= 0)
                    record_spike(a, src, a.user_id[nrn], 0, (double)n * a.dt + a.dt * (a.threshold - v0) / (v1 - v0), n);
            }
            return x;
        };
        auto substitute_path = [&](int pi) {
            const PathQ P = paths[pi];
            const int h = P.head;
            double x = substitute_head(P);
            if (P.parent >= 0) sdr[h].y = x;
            int j = h + 1;
            for (; j + kSweepChunk <= P.end; j += kSweepChunk) {
                double2 w[kSweepChunk];
#pragma unroll
                for (int k = 0; k < kSweepChunk; ++k) w[k] = sdr[j + k];
#pragma unroll
                for (int k = 0; k < kSweepChunk; ++k) {
                    x = fma(w[k].x, x, w[k].y);
                    sdr[j + k].y = x;
                }
            }
            const int cnt = P.end - j;
            double2 w[kSweepChunk - 1];
#pragma unroll
            for (int k = 0; k < kSweepChunk - 1; ++k) w[k] = sdr[min(j + k, P.end - 1)];
#pragma unroll
            for (int k = 0; k < kSweepChunk - 1; ++k) {
                if (k < cnt) {
                    x = fma(w[k].x, x, w[k].y);
                    sdr[j + k].y = x;
                }
            }
        };
        auto substitute_path_warp = [&](int pi) {
            const PathQ P = paths[pi];
            const int h = P.head, e = P.end;
            double x = 0.0;
            if (lane == 0) x = substitute_head(P);
            x = __shfl_sync(0xFFFFFFFFu, x, 0);
            const int m = e - 1 - h;  // t = 0 .. m-1 <-> j = h+1+t
            const int cs = (m + 31) >> 5;
            const int t0 = min(lane * cs, m), t1 = min(t0 + cs, m);
            double A = 1.0, B = 0.0;
            for (int t = t0; t < t1; ++t) {
                const double2 w = sdr[h + 1 + t];
                A *= w.x;
                B = fma(w.x, B, w.y);
            }
            for (int off = 1; off < 32; off <<= 1) {
                const double pa = __shfl_up_sync(0xFFFFFFFFu, A, off), pb = __shfl_up_sync(0xFFFFFFFFu, B, off);
                if (lane >= off) {
                    B = fma(A, pb, B);
                    A *= pa;
                }
            }
            const double ea = __shfl_up_sync(0xFFFFFFFFu, A, 1), eb = __shfl_up_sync(0xFFFFFFFFu, B, 1);
            double xs = lane ? fma(ea, x, eb) : x;
            for (int t = t0; t < t1; ++t) {
                const double2 w = sdr[h + 1 + t];
                xs = fma(w.x, xs, w.y);
                sdr[h + 1 + t].y = xs;
            }
            __syncwarp();
            if (lane == 0 && P.parent >= 0) sdr[h].y = x;
        };
        // the number of paths at the start of a level (paths run longest
        // first) that a whole warp takes
        auto warp_paths = [&](int pb, int pe) {
            int nw = 0;
            while (pb + nw < pe && paths[pb + nw].end - paths[pb + nw].head >= kWarpPath) ++nw;
            return nw;
        };

        // B from the deepest level up, the division, F from the somata down;
        // then gate chunks of the previous item.
        for (int k = team; k < G.nbundle; k += nteam) {
            const NrnQ Nk = nrns[k];
            const int16_t *lo = loffs + Nk.loff0;
            const int16_t *mc = mcnt + Nk.loff0;
            for (int l = Nk.nlevel - 1; l >= 0; --l) {
                const int pb = lo[l], pe = lo[l + 1];
                const int nw = warp_paths(pb, pe);
                for (int q = tl >> 5; q < nw; q += T) eliminate_path_warp(pb + q);
                for (int pi = pb + nw + tl; pi < pe; pi += TL) eliminate_path(pi);
                team_sync();
                if (mc[l] > 0) {
                    fold_shared(pb, pb + mc[l]);
                    team_sync();
                }
            }
            divide(Nk.comp0, Nk.comp0 + Nk.ncomp);
            team_sync();
            for (int l = 0; l < Nk.nlevel; ++l) {
                const int pb = lo[l], pe = lo[l + 1];
                const int nw = warp_paths(pb, pe);
                for (int q = tl >> 5; q < nw; q += T) substitute_path_warp(pb + q);
                for (int pi = pb + nw + tl; pi < pe; pi += TL) substitute_path(pi);
                team_sync();
            }
        }
        gate_chunks(a, s_pc0, s_pn, &s_gchunk, lane);
        __syncthreads();

        // C. V^{n+1} = V^n + dV, dV = s y, and the threshold test of the detection
        //    points other than somata.
        for (int i = tid; i < G.ncomp; i += NT) {
            const double v0 = V[i], v = fma(scale_of(i), sdr[i].y, v0);
            a.V[c0 + i] = v;
            if (a.pt_of && v0 < a.threshold && v >= a.threshold) {
                const int p = a.pt_of[c0 + i];
                if (p >= 0) point_spike(a, p, v0, v, n, a.dt);
            }
        }
        if (tid == 0) {  // this item's gates are pending until the next item's sweeps
            s_pc0 = c0;
            s_pn = G.ncomp;
            s_gchunk = 0;
        }
    }
    // the last item's gates, by the whole block
    gate_chunks(a, s_pc0, s_pn, &s_gchunk, tid & 31);
}

__global__ void advance_kernel(DevCtl *ctl, int steps) { ctl->step_base += (unsigned long long)steps; }

// Spikes of external sources into the ring slots of their steps, as if the
// step kernel had recorded them: source id N + src[i] appended to slot
// step[i] % R (and its bit in the fired mask of deterministic delivery).  A
// slot holds at most Nsrc ids: an append beyond that is undone and flagged.
__global__ void inject_kernel(int32_t *ring_nrn, int32_t *ring_cnt, int32_t R, int32_t Nsrc, int32_t N,
                              uint32_t *fired, int32_t fired_words, const int32_t *src, const int64_t *step, int64_t n,
                              DevCtl *ctl)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int slot = (int)(step[i] % R);
        const int id = N + src[i];
        const int p = atomicAdd(&ring_cnt[slot], 1);
        if (p >= Nsrc) {
            atomicSub(&ring_cnt[slot], 1);
            atomicOr(&ctl->err, MMK_ERR_OVERFLOW);
            continue;
        }
        ring_nrn[(long long)slot * Nsrc + p] = id;
        if (fired) atomicOr(&fired[(long long)slot * fired_words + (id >> 5)], 1u << (id & 31));
    }
}

__global__ void gather_f64_kernel(const double *src, const int64_t *idx, double *dst, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[idx[i]];
}

__global__ void scatter_f64_kernel(const double *src, const int64_t *idx, double *dst, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[idx[i]] = src[i];
}

__global__ void fill_f64_kernel(double *dst, double v, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = v;
}

int grid_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 8) b = 152 * 8;
    return (int)b;
}

}  // namespace

int mmk_launch_init(const InitArgs &a, void *stream)
{
    init_kernel<<<grid_for(a.C, 256), 256, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

int mmk_launch_scale(const ScaleArgs64 &a, int n_groups, void *stream)
{
    scale_kernel<<<n_groups, 128, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

int mmk_launch_deliver(const DeliverArgs &a, int blocks, void *stream)
{
    if (a.n_dclass > kMaxDClass) return (int)cudaErrorInvalidValue;
    deliver_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

int mmk_launch_deliver_ordered(const DeliverArgs &a, int blocks, void *stream)
{
    deliver_ordered_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

int mmk_launch_step_fp64(const StepArgs &a, int blocks, int threads, void *stream)
{
    const size_t smem = (size_t)a.smem_bytes;
    cudaStream_t s = (cudaStream_t)stream;
    switch (threads) {
    case 128:
        step_fp64_kernel<128><<<blocks, 128, smem, s>>>(a);
        break;
    case 256:
        step_fp64_kernel<256><<<blocks, 256, smem, s>>>(a);
        break;
    case 512:
        step_fp64_kernel<512><<<blocks, 512, smem, s>>>(a);
        break;
    default:
        return (int)cudaErrorInvalidValue;
    }
    return (int)cudaGetLastError();
}

// The dynamic shared-memory limit only ever grows (see the FP32c kernels:
// several networks of one process share the kernel's attribute).
template <int NT>
static int fp64_attr_and_occupancy(int smem, int *blocks)
{
    static std::mutex mu;
    static int limit = 0;
    cudaError_t e = cudaSuccess;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (smem > limit) {
            e = cudaFuncSetAttribute(step_fp64_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e == cudaSuccess) limit = smem;
        }
    }
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, step_fp64_kernel<NT>, NT, smem);
    return (int)e;
}

int mmk_step_fp64_blocks_per_sm(int threads, int smem_bytes, int *blocks)
{
    switch (threads) {
    case 128: return fp64_attr_and_occupancy<128>(smem_bytes, blocks);
    case 256: return fp64_attr_and_occupancy<256>(smem_bytes, blocks);
    case 512: return fp64_attr_and_occupancy<512>(smem_bytes, blocks);
    default: return (int)cudaErrorInvalidValue;
    }
}

int mmk_launch_inject(int32_t *ring_nrn, int32_t *ring_cnt, int32_t R, int32_t Nsrc, int32_t N, uint32_t *fired,
                      int32_t fired_words, const int32_t *src, const int64_t *step, int64_t n, DevCtl *ctl,
                      void *stream)
{
    if (n <= 0) return 0;
    inject_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(ring_nrn, ring_cnt, R, Nsrc, N, fired,
                                                                      fired_words, src, step, n, ctl);
    return (int)cudaGetLastError();
}

int mmk_launch_advance(DevCtl *ctl, int steps, void *stream)
{
    advance_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(ctl, steps);
    return (int)cudaGetLastError();
}

int mmk_launch_gather_f64(const double *src, const int64_t *idx, double *dst, int64_t n, void *stream)
{
    if (n <= 0) return 0;
    gather_f64_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(src, idx, dst, n);
    return (int)cudaGetLastError();
}

int mmk_launch_scatter_f64(const double *src, const int64_t *idx, double *dst, int64_t n, void *stream)
{
    if (n <= 0) return 0;
    scatter_f64_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(src, idx, dst, n);
    return (int)cudaGetLastError();
}

int mmk_launch_fill_f64(double *dst, double v, int64_t n, void *stream)
{
    if (n <= 0) return 0;
    fill_f64_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(dst, v, n);
    return (int)cudaGetLastError();
}

namespace mmk {
__global__ void bounded_wait_selftest_kernel(int *err, uint32_t max_polls)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (!mbar_wait_bounded(&bar, 0u, max_polls) && threadIdx.x == 0) atomicOr(err, MMK_ERR_TIMEOUT);
}
}  // namespace mmk

int mmk_launch_wait_selftest(int *err, unsigned int max_polls, void *stream)
{
    mmk::bounded_wait_selftest_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(err, max_polls);
    return (int)cudaGetLastError();
}
