// Many passes of the fused scalar pass in one launch, for lattices small enough that a pass is
// latency, not bandwidth (sm_103a).
//
// A launch per pass of a small lattice spends its time around the sites: launch and drain, one
// thread's FP64 prefactors before the first load, the march's pipeline fill, the last block's
// reduction and FP64 epilogue (FP64 operations have 70 cycles latency here, a division 450) --
// 14 us for the 32768 sites of 32^3, whose arithmetic takes one.  This kernel stays resident (one
// block per SM at most, launched cooperatively) and runs the passes of up to kPersistPasses in a
// loop, one grid barrier a pass:
//  * every block owns a box of rows (BY x BZ full x rows), its threads the box's sites in row
//    order, any N.  A site loads phi, pi, c of itself and its six neighbours (L1 and L2
//    hold them: at most 4 times the state is read) and drifts all seven with the owner's own
//    operations, so one exchange a pass suffices;
//  * a'' is linear in the lattice sums, so once the sites are done a publishing warp writes one
//    number per block, its part of a'', and arrives at the barrier; a scalar warp waits there, adds
//    every block's number in block order (each block redundantly: the same bits everywhere) and
//    forms a', the next a and the next pass's prefactors.  What depends only on a is worked out
//    while the sites are computed, and the sites load their next values while the scalar warp
//    works.  An FP64 instruction occupies its scheduler for 64 cycles whether one lane or 32 take
//    part (measured), so independent scalars sit in different lanes and warps;
//  * block 0 keeps the status and, for the last pass (and a Hubble limit), the energies.
// Measured (us a pass, one launch a pass before): 16.4 -> 4.0 at 32^3 one field FP32 + Kahan, 21.9 ->
// 7.9 at 64^3 two fields, 22.5 -> 11.4 at 96^3 one field; FP64 22.5 -> 6.2 at 32^3.  Of the 4.0, about
// 1.0 is the barrier (release, arrival, poll), 1.0 FP64 instructions of the scalar warp.
// Over a launch of one pass that is 12 us more than the pass: calls of few passes go to the kernels
// launched per pass (persist_min_passes).
// Waits are bounded: a barrier that does not complete within two seconds sets ST_TIMEOUT and
// every block leaves.
#include <type_traits>

#include "cl_internal.cuh"
#include "kernel_common.cuh"
#include "scalar_pass_common.cuh"

namespace clk {

namespace {

constexpr int kNW = 16;             // warps that compute sites
constexpr int kCT = 32 * kNW;
constexpr int kThreads = kCT + 64;  // + the scalar warp and the publishing warp

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(unsigned* p)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Exponent alpha + const of the equations of motion: n = 0..4 of x^n (neg: of 1 / x^n) by
// multiplication, any other by pow (n < 0).
struct Expo {
    int n, neg;
    double e;
};
__device__ __forceinline__ Expo expo(double e)
{
    const double m = fabs(e);
    const int n = (int)m;
    return {m <= 4.0 && (double)n == m ? n : -1, e < 0.0 ? 1 : 0, e};
}
// x^|e| in at most two dependent multiplications (n >= 0).
__device__ __forceinline__ double ipow(double x, int n)
{
    const double x2 = x * x, h = x2 * (n == 3 ? x : x2);
    return n == 0 ? 1.0 : n == 1 ? x : n == 2 ? x2 : h;
}
__device__ __forceinline__ double spow(double x, const Expo& E)
{
    if (E.n < 0) return pow(x, E.e);
    const double p = ipow(x, E.n);
    return E.neg ? 1.0 / p : p;
}
// 1 / y from a nearby reciprocal r0: with e = 1 - y r0, r0 (1 + e + e^2 + e^3), whose relative
// error is e^4 -- below 2^-52 for |e| < 2^-13 -- in four operations instead of a division's ten.
__device__ __forceinline__ double recip_near(double y, double r0)
{
    const double e = __fma_rn(-y, r0, 1.0);
    if (fabsf((float)e) < 0x1p-13f) return __fma_rn(r0, __fma_rn(e, __fma_rn(e, e, e), e), r0);
    return 1.0 / y;
}

}  // namespace

template <typename T, int NF, bool KAHAN>
__global__ void __launch_bounds__(kThreads, 1) k_scalar_persist(const PersistArgs<T> A)
{
    using Pair = typename std::conditional<sizeof(T) == 4, float2, double>::type;
    __shared__ Pair s_acc[kMaxQ][kCT];
    __shared__ double s_q[8];    // the block's sums
    __shared__ double s_a;       // the pass's a
    __shared__ T s_coef[4];      // drift and kick prefactors
    __shared__ int s_stop;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = A.N, G = (int)gridDim.x;
    const int by0 = (int)(blockIdx.x % A.nby) * A.BY, bz0 = (int)(blockIdx.x / A.nby) * A.BZ;
    const int ry = min(A.BY, N - by0), rz = min(A.BZ, N - bz0);
    const bool expand = (A.flags & P_EXPANSION) != 0;
    // partials of a pass: the blocks' a'' terms, then their five sums (written when needed), in
    // three buffers in turn.  Block 0's scalar warp reads the sums of pass p (with a Hubble limit)
    // after it has let its own block go on; the blocks that write that buffer again, for pass
    // p + 3, have passed grid barrier p + 2, where block 0 arrives after its scalar warp has
    // worked out the factors that follow pass p + 1, hence after those reads.  (With two buffers
    // they would need barrier p + 1 only, where block 0 arrives without that warp.)
    double* const part0 = A.partials;
    const size_t part_stride = (size_t)G * (kMaxQ + 1);

    if (warp == kNW + 1) {
        // ------------------------------------------------------------ the publishing warp
        // a'' is linear in the lattice sums w_q, a'' = sum_q beta_q w_q with beta_q a function of
        // a alone (lanes 0..4, worked out while the sites are computed), so each block publishes
        // one number, its own sum_q beta_q w_q.  (Without expansion: rho, for the NaN check.)
        const double idx2 = 1.0 / (A.dx * A.dx), ivol = 1.0 / ((double)N * N * N), cr = 2.0 * A.alpha - 1.0;
        const Expo e2a = expo(2.0 * A.alpha);
        const int grp = lane < 2 ? 0 : lane < 4 ? 1 : lane == 4 ? 2 : 3;  // K, G, V, none
        // a'' = ca (cr rho - 3 p): rho = K + G + V, p = K - G/3 - V
        const double unit = expand ? (A.kappa * (1.0 / 6.0)) * (grp == 0 ? cr - 3.0 : grp == 1 ? cr + 1.0 : cr + 3.0) : 1.0;
        const double konst = grp == 3 ? 0.0 : unit * ivol * (grp == 0 ? 0.5 : grp == 1 ? 0.5 * idx2 : 1.0);
        bar_sync(4, kThreads);
        for (int p = 0; p < A.passes; ++p) {
            const double a = s_a, r = 1.0 / a, r2 = r * r;
            double beta = konst * (grp == 0 ? r2 * (r2 * r2) : grp == 1 ? r2 : 1.0);
            if (expand) beta *= a * spow(a, e2a);
            const bool full = p + 1 == A.passes || A.hubble_limit > 0.0;
            bar_sync(2, 32 * (kMaxQ + 1));
            double* part = part0 + (p % 3) * part_stride;
            const double w = lane < kMaxQ ? s_q[lane] : 0.0;
            double term = beta * w;
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) term += __shfl_xor_sync(0xffffffffu, term, off);
            if (full && lane < kMaxQ) __stcg(&part[(size_t)(lane + 1) * G + blockIdx.x], w);
            __syncwarp();
            if (lane == 0) {
                __stcg(&part[blockIdx.x], term);
                red_release(A.barrier);
            }
            bar_sync(4, kThreads);
            if (s_stop) return;
        }
        return;
    }
    if (warp == kNW) {
        // ------------------------------------------------------------ the scalar warp
        // Lanes side by side: lane 0 works on the midpoint a (drift factor), lanes 1 and 2 on the
        // new a (Laplacian and potential factors); every FP64 instruction occupies its scheduler
        // for 64 cycles however many lanes it has, so their count is what a pass waits for.
        const double idx2 = 1.0 / (A.dx * A.dx), ivol = 1.0 / ((double)N * N * N);
        const Expo ex = expo(lane == 0 ? A.alpha - 3.0 : lane == 1 ? 1.0 + A.alpha : 3.0 + A.alpha);
        const double half = lane == 0 ? 0.5 : 1.0;
        DevScal* S = A.scal;
        double a = S->a, b = S->b, t = S->t, a_prev = a;
        long long step = S->step;
        int st = 0;
        // the factors of the pass that drifts (a, b) by d; r0 is near 1 / ipow(x) on lane 0
        auto factors = [&](double d, double dl, double r0, bool near) -> double {
            const double x = expand ? __fma_rn(dl, b, a) : a;
            double f;
            if (ex.n < 0) f = pow(x, ex.e);
            else {
                f = ipow(x, ex.n);
                if (ex.neg) f = near ? recip_near(f, r0) : 1.0 / f;
            }
            f *= lane == 0 ? d : lane == 1 ? idx2 : 1.0;
            if (lane < 3) s_coef[lane] = (T)f;
            return __shfl_sync(0xffffffffu, x, 1);
        };
        double a1 = factors(A.d[0], half * A.d[0], 0.0, false);
        if (lane == 0) {
            s_a = a1;
            s_stop = 0;
        }
        bar_sync(4, kThreads);
        int c = 0;  // the pass within its step
        for (int p = 0; p < A.passes; ++p) {
            const int cn = c + 1 == A.pps ? 0 : c + 1;
            // while the sites are computed: the next drift factor's reciprocal, from the a' before
            // this pass's kick
            const double dl = half * A.d[cn], ka = A.k[c];
            double r0 = 0.0;
            if (ex.n >= 0 && ex.neg) r0 = 1.0 / ipow(expand ? __fma_rn(dl, b, a1) : a1, ex.n);
            const double* part = part0 + (p % 3) * part_stride;
            int ok = 1;
            if (lane == 0) {
                const unsigned want = (unsigned)(p + 1) * G;
                if (ld_acquire(A.barrier) < want) {
                    const uint64_t t0 = global_timer_ns();
                    while (ld_acquire(A.barrier) < want)
                        if (global_timer_ns() - t0 > 2000000000ull) {
                            ok = 0;
                            break;
                        }
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            bar_arrive(3, kThreads - 32);  // the other blocks' fields are there: the sites may load
            // a'': all blocks' terms, in block order
            double v[kPersistBlocks / 32];
#pragma unroll
            for (int i = 0; i < kPersistBlocks / 32; ++i) v[i] = lane + 32 * i < G ? __ldcg(&part[lane + 32 * i]) : 0.0;
            double sum = v[0];
#pragma unroll
            for (int i = 1; i < kPersistBlocks / 32; ++i)
                if (32 * i < G) sum += v[i];
            for (int off = G > 16 ? 16 : G > 4 ? 8 : 2; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            sum = G > 16 ? sum : __shfl_sync(0xffffffffu, sum, 0);  // (lane 0 holds all of few blocks)
            const double addot = expand ? sum : 0.0, b_old = b;
            const bool last = p + 1 == A.passes || !ok;
            a_prev = a;
            a = a1;
            b = __fma_rn(ka, addot, b);
            a1 = factors(A.d[cn], dl, r0, true);
            if (lane == 0) {
                s_a = a1;
                s_stop = last ? 1 : 0;
            }
            bar_sync(4, kThreads);
            t = t + A.d[c];
            if (cn == 0) step += 1;
            if (blockIdx.x == 0) {
                if (!ok) st |= ST_TIMEOUT;
                if (!isfinite(sum)) st |= ST_NAN;
                if (last || A.hubble_limit > 0.0) {  // the energies (Eq. energy-contrib, Eq. Friedmann2)
                    double w[kMaxQ];
                    for (int q = 0; q < kMaxQ; ++q) {
                        w[q] = 0.0;
                        for (int i = lane; i < G; i += 32) w[q] += __ldcg(&part[(size_t)(q + 1) * G + i]);
                        for (int off = 16; off > 0; off >>= 1) w[q] += __shfl_xor_sync(0xffffffffu, w[q], off);
                    }
                    const double ia = 1.0 / a, ia2 = ia * ia, ck = 0.5 * (ia2 * ia2 * ia2) * ivol, cg = 0.5 * ia2 * ivol * idx2;
                    const double K0 = w[0] * ck, K1 = w[1] * ck, G0 = w[2] * cg, G1 = w[3] * cg, V = w[4] * ivol;
                    const double K = K0 + K1, Gr = G0 + G1, rho = K + Gr + V, pr = K - Gr * (1.0 / 3.0) - V;
                    const double b_int = __fma_rn(A.e[c], addot, b_old), H = b_int / a;
                    const double rhs = apow(a, 2.0 * A.alpha) * A.kappa * rho * (1.0 / 3.0);
                    const double hv = H != 0.0 ? fabs(H * H - rhs) / (H * H) : 0.0;
                    if (!isfinite(rho) || !isfinite(pr)) st |= ST_NAN;
                    if (A.hubble_limit > 0.0 && hv > A.hubble_limit) st |= ST_CONSTRAINT;
                    if (last && lane == 0) {
                        S->a_prev = a_prev;
                        S->a = a;
                        S->b = b;
                        S->t = t;
                        S->step = step;
                        const double diag[D_NDIAG] = {t, a, b_int, K0, K1, G0, G1, V, 0.0, 0.0, rho, pr, hv, 0.0};
                        for (int i = 0; i < D_NDIAG; ++i) S->diag[i] = diag[i];
                        if (st) atomicOr(&S->status, st);
                    }
                }
            }
            if (last) return;
            c = cn;
        }
        return;
    }

    // ---------------------------------------------------------------- sites
    const PotCoef<T> Pc(A.m2, A.lam, A.g2);
    int c = 0;
    // The box's sites in row order: thread t takes t, t + kCT, ...  Where it stands: (x, row yr of
    // plane zr); a step moves on by kCT sites.
    struct Spot {
        int x, yr, zr;
    };
    const int adv_rows = kCT / N, adv_x = kCT - adv_rows * N;
    Spot first;
    first.zr = tid / (N * ry);
    first.yr = tid / N - first.zr * ry;
    first.x = tid - (tid / N) * N;
    auto advance = [&](Spot& s) {
        s.x += adv_x;
        s.yr += adv_rows;
        if (s.x >= N) {
            s.x -= N;
            s.yr += 1;
        }
        while (s.yr >= ry) {
            s.yr -= ry;
            s.zr += 1;
        }
    };
    // the site and its neighbours x -+ 1, y -+ 1, z -+ 1
    auto sites = [&](const Spot& s, int (&at)[7]) {
        const int x = s.x, y = by0 + s.yr, z = bz0 + s.zr;
        const int xm = x == 0 ? N - 1 : x - 1, xp = x + 1 == N ? 0 : x + 1;
        const int ym = y == 0 ? N - 1 : y - 1, yp = y + 1 == N ? 0 : y + 1;
        const int zm = z == 0 ? N - 1 : z - 1, zp = z + 1 == N ? 0 : z + 1;
        const int r0 = (z * N + y) * N;
        at[0] = r0 + x;
        at[1] = r0 + xm;
        at[2] = r0 + xp;
        at[3] = (z * N + ym) * N + x;
        at[4] = (z * N + yp) * N + x;
        at[5] = (zm * N + y) * N + x;
        at[6] = (zp * N + y) * N + x;
    };
    for (int p = 0;; ++p) {
        const int in = (A.in0 + p) & 1, out = in ^ 1;
        T ph[NF][7], pv[NF][7], cv[NF][7];
        int at[7];
        auto load = [&]() {
#pragma unroll
            for (int f = 0; f < NF; ++f)
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    ph[f][i] = A.phi[f][in][at[i]];
                    pv[f][i] = A.pi[f][in][at[i]];
                    cv[f][i] = KAHAN ? A.c[f][in][at[i]] : (T)0;
                }
        };
        // the first site's values come in while the scalar warp works out the prefactors
        Spot spot = first;
        if (spot.zr < rz) {
            sites(spot, at);
            load();
        }
        bar_sync(4, kThreads);
        if (s_stop) break;
        const T cd = s_coef[0], cL = s_coef[1], cV = s_coef[2];
        const T ce = (T)A.e[c], ck = (T)A.k[c];
        Acc<T> accK[NF], accG[NF], accV;
        for (bool more = false; spot.zr < rz; more = true) {
            if (more) {
                sites(spot, at);
                load();
            }
            {
#pragma unroll
                for (int f = 0; f < NF; ++f) {
#pragma unroll
                    for (int i = 0; i < 7; ++i) drift<T, KAHAN>(ph[f][i], cv[f][i], pv[f][i], cd);
                    A.phi[f][out][at[0]] = ph[f][0];
                    if (KAHAN) A.c[f][out][at[0]] = cv[f][0];
                }
                const T p0 = ph[0][0], p1 = NF > 1 ? ph[NF - 1][0] : (T)0;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const T* q = ph[f];
                    const T lap = ((q[2] + q[1]) + (q[4] + q[3]) + (q[6] + q[5])) - (T)6 * q[0];
                    const T gx = q[2] - q[0], gy = q[4] - q[0], gz = q[6] - q[0];
                    accG[f].add(gx * gx + gy * gy + gz * gz);
                    T dV;
                    if (f == 0) dV = p0 * (Pc.m20 + Pc.l0 * p0 * p0 + (NF > 1 ? Pc.g2 * p1 * p1 : (T)0));
                    else dV = p1 * (Pc.m21 + Pc.l1 * p1 * p1 + Pc.g2 * p0 * p0);
                    const T F = cL * lap - cV * dV;
                    const T pe = pv[f][0] + ce * F;
                    accK[f].add(pe * pe);
                    A.pi[f][out][at[0]] = pv[f][0] + ck * F;
                }
                T v = p0 * p0 * (Pc.h_m20 + Pc.q_l0 * p0 * p0);
                if (NF > 1) v += p1 * p1 * (Pc.h_m21 + Pc.q_l1 * p1 * p1) + Pc.h_g2 * p0 * p0 * p1 * p1;
                accV.add(v);
            }
            advance(spot);
        }
        // block sums: warp q adds quantity q over the threads -- compensated FP32 sums as float
        // pairs over each warp's lanes, then in FP64 over the warps, as the other passes do; FP64
        // as it is
        const Acc<T>* const acc[kMaxQ] = {&accK[0], NF > 1 ? &accK[NF - 1] : nullptr, &accG[0],
                                          NF > 1 ? &accG[NF - 1] : nullptr, &accV};
#pragma unroll
        for (int q = 0; q < kMaxQ; ++q) {
            if constexpr (sizeof(T) == 4) s_acc[q][tid] = acc[q] ? make_float2(acc[q]->s, -acc[q]->c) : make_float2(0.f, 0.f);
            else s_acc[q][tid] = acc[q] ? acc[q]->value() : 0.0;
        }
        bar_sync(1, kCT);
        if (warp < kMaxQ) {
            if constexpr (sizeof(T) == 4) {
                F2 x[kNW];
#pragma unroll
                for (int i = 0; i < kNW; ++i) {
                    const float2 o = s_acc[warp][32 * i + lane];
                    x[i] = F2{o.x, o.y};
                }
                // a pair of lanes holds a warp's sum: one takes the high part, the other the low
                const F2 w = warp_sums<kNW>(x, lane);
                double d = (double)(lane & 1 ? w.lo : w.hi);
                for (int off = 1; off < 32; off *= 2) d += __shfl_xor_sync(0xffffffffu, d, off);
                if (lane == 0) s_q[warp] = d;
            } else {
                double x = 0.0;
                if (NF == 2 || (warp != 1 && warp != 3)) {
                    const int nw = min(kNW, (ry * rz * N + 31) / 32);  // warps with sites
                    for (int i = 0; i < nw; ++i) x += s_acc[warp][32 * i + lane];
                    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
                }
                if (lane == 0) s_q[warp] = x;
            }
            __syncwarp();
            bar_arrive(2, 32 * (kMaxQ + 1));
        }
        bar_sync(3, kThreads - 32);
        c = c + 1 == A.pps ? 0 : c + 1;
    }
}

// The box of rows of a block: the fewest rounds of the threads over an SM's sites (FP64: of one
// warp, the FP64 pipe being the bound), then the fewest blocks, then the smallest surface.
bool persist_tiles(int precision, int N, int nsm, int* BY, int* BZ)
{
    if (N > 1024) return false;
    if (nsm > kPersistBlocks) nsm = kPersistBlocks;
    const int at_once = precision == CL_PREC_FP64 ? 32 : kCT;
    long long best = -1;
    for (int by = 1; by <= N; ++by) {
        const int nby = (N + by - 1) / by;
        if (nby > nsm || (N + nby - 1) / nby != by) continue;
        for (int bz = (N + nsm / nby - 1) / (nsm / nby); bz <= N; ++bz) {
            const int nbz = (N + bz - 1) / bz;
            if ((N + nbz - 1) / nbz != bz) continue;
            const long long rounds = ((long long)by * bz * N + at_once - 1) / at_once;
            const long long cost = (rounds * 1000 + nby * nbz) * 100000 + (by + 2) * bz + by * 2;
            if (best < 0 || cost < best) {
                best = cost;
                *BY = by;
                *BZ = bz;
            }
        }
    }
    return best >= 0;
}

template <typename T, int NF, bool KAHAN>
static cudaError_t launch_persist_t(const PersistArgs<T>& A, int grid, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_scalar_persist<T, NF, KAHAN>, A);
}

cudaError_t launch_scalar_persist(int precision, int nf, const void* args, int grid, cudaStream_t s)
{
    if (precision == CL_PREC_FP64) {
        const auto& A = *static_cast<const PersistArgs<double>*>(args);
        return nf == 1 ? launch_persist_t<double, 1, false>(A, grid, s) : launch_persist_t<double, 2, false>(A, grid, s);
    }
    const auto& A = *static_cast<const PersistArgs<float>*>(args);
    if (precision == CL_PREC_FP32_KAHAN)
        return nf == 1 ? launch_persist_t<float, 1, true>(A, grid, s) : launch_persist_t<float, 2, true>(A, grid, s);
    return nf == 1 ? launch_persist_t<float, 1, false>(A, grid, s) : launch_persist_t<float, 2, false>(A, grid, s);
}

}  // namespace clk
