// Weight gradients of a surrogate layer (CI -> CO channels, padded to CIP, COP = 16, 32 or
// 48) on the tensor cores (tcgen05, BF16 operands, FP32 accumulation in TMEM):
//
//   dW[t][co][ci] = sum_n g[n][co] h[n + o(t)][ci],    t = (tz*3 + ty)*3 + tx, o = (tx-1, ty-1, tz-1)
//
// with g the gradient of the layer's output and h its (activated) input: BF16 [site][C]
// activations, or the thin FP32 network input / loss gradient, converted to BF16 and
// zero-padded while staged.  The sites are the reduction (K) dimension, so both operands are read
// MN-major: shared memory holds 16-byte entries (8 channels of one site) laid out
// [channel group][site], where eight consecutive sites form one 128-byte core matrix and
// a one-site shift of a tap is a 16-byte shift of the descriptor's start address.
//
// A work unit is one x row (z, y) of N sites, split into K chunks of 16 sites.  Per chunk
// and x tap (three MMAs, M = 128, N = 3 CIP, K = 16):
//  * B (N rows) is h of the three rows y-1, y, y+1 of one plane, staged [row][group][x]
//    with a one-site periodic halo in x: the 3 CIP rows (y tap, input channel) are evenly
//    strided, so the three y taps are one MMA (N = 3 CIP);
//  * A (M = 128 rows) is g of row (z, y) in rows 0 .. COP-1 and, in the first block group, g of
//    row (z-1, y) in the COP rows after them; the other rows are nobody's.
// The first group stages h of plane z-1: the first rows accumulate the tz = 0 taps of output
// plane z and the next ones the tz = 1 taps of plane z-1 (each plane is the z-1 of exactly
// one unit, periodic in z).  The second group stages h of plane z+1 (tz = 2) and multiplies g by a constant block of ones as well (N = 16), which sums
// db[co] = sum_n g[n][co].  A block accumulates its units in TMEM and writes one partial per
// tap (and per bias); a second kernel sums the partials in a fixed order.
//
// A block's units follow each other in y, so a unit needs one new row of h: the rows live in a
// ring of their own (kDwRowsExtra more than the units in flight, which keeps every row that an
// unfinished unit reads), and an MMA is split in two where its three rows wrap around the ring.
// Staging all three rows with every unit moved 4.5 GB through L2 for a 48-channel layer at 128^3,
// 9 TB/s in 500 us.
//
// Warp roles, synchronised by mbarriers only: an elected lane of warp 0 issues the MMAs; warps 1-6 stage
// units with cp.async, whose arrivals on the slot's barrier come when they land, as many units
// ahead as there are slots (FP32 operands: loaded into registers a unit ahead, converted and
// stored); warps 7-10 read the accumulators back at the end.  All
// waits are bounded and report through the status word.
#include <cuda_bf16.h>
#include <stdint.h>

#include "cl_internal.cuh"
#include "kernel_common.cuh"
#include "surrogate_common.cuh"
#include "tcgen05_ops.cuh"

namespace clk {

constexpr int kDwMaxSlots = 6;   // units in flight (slots of A) at most
constexpr int kDwStage = 192;    // staging threads (warps 1-6)
// Rows of the h ring beyond the units in flight: a unit reads three rows, and the next one's rows
// start one further, or three further where a new plane begins (at most once in kDwMaxSlots
// units, N being 16 or more).  When unit s is staged, unit s - slots is done; the rows of the
// slots - 1 units in between and of s itself number at most slots - 1 + 2 + 3 = slots + 4.
constexpr int kDwRowsExtra = 4;
constexpr int kDwThreads = 32 + kDwStage + 128;
constexpr int kDwF32 = 4;        // FP32 entries a staging thread holds a unit ahead

// 16-byte entries of an A slot (the channel blocks of the two g rows, N + 1 sites each: the +1
// spreads the blocks over the shared-memory banks; an MMA's M = 128 rows read 16 blocks, those past
// the slot into whatever follows, rows of the accumulator that nobody reads), of a row of h (CIP / 8
// groups of N + 2 sites), and of the block of ones and its zero block (16 sites each).
__host__ __device__ inline int dw_a_entries(int COP, int N) { return 2 * (COP / 8) * (N + 1); }
__host__ __device__ inline int dw_row_entries(int CIP, int N) { return (CIP / 8) * (N + 2); }
constexpr int kDwOnes = 32;

template <int CIP, int COP>
struct DwTCShape {
    static constexpr int CGA = COP / 8;     // channel groups of g (A, per half)
    static constexpr int CG = CIP / 8;      // channel groups of h (B)
    static constexpr int NT = 3 * CIP;      // MMA N of an x tap: three y taps x CIP input channels
    static constexpr int COLS = 3 * NT + 16;  // the x taps, then the ones (bias) block
    static constexpr int TMEM_COLS = COLS <= 256 ? 256 : 512;
    static_assert(COLS <= 512, "accumulators exceed TMEM");
    static_assert(kDwStage % CGA == 0 && kDwStage % CG == 0, "staging threads per channel group");
};

template <int CIP, int COP, bool GF32, bool HF32>
__global__ void __launch_bounds__(kDwThreads, 1) k_conv_dw_tc(const ConvDWTCArgs A)
{
    using S = DwTCShape<CIP, COP>;
    constexpr int CGA = S::CGA, CG = S::CG, NT = S::NT;
    extern __shared__ __align__(128) uint4 smem[];
    __shared__ __align__(8) uint64_t s_full[kDwMaxSlots];   // unit staged in the slot (an arrival a staging thread)
    __shared__ __align__(8) uint64_t s_freeb[kDwMaxSlots];  // slot's unit read by its MMAs (commit)
    __shared__ __align__(8) uint64_t s_done;                // every MMA of the block complete (commit)
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int N = A.N, NS = A.nslot, HR = NS + kDwRowsExtra, grp = blockIdx.y;
    const int AST = N + 1, BST = N + 2;  // entries between channel blocks of A, of B
    const int AENT = dw_a_entries(COP, N), ROW = dw_row_entries(CIP, N);
    uint4* const hring = smem + (size_t)NS * AENT;
    uint4* const ones = hring + (size_t)HR * ROW;
    const long long units = (long long)N * N;
    const long long u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
    const int nblk_a = grp == 0 ? 2 : 1;  // g rows staged into A
    // channel groups that are staged: FP32 operands have at most three channels, one group
    constexpr int GA = GF32 ? 1 : CGA, GB = HF32 ? 1 : CG;

    // zeros once: channels that are not staged, and everything an MMA may read past an A slot
    for (int e = tid; e < NS * AENT + HR * ROW; e += blockDim.x) smem[e] = make_uint4(0u, 0u, 0u, 0u);
    // the block of ones (channel 0 = 1) beside a zero block
    if (tid < kDwOnes) ones[tid] = make_uint4(tid < kDwOnes / 2 ? 0x3F80u : 0u, 0u, 0u, 0u);  // BF16 1.0
    if (tid == 0) {
        for (int k = 0; k < NS; ++k) {
            mbar_init(&s_full[k], kDwStage * (1 + (GF32 || HF32)));  // copies landed (, stores done)
            mbar_init(&s_freeb[k], 1);
        }
        mbar_init(&s_done, 1);
        mbar_fence_init();
        s_fail = 0;
    }
    if (warp == 0) {
        tmem_alloc(&s_tmem, S::TMEM_COLS);
        tmem_relinquish();
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = s_tmem;
    auto wait = [&](uint64_t* bar, uint32_t& phases, int bit) {
        if (!mbar_wait_bounded(bar, (phases >> bit) & 1u, s_fail ? 1000000ull : 2000000000ull)) s_fail = 1;
        phases ^= 1u << bit;
    };

    if (warp == 0) {
        // ------------------------------------------------------------ MMA issuer
        // accumulator columns: x tap dx at dx NT, the bias at 3 NT
        if (elect_one()) {
            uint32_t full_ph = 0;
            int seq = 0, row = 0;  // ring slot of the unit's row y - 1
            const uint32_t sbo_a = (uint32_t)AST * 16, sbo_b = (uint32_t)BST * 16, h0 = smem_u32(hring);
            const uint64_t odesc = smem_desc(smem_u32(ones), 128, kDwOnes / 2 * 16);
            constexpr uint32_t idesc1 = idesc_bf16_mn(128, 16);
            int y = (int)(u0 % N);
            for (long long u = u0; u < u1; ++u, ++seq) {
                const int slot = seq % NS;
                wait(&s_full[slot], full_ph, slot);
                fence_proxy_async_smem();  // the copies wrote through the generic proxy
                tc_fence_after();
                // the rows y-1, y, y+1: n1 of them before the ring's end, the others from its start
                const int n1 = min(3, HR - row);
                const uint32_t id1 = idesc_bf16_mn(128, CIP) + (uint32_t)((n1 - 1) * (CIP >> 3) << 17);
                const uint32_t id2 = idesc_bf16_mn(128, CIP) + (uint32_t)((2 - n1) * (CIP >> 3) << 17);
                // descriptors of chunk 0; one step of their start address is 16 bytes: a chunk of 16
                // sites is 16 steps on, an x tap one.  One thread issues every MMA, so what it
                // computes for each is time the tensor core waits: building both descriptors,
                // choosing the shape and the predicate for each MMA took 150 cycles, where M = 128,
                // N = 144 runs at 72 (hidden layer at 128^3: 434 -> 319 us)
                const uint64_t ad = smem_desc(smem_u32(smem + (size_t)slot * AENT), 128, sbo_a);
                const uint64_t b1 = smem_desc(h0 + (uint32_t)(row * ROW) * 16, 128, sbo_b), b2 = smem_desc(h0, 128, sbo_b);
                const uint32_t t2 = tbase + n1 * CIP;
                int kc = 0;
                if (u == u0) {  // the first chunk overwrites
                    kc = 1;
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) tc_mma(tbase + dx * NT, ad, b1 + dx, id1, 0);
                    if (n1 < 3) {
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx) tc_mma(t2 + dx * NT, ad, b2 + dx, id2, 0);
                    }
                    if (grp == 1) tc_mma(tbase + 3 * NT, ad, odesc, idesc1, 0);
                }
                auto chunks = [&](uint32_t t, uint64_t b, uint32_t id) {
                    uint64_t a = ad + 16 * kc;
                    b += 16 * kc;
#pragma unroll 4
                    for (int k = kc; k < N / 16; ++k, a += 16, b += 16) {
                        tc_mma_acc(t, a, b, id);
                        tc_mma_acc(t + NT, a, b + 1, id);
                        tc_mma_acc(t + 2 * NT, a, b + 2, id);
                    }
                };
                chunks(tbase, b1, id1);
                if (n1 < 3) chunks(t2, b2, id2);
                if (grp == 1) {
                    uint64_t a = ad + 16 * kc;
#pragma unroll 4
                    for (int k = kc; k < N / 16; ++k, a += 16) tc_mma_acc(tbase + 3 * NT, a, odesc, idesc1);
                }
                tc_commit(&s_freeb[slot]);  // the slot may be restaged once these MMAs completed
                y = y + 1 == N ? 0 : y + 1;
                row += y == 0 ? 3 : 1;  // a new plane starts with three rows of its own
                if (row >= HR) row -= HR;
            }
            if (u1 > u0) tc_commit(&s_done);
        }
        __syncwarp();
    } else if (warp < 1 + kDwStage / 32) {
        // ------------------------------------------------------------ staging warps
        // Each thread keeps one channel group (its index mod the groups of a site) and steps
        // through the sites: no division in the loops.
        const int st = tid - 32;
        const int dzh = grp == 0 ? -1 : 1;  // plane of h relative to the unit
        constexpr int SXA = kDwStage / GA, SXB = kDwStage / GB;
        const int cga = st % GA, xa0 = st / GA;
        const int cgb = st % GB, pb0 = st / GB;
        uint32_t free_ph = 0;
        int seq = 0, row = 0;
        auto wrap = [&](int v) { return v < 0 ? v + N : (v >= N ? v - N : v); };
        // FP32 operands: channels (up to three) of the entries xa0, xa0 + 96, .. of the unit's g
        // rows, or pb0, pb0 + 96, .. of its row y + 1 of h, in registers
        float fr[kDwF32][3];
        auto site3 = [&](const float* p, int nc, float (&f)[3]) {
#pragma unroll
            for (int c = 0; c < 3; ++c) f[c] = c < nc ? __ldg(p + c) : 0.f;
        };
        auto entry3 = [&](const float (&f)[3]) {
            const float v[8] = {f[0], f[1], f[2], 0.f, 0.f, 0.f, 0.f, 0.f};
            return pack_bf16x8(v);
        };
        auto load_f32 = [&](long long u) {
            if constexpr (GF32) {
                const int z = (int)(u / N), y = (int)(u - (long long)z * N);
#pragma unroll
                for (int i = 0; i < kDwF32; ++i) {
                    const int e = xa0 + i * kDwStage, half = e >= N ? 1 : 0, x = e - half * N;
                    if (e < nblk_a * N)
                        site3(reinterpret_cast<const float*>(A.g) + (((size_t)(half ? wrap(z - 1) : z) * N + y) * N + x) * A.g_c,
                              A.g_c, fr[i]);
                }
            }
            if constexpr (HF32) {
                const int z = (int)(u / N), y = (int)(u - (long long)z * N);
                const size_t r0 = ((size_t)wrap(z + dzh) * N + wrap(y + 1)) * N;
#pragma unroll
                for (int i = 0; i < kDwF32; ++i) {
                    const int p = pb0 + i * kDwStage;
                    if (p < BST) site3(reinterpret_cast<const float*>(A.h) + (r0 + wrap(p - 1)) * A.h_c, A.h_c, fr[i]);
                }
            }
        };
        if (u1 > u0) load_f32(u0);
        for (long long u = u0; u < u1; ++u, ++seq) {
            const int slot = seq % NS;
            if (seq >= NS) wait(&s_freeb[slot], free_ph, slot);
            const int z = (int)(u / N), y = (int)(u - (long long)z * N);
            uint4* sa = smem + (size_t)slot * AENT;
            // A: g of row (z, y) into channel blocks 0.., and of row (z-1, y) into the blocks after them
            if constexpr (GF32) {
#pragma unroll
                for (int i = 0; i < kDwF32; ++i) {
                    const int e = xa0 + i * kDwStage, half = e >= N ? 1 : 0;
                    if (e < nblk_a * N) sa[half * CGA * AST + (e - half * N)] = entry3(fr[i]);
                }
            } else {
                for (int half = 0; half < nblk_a; ++half) {
                    const size_t r0 = ((size_t)(half ? wrap(z - 1) : z) * N + y) * N;
                    uint4* d = sa + (half * CGA + cga) * AST;
                    for (int x = xa0; x < N; x += SXA)
                        cp_async16(d + x, reinterpret_cast<const __nv_bfloat16*>(A.g) + (r0 + x) * COP + cga * 8);
                }
            }
            // B: h of row y+1 of plane z + dzh, x from -1 to N (periodic); at the start of a plane
            // (and of the block) the rows y-1 and y before it
            const int zh = wrap(z + dzh);
            for (int dy = (u == u0 || y == 0) ? 0 : 2; dy < 3; ++dy) {
                const int rs = row + dy >= HR ? row + dy - HR : row + dy;
                const size_t r0 = ((size_t)zh * N + wrap(y + dy - 1)) * N;
                uint4* d = hring + (size_t)rs * ROW + cgb * BST;
                if constexpr (HF32) {
#pragma unroll
                    for (int i = 0; i < kDwF32; ++i) {
                        const int p = pb0 + i * kDwStage;
                        if (p < BST) {
                            float f[3];
                            if (dy < 2) site3(reinterpret_cast<const float*>(A.h) + (r0 + wrap(p - 1)) * A.h_c, A.h_c, f);
                            d[p] = entry3(dy < 2 ? f : fr[i]);
                        }
                    }
                } else {
                    for (int p = pb0; p < BST; p += SXB)
                        cp_async16(d + p, reinterpret_cast<const __nv_bfloat16*>(A.h) + (r0 + wrap(p - 1)) * CIP + cgb * 8);
                }
            }
            row += y + 1 == N ? 3 : 1;
            if (row >= HR) row -= HR;
            // the slot is full when every thread's copies have landed: the arrivals come by
            // themselves, so the next unit's copies wait for its slot only
            cp_async_arrive(&s_full[slot]);
            if constexpr (GF32 || HF32) {
                fence_proxy_async_smem();
                mbar_arrive(&s_full[slot]);
            }
            if (u + 1 < u1) load_f32(u + 1);
        }
        cp_async_wait0();
    } else {
        // ------------------------------------------------------------ epilogue warps
        const int q = warp & 3;           // TMEM lane quarter of this warp
        const int r = 32 * q + lane;      // accumulator row
        const int half = r / COP, co = r - half * COP;
        const bool any = u1 > u0;
        uint32_t done_ph = 0;
        if (any) {
            wait(&s_done, done_ph, 0);
            tc_fence_after();
        }
        const bool valid = half < nblk_a;
        float* P = grp == 0 ? A.part0 + (size_t)blockIdx.x * 18 * COP * CIP : A.part1 + (size_t)blockIdx.x * 9 * COP * CIP;
        auto load16 = [&](int col, uint32_t (&raw)[16]) {
            if (any) {
                tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + col, raw);
                tmem_wait<16>(raw);
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) raw[e] = 0u;
            }
        };
#pragma unroll 1
        for (int dx = 0; dx < 3; ++dx) {
            const int cbase = dx * NT;
#pragma unroll 1
            for (int c16 = 0; c16 < NT / 16; ++c16) {
                uint32_t raw[16];
                load16(cbase + c16 * 16, raw);
                if (valid) {
                    const int col = c16 * 16, dy = col / CIP, ci0 = col - dy * CIP;
                    const int tl = (half * 3 + dy) * 3 + dx;  // tap within the group's planes
                    float4* o = reinterpret_cast<float4*>(P + ((size_t)tl * COP + co) * CIP + ci0);
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        o[v] = make_float4(__uint_as_float(raw[4 * v]), __uint_as_float(raw[4 * v + 1]),
                                           __uint_as_float(raw[4 * v + 2]), __uint_as_float(raw[4 * v + 3]));
                }
            }
        }
        {  // the ones column: sum of g over this block's sites (the second group's rows 0-63)
            uint32_t raw[16];
            load16(3 * NT, raw);
            if (grp == 1 && half == 0) A.bpart[(size_t)blockIdx.x * COP + co] = __uint_as_float(raw[0]);
        }
        tc_fence_before();
    }
    __syncthreads();  // the epilogue waited for every MMA; no copy is in flight
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tbase, S::TMEM_COLS);
    if (tid == 0 && s_fail) atomicOr(A.status, ST_TIMEOUT);
}

// dW[t][co][ci] (CO x CI real channels) = sum over the blocks of the group owning plane tz
// of their padded partials, db[co] = sum of the bias partials (fixed orders).
__global__ void k_conv_dw_tc_reduce(const ConvDWTCArgs A, int CIP, int COP)
{
    const int cc = A.CO * A.CI, pp = COP * CIP, total = 27 * cc + A.CO;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        if (i < 27 * cc) {
            const int t = i / cc, r = i - t * cc, co = r / A.CI, ci = r - co * A.CI;
            float s = 0.f;
            if (t < 18) {
                const size_t j = (size_t)t * pp + co * CIP + ci;
                for (int b = 0; b < A.nb; ++b) s += A.part0[(size_t)b * 18 * pp + j];
            } else {
                const size_t j = (size_t)(t - 18) * pp + co * CIP + ci;
                for (int b = 0; b < A.nb; ++b) s += A.part1[(size_t)b * 9 * pp + j];
            }
            A.dW[i] = s;
        } else {
            const int co = i - 27 * cc;
            double s = 0.0;
            for (int b = 0; b < A.nb; ++b) s += A.bpart[(size_t)b * COP + co];
            A.db[co] = (float)s;
        }
    }
}

size_t conv_dw_tc_smem(int CIP, int COP, int N, int nslot)
{
    // (the last slot's MMAs read up to 16 blocks from its start)
    const size_t rest = (size_t)(nslot + kDwRowsExtra) * dw_row_entries(CIP, N) + kDwOnes;
    const size_t past = (size_t)16 * (N + 1) - dw_a_entries(COP, N);
    return ((size_t)nslot * dw_a_entries(COP, N) + (rest > past ? rest : past)) * 16;
}

int conv_dw_tc_slots(int CIP, int COP, int N)
{
    if ((CIP != 16 && CIP != 32 && CIP != 48) || (COP != 16 && COP != 32 && COP != 48) || N < 16 || N % 16 != 0) return 0;
    // larger lattices keep their weight gradients in FP32 on the CUDA cores
    if (N > (CIP == 16 ? 288 : CIP == 32 ? 224 : 192)) return 0;
    static_assert(2 * 288 <= kDwF32 * kDwStage, "FP32 entries a staging thread holds");
    for (int s = kDwMaxSlots; s >= 2; --s)
        if (conv_dw_tc_smem(CIP, COP, N, s) <= (size_t)kPassMaxSmem) return s;
    return 0;
}

template <int CIP, int COP, bool GF32, bool HF32>
static cudaError_t launch_dw_tc_t(const ConvDWTCArgs& A, cudaStream_t s)
{
    const size_t smem = conv_dw_tc_smem(CIP, COP, A.N, A.nslot);
    cudaError_t e = cudaFuncSetAttribute(k_conv_dw_tc<CIP, COP, GF32, HF32>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_conv_dw_tc<CIP, COP, GF32, HF32><<<dim3(A.nb, 2), kDwThreads, smem, s>>>(A);
    return cudaGetLastError();
}

// (CIP, COP, FP32 g, FP32 h): hidden layers, the first layer (FP32 network input) and the
// last layer (FP32 loss gradient) of hidden widths 16, 32 and 48
#define CL_DW_SHAPES(X)                                                                            \
    X(16, 16, false, false) X(32, 32, false, false) X(48, 48, false, false) X(16, 16, false, true) \
    X(16, 32, false, true) X(16, 48, false, true) X(16, 16, true, false) X(32, 16, true, false)   \
    X(48, 16, true, false)

cudaError_t launch_conv_dw_tc(int CIP, int COP, const ConvDWTCArgs& A, cudaStream_t s)
{
    if (A.nslot < 2 || A.nslot > kDwMaxSlots || A.nslot > conv_dw_tc_slots(CIP, COP, A.N) || A.nb < 1 || A.CI < 1 ||
        A.CI > CIP || A.CO < 1 || A.CO > COP || (A.h_f32 && A.h_c != A.CI) || (A.g_f32 && A.g_c != A.CO) ||
        (!A.h_f32 && A.CI != CIP) || (!A.g_f32 && A.CO != COP) || (A.g_f32 && A.h_f32))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaErrorInvalidValue;
    const bool gf = A.g_f32 != 0, hf = A.h_f32 != 0;
#define CL_DW_LAUNCH(a, b, c, d) \
    if (CIP == a && COP == b && gf == c && hf == d) e = launch_dw_tc_t<a, b, c, d>(A, s);
    CL_DW_SHAPES(CL_DW_LAUNCH)
#undef CL_DW_LAUNCH
    if (e != cudaSuccess) return e;
    const int total = 27 * A.CO * A.CI + A.CO;
    k_conv_dw_tc_reduce<<<(total + 255) / 256, 256, 0, s>>>(A, CIP, COP);
    return cudaGetLastError();
}

}  // namespace clk
