// GW pass with staged planes (FP32 rows of whole 16-byte units; included by gw_pass.cu).
//
// Nothing couples the five components within a pass, so a work unit is one component of one
// (y tile, z chunk): it stages only the scalars, its v and its pi_v (NF + 2 arrays a plane instead
// of NF + 10), which leaves room for tiles of up to 14 warps' rows and five or six planes in
// flight, where all components together leave three rows.  The units of a tile are neighbours in
// the grid-stride order, so the five blocks that need a tile's scalars read them together: four
// of the five reads hit L2.  One persistent block per SM, a producer warp copying plane after
// plane across unit boundaries, consumers as in k_scalar_pass_tma_nr: own row drifted into
// registers, z neighbours from registers, x neighbours by shuffles, the y neighbours' v drifted
// again from the stage (the same fused multiply-add as its owner's).  The arithmetic runs on pairs.
//
// Bound by HBM (88 bytes a site and pass with two fields): 5.3 TB/s at 256^3 FP32, two fields.
template <int NF>
__global__ void __launch_bounds__(480, 1) k_gw_pass_tma(const GwPassArgs<float> A, int S)
{
    constexpr int VW = 4, VP = 2, NARR = NF + 2;  // staged arrays: phi_f, v, pi_v
    extern __shared__ __align__(128) unsigned char gw_smem[];
    __shared__ __align__(8) uint64_t s_full[kGwStages], s_empty[kGwStages];
    __shared__ double s_coef[2];
    __shared__ int s_timeout;
    const int N = A.N, BY = A.BY, TX = N / VW;
    const int tid = threadIdx.x, nthr = blockDim.x, CT = nthr - 32, CW = CT / 32;
    const bool producer = tid >= CT;
    const int r = tid < BY * TX ? tid / TX : BY, tx = tid < BY * TX ? tid % TX : 0;
    const int x0 = tx * VW;
    const int arr_stride = (BY + 2) * N, stage_stride = NARR * arr_stride;
    float* stage = reinterpret_cast<float*>(gw_smem);
    const int units = A.nby * A.nbz * kGwC;
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&s_full[s], 1);
            mbar_init(&s_empty[s], CW);
        }
        mbar_fence_init();
        s_timeout = 0;
    }
    __syncthreads();
    auto unit = [&](int u, int& c, int& y0, int& z0, int& NZ) {
        c = u % kGwC;
        const int t = u / kGwC, by = t % A.nby, bz = t / A.nby;
        y0 = by * BY;
        z0 = bz * A.DZ;
        NZ = min(A.DZ, N - z0);
    };
    if (producer) {
        const int lane = tid - CT;
        int st = 0, issued = 0;
        uint32_t empty_phase = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            int c, y0, z0, NZ;
            unit(u, c, y0, z0, NZ);
            const int R = min(BY, N - y0);
            const int ylo = y0 == 0 ? N - 1 : y0 - 1, yhi = y0 + R == N ? 0 : y0 + R;
            const uint32_t plane_bytes = (uint32_t)(NARR * (R + 2) * N * sizeof(float));
            const int a = lane / 3, part = lane - 3 * (lane / 3);
            const float* src = a < NF ? A.phi_in[a < NF ? a : 0] : (a == NF ? A.v_in[c] : A.pv_in[c]);
            const int y = part == 0 ? ylo : (part == 1 ? y0 : yhi);
            const int srow = part == 0 ? 0 : (part == 1 ? 1 : R + 1), nrows = part == 1 ? R : 1;
            int zz = z0 == 0 ? N - 1 : z0 - 1;
            for (int j = 0; j < NZ + 2; ++j) {
                if (issued >= S) {
                    if (!mbar_wait_bounded(&s_empty[st], (empty_phase >> st) & 1u,
                                           s_timeout ? 1000000ull : 2000000000ull))
                        s_timeout = 1;
                    empty_phase ^= 1u << st;
                }
                if (lane == 0) mbar_arrive_expect_tx(&s_full[st], plane_bytes);
                __syncwarp();
                if (lane < 3 * NARR)
                    tma_bulk_g2s(stage + st * stage_stride + a * arr_stride + srow * N, src + ((size_t)zz * N + y) * N,
                                 (uint32_t)(nrows * N * sizeof(float)), &s_full[st]);
                __syncwarp();
                ++issued;
                st = st + 1 == S ? 0 : st + 1;
                zz = zz + 1 == N ? 0 : zz + 1;
            }
        }
        if (!copies_landed(s_full, S, issued, s_timeout != 0)) s_timeout = 1;
    } else {
        using P2 = Two;
        const bool do_drift = (A.flags & P_DRIFT) != 0;
        if (tid < 2) {  // beside the copies of the first planes
            const bool expand = (A.flags & P_EXPANSION) != 0;
            const double a_new = A.scal->a, a_old = expand ? A.scal->a_prev : a_new;
            const double p = apow(tid == 0 ? 0.5 * (a_old + a_new) : a_new, tid == 0 ? A.alpha - 3.0 : 1.0 + A.alpha);
            s_coef[tid] = tid == 0 ? A.d * p : p;
        }
        named_barrier_sync(3, CT);
        const P2 cd = both((float)s_coef[0]), six = both(-6.f);
        const P2 cL = both((float)(s_coef[1] / (A.dx * A.dx)));
        const P2 cS = both((float)(2.0 * A.kappa * s_coef[1] * 0.25 / (A.dx * A.dx)));  // with the (1/2dx)^2 of the source
        const P2 ck = both((float)A.k), third = both(-1.f / 3.f);
        const int lane = tid & 31;
        const bool own = tid < BY * TX;
        const bool xm_lane = own && lane > 0 && tx > 0, xp_lane = own && lane < 31 && tx < TX - 1;
        const int xm_idx = x0 == 0 ? N - 1 : x0 - 1, xp_idx = x0 + VW == N ? 0 : x0 + VW;
        const size_t plane = (size_t)N * N;
        P2 plo[NF][VP], pmid[NF][VP], pnew[NF][VP];  // scalars of planes j-2, j-1, j
        P2 vlo[VP], vmid[VP], vnew[VP], pcur[VP], pnext[VP];
        int st = 0, st_prev = 0;
        uint32_t full_phase = 0;
        auto load4 = [&](P2(&d)[VP], const float* p) {
            const float4 q = *reinterpret_cast<const float4*>(p);
            d[0] = P2(q.x, q.y);
            d[1] = P2(q.z, q.w);
        };
        auto store4 = [&](float* p, const P2(&s)[VP]) {
            *reinterpret_cast<float4*>(p) = make_float4(s[0].lo(), s[0].hi(), s[1].lo(), s[1].hi());
        };
        auto drifted_row = [&](P2(&v)[VP], P2(&pv)[VP], const float* p) {  // p: the row in the stage's v
            load4(v, p);
            load4(pv, p + arr_stride);
            if (do_drift) {
                v[0] = fma2(cd, pv[0], v[0]);
                v[1] = fma2(cd, pv[1], v[1]);
            }
        };
        // the pairs (x-1, x) and (x+1, x+2) of a row vector c whose outer neighbours are xm, xp
        auto left = [&](const P2(&c)[VP], float xm, int i) { return i == 0 ? P2(xm, c[0].lo()) : P2(c[0].hi(), c[1].lo()); };
        auto right = [&](const P2(&c)[VP], float xp, int i) { return i == 0 ? P2(c[0].hi(), c[1].lo()) : P2(c[1].hi(), xp); };
        auto release = [&](int s_idx) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[s_idx]);
        };
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            int c, y0, z0, NZ;
            unit(u, c, y0, z0, NZ);
            const int R = min(BY, N - y0);
            float* v_out = A.v_out[c];
            float* pv_out = A.pv_out[c];
            const size_t row_off = (size_t)(y0 + r) * N + x0;
            int zz = z0 == 0 ? N - 1 : z0 - 1;
            for (int j = 0; j < NZ + 2; ++j) {
                if (!mbar_wait_bounded(&s_full[st], (full_phase >> st) & 1u, s_timeout ? 1000000ull : 2000000000ull))
                    s_timeout = 1;
                full_phase ^= 1u << st;
                if (r < R) {  // own row of plane j
                    const float* sb = stage + st * stage_stride + (r + 1) * N + x0;
#pragma unroll
                    for (int f = 0; f < NF; ++f) load4(pnew[f], sb + f * arr_stride);
                    drifted_row(vnew, pnext, sb + NF * arr_stride);
                    if (j >= 1 && j <= NZ) store4(v_out + (size_t)zz * plane + row_off, vnew);
                }
                if (j >= 2) {  // kick plane j-1
                    const float* sp = stage + st_prev * stage_stride + r * N;  // the row below, in the stage
                    P2 src[VP] = {both(0.f), both(0.f)}, lap[VP];
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const float xm_s = __shfl_up_sync(0xffffffffu, pmid[f][1].hi(), 1);
                        const float xp_s = __shfl_down_sync(0xffffffffu, pmid[f][0].lo(), 1);
                        if (r < R) {
                            const float* q = sp + f * arr_stride;
                            P2 ym[VP], yp[VP];
                            load4(ym, q + x0);
                            load4(yp, q + 2 * N + x0);
                            const float xm = xm_lane ? xm_s : q[N + xm_idx], xp = xp_lane ? xp_s : q[N + xp_idx];
#pragma unroll
                            for (int i = 0; i < VP; ++i) {
                                const P2 g0 = sub2(right(pmid[f], xp, i), left(pmid[f], xm, i));
                                const P2 g1 = sub2(yp[i], ym[i]), g2 = sub2(pnew[f][i], plo[f][i]);
                                // components 11, 12, 13, 22, 23 of Pi - delta tr / 3
                                if (c == 1) src[i] = fma2(g0, g1, src[i]);
                                else if (c == 2) src[i] = fma2(g0, g2, src[i]);
                                else if (c == 4) src[i] = fma2(g1, g2, src[i]);
                                else {
                                    const P2 tr = fma2(g0, g0, fma2(g1, g1, mul2(g2, g2))), d = c == 0 ? g0 : g1;
                                    src[i] = fma2(third, tr, fma2(d, d, src[i]));
                                }
                            }
                        }
                    }
                    {
                        const float xm_s = __shfl_up_sync(0xffffffffu, vmid[1].hi(), 1);
                        const float xp_s = __shfl_down_sync(0xffffffffu, vmid[0].lo(), 1);
                        if (r < R) {
                            const float* q = sp + NF * arr_stride;
                            P2 ym[VP], yp[VP], pv[VP];
                            drifted_row(ym, pv, q + x0);
                            drifted_row(yp, pv, q + 2 * N + x0);
                            auto edge = [&](int x) {
                                const float v = q[N + x];
                                return do_drift ? fma_rn(cd.lo(), q[arr_stride + N + x], v) : v;
                            };
                            const float xm = xm_lane ? xm_s : edge(xm_idx), xp = xp_lane ? xp_s : edge(xp_idx);
#pragma unroll
                            for (int i = 0; i < VP; ++i) {
                                const P2 s = add2(add2(add2(right(vmid, xp, i), left(vmid, xm, i)), add2(yp[i], ym[i])),
                                                  add2(vnew[i], vlo[i]));
                                lap[i] = fma2(six, vmid[i], s);
                                pcur[i] = fma2(ck, fma2(cL, lap[i], mul2(cS, src[i])), pcur[i]);
                            }
                            store4(pv_out + (size_t)(z0 + j - 2) * plane + row_off, pcur);
                        }
                    }
                }
                if (j >= 1) release(st_prev);
#pragma unroll
                for (int i = 0; i < VP; ++i) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        plo[f][i] = pmid[f][i];
                        pmid[f][i] = pnew[f][i];
                    }
                    vlo[i] = vmid[i];
                    vmid[i] = vnew[i];
                    pcur[i] = pnext[i];
                }
                st_prev = st;
                st = st + 1 == S ? 0 : st + 1;
                zz = zz + 1 == N ? 0 : zz + 1;
            }
            release(st_prev);
        }
    }
    __syncthreads();  // producer and consumers meet; no copy is in flight past this point
    if (tid == 0 && s_timeout) atomicOr(&A.scal->status, ST_TIMEOUT);
}

// Where the staged pass runs: from 96^3 (us a leapfrog pass with the scalars, direct / staged: 39.6 /
// 41.7 at 80^3, 59.6 / 51.9 at 100^3, 85.6 / 81.4 at 128^3, 520 / 413 at 256^3; of the last, the GW launch
// 375 / 277, floor 220 at the copy rate).  Its tiling: the tallest tile of up to 448 consumer threads that leaves four
// stages or more (at most kGwStages), z chunks that minimise waves x (planes + 2) of the busiest SM.
bool gw_tma_tiles(int precision, int nf, int N, int nsm, int* BY, int* DZ, int* stages)
{
    if (precision == CL_PREC_FP64 || N % 4 != 0 || N < 96 || N / 4 > 448) return false;
    const int TX = N / 4;
    int by = std::min(N, 448 / TX), S = 0;
    for (; by >= 1; --by) {
        const size_t per = (size_t)(nf + 2) * (by + 2) * N * sizeof(float);
        S = (int)std::min<size_t>(kGwStages, (size_t)kPassMaxSmem / per);
        if (S >= 4) break;
    }
    if (by < 1) return false;
    const int nby = (N + by - 1) / by;
    by = (N + nby - 1) / nby;
    long long best = -1;
    for (int nbz = 1; nbz <= N; ++nbz) {
        const int dz = (N + nbz - 1) / nbz;
        if ((N + dz - 1) / dz != nbz) continue;
        const long long waves = ((long long)nby * nbz * kGwC + nsm - 1) / nsm, cost = waves * (dz + 2);
        if (best < 0 || cost < best) {
            best = cost;
            *DZ = dz;
        }
    }
    *BY = by;
    *stages = S;
    return true;
}

template <int NF>
static cudaError_t launch_gw_tma_t(const GwPassArgs<float>& A, int stages, int grid, cudaStream_t s)
{
    const size_t smem = (size_t)stages * (NF + 2) * (A.BY + 2) * A.N * sizeof(float);
    const int threads = (A.BY * (A.N / 4) + 31) / 32 * 32 + 32;
    if (A.N % 4 != 0 || stages < 3 || stages > kGwStages || smem > (size_t)kPassMaxSmem || threads > 480)
        return cudaErrorInvalidValue;
    static DevFlag attr;
    if (!attr) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_gw_pass_tma<NF>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPassMaxSmem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_gw_pass_tma<NF><<<grid, threads, smem, s>>>(A, stages);
    return cudaGetLastError();
}

cudaError_t launch_gw_pass_tma(int nf, const void* args, int stages, int grid, cudaStream_t s)
{
    const auto& A = *static_cast<const GwPassArgs<float>*>(args);
    return nf == 1 ? launch_gw_tma_t<1>(A, stages, grid, s) : launch_gw_tma_t<2>(A, stages, grid, s);
}
