// Ringless TMA-staged fused pass for rows that are no multiple of 16 bytes (included by
// scalar_pass.cu after the vector kernel).  The producer, the stage protocol and the
// arithmetic are those of k_scalar_pass_tma_nr; what differs is the row geometry.
//
// Bulk copies start on 16-byte boundaries, but row (z, y) starts at element (z N + y) N.  Each
// part of a plane (lower halo row, the R own rows, upper halo row) is therefore copied from the
// boundary at or below its first element to the one at or above its last, into a region of its
// own, and is read from the shift that its first element has to that boundary: 0..E-1 elements
// (E = 16 / sizeof(T)), the same for every array, from the plane and the row alone.  The last
// copy of an array may read up to 12 bytes past its last element: arrays passed to this kernel
// are allocated in multiples of 256 bytes.
//
// A warp owns 32 CH consecutive sites of the tile's R N own sites (whole rows are consecutive
// in memory), lane l the sites 32 k + l: shared loads and global stores are lane-contiguous at
// any alignment (the vectors of the aligned kernel would split here), and the tile fills the
// threads whatever N is.  x neighbours come from the warp's registers by shuffles; the first
// and last site of a row or of a warp's sites drift their neighbour again from the stage.
//
// The arithmetic runs on pairs of sites (Two): the kernel is bound by issue and the latency
// behind it (14 consumer warps an SM, 56 % of the issue slots at 251^3, two fields), and packed
// instructions take half the slots of the scalar ones: 213 -> 174 us a pass.  The energy sums stay
// scalar, every site added to the thread's compensated sum by itself: pairs of sums take twice the
// registers of the sums and spill (227 us with them; sums of the two fields in pairs 192).  Copying every row
// with scalar loads through the direct loader took 619 us there (363 -> 92 with one field; 125^3
// two fields 94 -> 36; 250^3, 8-byte vectors, 263 -> 174); HBM alone would need 113 us.
template <int NF, bool KAHAN, int CH, int S>
__global__ void __launch_bounds__(480, 1) k_scalar_pass_tma_any(const ScalarPassArgs<float> A)
{
    using T = float;
    constexpr int KPF = KAHAN ? 3 : 2;
    constexpr int NARR = NF * KPF;
    constexpr int E = 16 / (int)sizeof(T);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t s_full[S];
    __shared__ __align__(8) uint64_t s_empty[S];
    __shared__ double s_coef[4];
    __shared__ double s_red[32][kMaxQ];
    __shared__ int s_last, s_timeout;

    const int N = A.N, BY = A.BY;
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int CT = nthr - 32, CW = CT / 32;
    const bool producer = tid >= CT;
    const int HN = any_region<E>(N), ON = any_own_region<E>(N, BY);  // elements of a halo row's and the own rows' region
    const int arr_stride = 2 * HN + ON;
    const int stage_stride = NARR * arr_stride;
    T* stage = reinterpret_cast<T*>(smem_raw);
    long long u0, u1;
    block_units(N, A.nby, A.DZ, u0, u1);

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            mbar_init(&s_full[s], 1);
            mbar_init(&s_empty[s], CW);
        }
        mbar_fence_init();
        s_timeout = 0;
    }
    __syncthreads();
    Acc<T> accK[NF], accG[NF], accV;

    if (producer) {
        const int lane = tid - CT;
        int st = 0;
        uint32_t empty_phase = 0;
        int issued = 0;
        for (long long u = u0; u < u1;) {
            const int tile = (int)(u / N);
            const int z0 = (int)(u - (long long)tile * N);
            const int NZ = (int)min((long long)(N - z0), u1 - u);
            const int y0 = tile * BY, R = min(BY, N - y0);
            const int ylo = y0 == 0 ? N - 1 : y0 - 1;
            const int yhi = y0 + R == N ? 0 : y0 + R;
            u += NZ;
            // this lane's copy of a plane: array lane / 3, part lane % 3
            const int a = lane / 3, part = lane - 3 * (lane / 3);
            const int f = a / KPF, kind = a - KPF * (a / KPF);
            const T* src = lane < 3 * NARR ? (kind == 0 ? A.phi_in[f] : (kind == 1 ? A.pi_in[f] : A.c_in[f])) : nullptr;
            const int y = part == 0 ? ylo : (part == 1 ? y0 : yhi);
            const int n = part == 1 ? R * N : N;
            const int dst_off = a * arr_stride + (part == 0 ? 0 : (part == 1 ? HN : HN + ON));
            int zz = z0 == 0 ? N - 1 : z0 - 1;
            for (int j = 0; j < NZ + 2; ++j) {
                if (issued >= S) {
                    if (!mbar_wait_bounded(&s_empty[st], (empty_phase >> st) & 1u,
                                           s_timeout ? 1000000ull : 2000000000ull))
                        s_timeout = 1;
                    empty_phase ^= 1u << st;
                }
                const size_t i0 = ((size_t)zz * N + y) * N;
                const int sh = (int)(i0 & (E - 1));
                const uint32_t bytes = (uint32_t)((sh + n + E - 1) / E * 16);
                // parts 0..2 of array 0 sit in lanes 0..2; the other arrays' copies are as large
                const uint32_t plane_bytes = NARR * (__shfl_sync(0xffffffffu, bytes, 0) + __shfl_sync(0xffffffffu, bytes, 1) +
                                                     __shfl_sync(0xffffffffu, bytes, 2));
                if (lane == 0) mbar_arrive_expect_tx(&s_full[st], plane_bytes);
                __syncwarp();
                if (lane < 3 * NARR) tma_bulk_g2s(stage + st * stage_stride + dst_off, src + (i0 - sh), bytes, &s_full[st]);
                __syncwarp();
                ++issued;
                st = st + 1 == S ? 0 : st + 1;
                zz = zz + 1 == N ? 0 : zz + 1;
            }
        }
        if (!copies_landed(s_full, S, issued, s_timeout != 0)) s_timeout = 1;
    } else {
        constexpr int CP = CH / 2;  // pairs of sites (k = 2 i, 2 i + 1)
        consumer_coefficients(tid, CT, A.scal->a, A.scal->b, A.d, A.alpha, A.dx, (A.flags & P_EXPANSION) != 0, s_coef);
        const T cd = (T)s_coef[0];
        const Two cd2 = both(cd), ncd2 = both(-cd), six = both((T)-6);
        const bool do_drift = (A.flags & P_DRIFT) != 0;
        const PotCoef<T> P(A.m2, A.lam, A.g2);
        const KickCoef2 KC((T)s_coef[1], (T)s_coef[2], (T)A.e, (T)A.k, P);
        const int lane = tid & 31;
        const int first = (tid >> 5) * 32 * CH + lane;  // the lane's first site of the tile
        Two pcur[NF][CP], pnext[NF][CP];
        Two zlo[NF][CP], zmid[NF][CP], znew[NF][CP];
        int st = 0, st_prev = 0;
        uint32_t full_phase = 0;
        const size_t plane = (size_t)N * N;
        // drifted value of the field whose array starts at sa, element `off`
        auto drifted1 = [&](const T* sa, int off) -> T {
            T ph = sa[off];
            if (do_drift) {
                T cv = KAHAN ? sa[2 * arr_stride + off] : (T)0;
                drift<T, KAHAN>(ph, cv, sa[arr_stride + off], cd);
            }
            return ph;
        };
        auto release = [&](int s_idx) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[s_idx]);
        };
        for (long long u = u0; u < u1;) {
            const int tile = (int)(u / N);
            const int z0 = (int)(u - (long long)tile * N);
            const int NZ = (int)min((long long)(N - z0), u1 - u);
            const int y0 = tile * BY, R = min(BY, N - y0);
            const int ylo = y0 == 0 ? N - 1 : y0 - 1;
            const int yhi = y0 + R == N ? 0 : y0 + R;
            const int own_n = R * N;
            u += NZ;
            // which of the lane's sites are in the tile (the others compute on whatever the stage
            // holds and neither store nor add), in its first or last row, or at a row's end
            unsigned valid = 0, lo_row = 0, hi_row = 0, row_first = 0, row_last = 0;
#pragma unroll
            for (int k = 0; k < CH; ++k) {
                const int q = first + 32 * k, r = q / N, x = q - r * N;
                if (q < own_n) valid |= 1u << k;
                if (r == 0) lo_row |= 1u << k;
                if (r == R - 1) hi_row |= 1u << k;
                if (x == 0) row_first |= 1u << k;
                if (x == N - 1) row_last |= 1u << k;
            }
            const bool warp_lo = __any_sync(0xffffffffu, lo_row), warp_hi = __any_sync(0xffffffffu, hi_row);
            const size_t row_off = (size_t)y0 * N;
            int zz = z0 == 0 ? N - 1 : z0 - 1;
            int sh_prev[3] = {0, 0, 0};
            for (int j = 0; j < NZ + 2; ++j) {
                if (!mbar_wait_bounded(&s_full[st], (full_phase >> st) & 1u, s_timeout ? 1000000ull : 2000000000ull))
                    s_timeout = 1;
                full_phase ^= 1u << st;
                const T* sb = stage + st * stage_stride;
                const size_t zrow = (size_t)zz * N;
                const int sh[3] = {(int)(((zrow + ylo) * N) & (E - 1)), (int)(((zrow + y0) * N) & (E - 1)),
                                   (int)(((zrow + yhi) * N) & (E - 1))};
                const bool write_out = j >= 1 && j <= NZ;
                {  // own sites of plane j: drift, write out, keep in registers
                    const size_t base = zrow * N + row_off + first;
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const T* sa = sb + f * KPF * arr_stride + HN + sh[1] + first;
                        const T *sv = sa + arr_stride, *sc = sv + arr_stride;
                        Two cv[CP];
#pragma unroll
                        for (int i = 0; i < CP; ++i) {
                            znew[f][i] = Two(sa[64 * i], sa[64 * i + 32]);
                            pnext[f][i] = Two(sv[64 * i], sv[64 * i + 32]);
                            if (KAHAN) cv[i] = Two(sc[64 * i], sc[64 * i + 32]);
                            if (do_drift) drift2<KAHAN>(znew[f][i], cv[i], pnext[f][i], cd2, ncd2);
                        }
                        if (write_out) {
                            T *po = A.phi_out[f] + base, *co = A.c_out[f] + base;
#pragma unroll
                            for (int i = 0; i < CP; ++i) {
                                if (valid >> (2 * i) & 1u) {
                                    po[64 * i] = znew[f][i].lo();
                                    if (KAHAN) co[64 * i] = cv[i].lo();
                                }
                                if (valid >> (2 * i + 1) & 1u) {
                                    po[64 * i + 32] = znew[f][i].hi();
                                    if (KAHAN) co[64 * i + 32] = cv[i].hi();
                                }
                            }
                        }
                    }
                }
                if (j >= 2) {
                    const T* sp = stage + st_prev * stage_stride;
                    Two lap[NF][CP];
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const T* sa = sp + f * KPF * arr_stride;
                        const int own = HN + sh_prev[1] + first;
                        // y neighbours (y2): a row down or up in the own region -- one unbroken
                        // stretch, 32 elements between a lane's sites -- or the halo row
                        Two y2[CP];
                        auto load_row = [&](const T* s0) {
                            const T *s1 = s0 + arr_stride, *s2 = s1 + arr_stride;
#pragma unroll
                            for (int i = 0; i < CP; ++i) {
                                y2[i] = Two(s0[64 * i], s0[64 * i + 32]);
                                if (do_drift) {
                                    const Two m(s1[64 * i], s1[64 * i + 32]);
                                    Two c;
                                    if (KAHAN) c = Two(s2[64 * i], s2[64 * i + 32]);
                                    drift2<KAHAN>(y2[i], c, m, cd2, ncd2);
                                }
                            }
                        };
                        auto load_halo = [&](unsigned in_halo, int own_off, int halo_off) {
                            T y[CH];
#pragma unroll
                            for (int k = 0; k < CH; ++k)
                                y[k] = drifted1(sa, (in_halo >> k & 1u ? halo_off : own_off) + 32 * k);
#pragma unroll
                            for (int i = 0; i < CP; ++i) y2[i] = Two(y[2 * i], y[2 * i + 1]);
                        };
                        Two ysum[CP];
                        if (warp_lo) load_halo(lo_row, own - N, sh_prev[0] + first);
                        else load_row(sa + own - N);
#pragma unroll
                        for (int i = 0; i < CP; ++i) ysum[i] = y2[i];
                        if (warp_hi) load_halo(hi_row, own + N, HN + ON + sh_prev[2] + first - (R - 1) * N);
                        else load_row(sa + own + N);
                        Two gs[CP];
#pragma unroll
                        for (int i = 0; i < CP; ++i) {
                            const Two gy = sub2(y2[i], zmid[f][i]);
                            gs[i] = mul2(gy, gy);
                            ysum[i] = add2(y2[i], ysum[i]);
                        }
                        T xmv[CH], xpv[CH];
#pragma unroll
                        for (int k = 0; k < CH; ++k) {
                            // x neighbours: lane -+ 1, across the k blocks at the warp's ends; the
                            // first and last site of the warp and of a row from the stage
                            auto at = [&](int q) -> T { return q & 1 ? zmid[f][q / 2].hi() : zmid[f][q / 2].lo(); };
                            T xm = __shfl_sync(0xffffffffu, k > 0 && lane == 31 ? at(k > 0 ? k - 1 : 0) : at(k), (lane + 31) & 31);
                            T xp = __shfl_sync(0xffffffffu, k + 1 < CH && lane == 0 ? at(k + 1 < CH ? k + 1 : k) : at(k),
                                               (lane + 1) & 31);
                            if ((row_first >> k & 1u) || (k == 0 && lane == 0))
                                xm = drifted1(sa, own + 32 * k + (row_first >> k & 1u ? N - 1 : -1));
                            if ((row_last >> k & 1u) || (k == CH - 1 && lane == 31))
                                xp = drifted1(sa, own + 32 * k + (row_last >> k & 1u ? 1 - N : 1));
                            xmv[k] = xm;
                            xpv[k] = xp;
                        }
#pragma unroll
                        for (int i = 0; i < CP; ++i) {
                            const Two c = zmid[f][i], xm(xmv[2 * i], xmv[2 * i + 1]), xp(xpv[2 * i], xpv[2 * i + 1]);
                            lap[f][i] = fma2(six, c, add2(add2(add2(xp, xm), ysum[i]), add2(znew[f][i], zlo[f][i])));
                            const Two gx = sub2(xp, c), gz = sub2(znew[f][i], c);
                            gs[i] = fma2(gx, gx, fma2(gz, gz, gs[i]));
                            accG[f].add(valid >> (2 * i) & 1u ? gs[i].lo() : (T)0);
                            accG[f].add(valid >> (2 * i + 1) & 1u ? gs[i].hi() : (T)0);
                        }
                    }
                    const size_t base = (size_t)(z0 + j - 2) * plane + row_off + first;
#pragma unroll
                    for (int i = 0; i < CP; ++i) {
                        Two p[NF], l[NF], q[NF], k1[NF], v1 = both((T)0);
#pragma unroll
                        for (int f = 0; f < NF; ++f) {
                            p[f] = zmid[f][i];
                            l[f] = lap[f][i];
                            q[f] = pcur[f][i];
                            k1[f] = both((T)0);
                        }
                        kick_two<NF>(p, l, q, KC, k1, v1);
                        const bool va = valid >> (2 * i) & 1u, vb = valid >> (2 * i + 1) & 1u;
#pragma unroll
                        for (int f = 0; f < NF; ++f) {
                            if (va) A.pi_out[f][base + 64 * i] = q[f].lo();
                            if (vb) A.pi_out[f][base + 64 * i + 32] = q[f].hi();
                            accK[f].add(va ? k1[f].lo() : (T)0);
                            accK[f].add(vb ? k1[f].hi() : (T)0);
                        }
                        accV.add(va ? v1.lo() : (T)0);
                        accV.add(vb ? v1.hi() : (T)0);
                    }
                }
                if (j >= 1) release(st_prev);
#pragma unroll
                for (int f = 0; f < NF; ++f)
#pragma unroll
                    for (int i = 0; i < CP; ++i) {
                        zlo[f][i] = zmid[f][i];
                        zmid[f][i] = znew[f][i];
                        pcur[f][i] = pnext[f][i];
                    }
#pragma unroll
                for (int q = 0; q < 3; ++q) sh_prev[q] = sh[q];
                st_prev = st;
                st = st + 1 == S ? 0 : st + 1;
                zz = zz + 1 == N ? 0 : zz + 1;
            }
            release(st_prev);
        }
    }
    __syncthreads();
    finish_pass<T, NF>(A, accK, accG, accV, s_coef, s_red, &s_last, tid, nthr, s_timeout);
}
