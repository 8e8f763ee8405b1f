// ks_reg.cuh - the float phases of a tau-step with the transforms in registers (four-launch form).
//
// The items of ks_items.cuh walk a transform through shared memory pass by pass: a 64-point float
// row pair costs six trips through it per transform, with run-time index arithmetic and a block
// barrier between them, and keeps the FMA pipe under a tenth busy.  Here a thread holds sixteen
// points and takes two radix-4 passes (or a radix-2 and a radix-4 pass) on them between trips, with
// every index known at compile time:
//   * a transform of length N = 16 T belongs to T threads; thread id holds elements id + T s,
//     s = 0 .. 15, at its input and at its output, so what is computed point by point between two
//     transforms (u u_x, u r_x, r_hat, the update) stays in registers;
//   * its passes are those of fft_batch in the same order with the same twiddles and operations,
//     so the results are the same bits in every launch form;
//   * the groups of passes exchange through shared memory once (N <= 256) or twice, within one warp
//     for N <= 512 (no block barrier), at addresses padded by one value in sixteen so that neither
//     side conflicts; the threads of a 1024-point transform are two warps that meet at a named
//     barrier.
// A warp takes 32 / T transforms: row pairs (neighbouring lanes hold neighbouring pairs: the mixed
// values of one x-mode are one 128-byte line per eight pairs) or columns of one loop.
// Lengths 32 .. 512 in x and 32 .. 1024 in s; other lengths, the centre-symmetric subspace and the
// other launch forms take the items.
#pragma once

#include "ks_items.cuh"

namespace ks {

constexpr int RG_THREADS = 128;

// two floats, loaded and stored as one
struct alignas(8) rgv {
    float x, y;
};

// ---- passes in registers --------------------------------------------------------------------
template <int DIR>
KS_HD cpx<float> rg_w(cpx<float> w) {
    return DIR > 0 ? w : conj(w);
}

// products that a transform's first additions follow: rounded, as where they pass through memory
KS_HD cpx<float> rg_scale(cpx<float> a, float g) { return mk<float>(mul_rn(a.x, g), mul_rn(a.y, g)); }

// radix-4 butterfly without twiddles (the span-1 pass of fft_batch)
template <int DIR>
KS_HD void rg_bfly(cpx<float>& a, cpx<float>& b, cpx<float>& c, cpx<float>& d) {
    const cpx<float> t0 = a + c, t1 = a - c, t2 = b + d, t3 = mul_i(b - d, DIR);
    a = t0 + t2;
    b = t1 + t3;
    c = t0 - t2;
    d = t1 - t3;
}
// with unit twiddles in a pass that has them: the same bits as bfly4_tw with w = 1
template <int DIR>
KS_HD void rg_bfly_one(cpx<float>& a, cpx<float>& b, cpx<float>& c, cpx<float>& d) {
    const cpx<float> t0 = a + c, t1 = twice_minus(a, t0), t2 = b + d;
    const cpx<float> t3 = mul_i(twice_minus(b, t2), DIR);
    a = t0 + t2;
    b = t1 + t3;
    c = t0 - t2;
    d = t1 - t3;
}
template <int DIR>
KS_HD void rg_bfly_tw(cpx<float>& a, cpx<float>& b, cpx<float>& c, cpx<float>& d,
                                           cpx<float> w1, cpx<float> w2, cpx<float> w3) {
    cpx<float> o0, o1, o2, o3;
    bfly4_tw(a, b, c, d, rg_w<DIR>(w1), rg_w<DIR>(w2), rg_w<DIR>(w3), DIR, o0, o1, o2, o3);
    a = o0;
    b = o1;
    c = o2;
    d = o3;
}

// exp(2 pi i t / 16) as the table holds it (float of the double value)
KS_HD cpx<float> rg_w16(int t) {
    constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, r = 0.70710678118654752440;
    constexpr float C[16] = {1.f, (float)c1, (float)r, (float)s1, 0.f, (float)-s1, (float)-r, (float)-c1,
                             -1.f, (float)-c1, (float)-r, (float)-s1, 0.f, (float)s1, (float)r, (float)c1};
    return mk<float>(C[t & 15], C[(t + 12) & 15]);
}

// Twiddles of the later groups, per length: the group of spans S and 4 S reads, for thread
// r = id mod S, entry i S + r: i = 0 .. 2 the radix-4 pass of span S (w_{4S}^{r q}, q = 1, 2, 3),
// i = 3 + 3 m + q - 1 the one of span 4 S (w_{16S}^{(S m + r) q}, m = 0 .. 3); a last group of one
// pass (span N / 4) reads, for thread id, entry 3 T k + T (q - 1) + id: w_N^{(id + T k) q}.
KS_HDX constexpr int rg_s(int lg) { return (lg & 1) ? 8 : 16; }     // span after the first group
KS_HDX constexpr int rg_two(int lg) { return lg >= 7 ? 15 * rg_s(lg) : 0; }   // entries of the two-pass group
KS_HDX constexpr int rg_one(int lg) { return (lg <= 6 || lg >= 9) ? 12 * (1 << (lg - 4)) : 0; }
KS_HDX constexpr int rg_len(int lg) { return rg_two(lg) + rg_one(lg); }
KS_HDX constexpr int rg_at(int lg) { return lg <= 5 ? 0 : rg_at(lg - 1) + rg_len(lg - 1); }
constexpr int RG_TABLE = rg_at(11);
// entry e of length 2^lg is exp(2 pi i t / m)
inline void rg_entry(int lg, int e, int& t, int& m) {
    const int N = 1 << lg, T = N / 16, S = rg_s(lg);
    if (e < rg_two(lg)) {
        const int i = e / S, r = e % S;
        if (i < 3) {
            m = 4 * S;
            t = r * (i + 1);
        } else {
            m = 16 * S;
            t = (S * ((i - 3) / 3) + r) * ((i - 3) % 3 + 1);
        }
        return;
    }
    e -= rg_two(lg);
    const int k = e / (3 * T), q = e / T % 3 + 1, id = e % T;
    m = N;
    t = (id + T * k) * q;
}

// Address of element p of a transform in its exchange buffer, and the buffers' stride.
KS_HDX constexpr int rg_pad(int p) { return p + (p >> 4); }
template <int LG>
struct RgShape {
    static constexpr int N = 1 << LG, T = N / 16, F = T >= 32 ? 1 : 32 / T;  // transforms of a team
    static constexpr int TEAM = T > 32 ? T : 32;                             // threads of a team
    // spreads the F transforms' lanes over the banks (see the odd lengths' first exchange)
    static constexpr int STRIDE = LG == 5 ? 33 : LG == 7 ? 140 : 17 * T;
};
constexpr int RG_XBYTES = 2 * 4 * 140 * 8;  // exchange buffer of 64 threads (128-point transforms need most)

// barrier of a team: its warp, or its two warps (named barriers 1, 2: pair of warps w / 2)
#ifdef KS_HOST_EMULATION
void rg_host_sync();  // the host build runs a team as threads
#endif
template <int LG>
KS_HD void rg_sync() {
#ifdef KS_HOST_EMULATION
    rg_host_sync();
#else
    if constexpr (RgShape<LG>::TEAM == 32) __syncwarp();
    else asm volatile("bar.sync %0, 64;\n" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
#endif
}

// The transform of the team's threads: v[s] is element id + T s.  x: this transform's exchange
// buffer; tw: the length's twiddles (rg_at(LG) into the table).
template <int LG, int DIR>
KS_HD void rg_fft(cpx<float> (&v)[16], int id, rgv* x, const rgv* tw) {
    constexpr int T = RgShape<LG>::T, S = rg_s(LG);
    auto put = [&](int p, cpx<float> a) { x[rg_pad(p)] = rgv{a.x, a.y}; };
    auto get = [&](int p) {
        const rgv a = x[rg_pad(p)];
        return mk<float>(a.x, a.y);
    };
    auto w = [&](int i) {
        const rgv a = tw[i];
        return mk<float>(a.x, a.y);
    };
    rg_sync<LG>();  // the previous transform's reads of x are done
    if constexpr ((LG & 1) == 0) {
        // spans 1 and 4: butterflies q on s = q + 4 p, then m on the outputs m of those
#pragma unroll
        for (int q = 0; q < 4; ++q) rg_bfly<DIR>(v[q], v[q + 4], v[q + 8], v[q + 12]);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            if (m == 0) rg_bfly_one<DIR>(v[0], v[1], v[2], v[3]);
            else rg_bfly_tw<DIR>(v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3], rg_w16(m), rg_w16(2 * m),
                                 rg_w16(3 * m));
#pragma unroll
            for (int k = 0; k < 4; ++k) put(16 * id + m + 4 * k, v[4 * m + k]);
        }
    } else {
        // spans 1 (radix 2) and 2: two groups g of eight, s = g + 2 q + 8 h
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            cpx<float> y[2][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const cpx<float> a = v[g + 2 * q], b = v[g + 2 * q + 8];
                y[0][q] = a + b;
                y[1][q] = a - b;
            }
            rg_bfly_one<DIR>(y[0][0], y[0][1], y[0][2], y[0][3]);
            rg_bfly_tw<DIR>(y[1][0], y[1][1], y[1][2], y[1][3], rg_w16(2), rg_w16(4), rg_w16(6));
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < 4; ++k) put(8 * (id + g * T) + m + 2 * k, y[m][k]);
        }
    }
    rg_sync<LG>();
#pragma unroll
    for (int s = 0; s < 16; ++s) v[s] = get(id + T * s);
    if constexpr (LG >= 7) {
        // spans S and 4 S
        const int r = id & (S - 1), e = id / S;
        const cpx<float> a1 = w(r), a2 = w(S + r), a3 = w(2 * S + r);
#pragma unroll
        for (int q = 0; q < 4; ++q) rg_bfly_tw<DIR>(v[q], v[q + 4], v[q + 8], v[q + 12], a1, a2, a3);
        if constexpr (LG >= 9) rg_sync<LG>();  // the reads above precede the writes below
        cpx<float> o[16];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            rg_bfly_tw<DIR>(v[4 * m], v[4 * m + 1], v[4 * m + 2], v[4 * m + 3], w((3 + 3 * m) * S + r),
                            w((4 + 3 * m) * S + r), w((5 + 3 * m) * S + r));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if constexpr (LG >= 9) put(16 * S * e + r + S * (m + 4 * k), v[4 * m + k]);
                else o[m + 4 * k] = v[4 * m + k];
            }
        }
        if constexpr (LG < 9) {
#pragma unroll
            for (int s = 0; s < 16; ++s) v[s] = o[s];
        } else {
            rg_sync<LG>();
#pragma unroll
            for (int s = 0; s < 16; ++s) v[s] = get(id + T * s);
        }
    }
    if constexpr (LG <= 6 || LG >= 9) {
        // the last pass alone: butterflies k on s = k + 4 p
        constexpr int B = rg_two(LG);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            rg_bfly_tw<DIR>(v[k], v[k + 4], v[k + 8], v[k + 12], w(B + 3 * T * k + id), w(B + 3 * T * k + T + id),
                            w(B + 3 * T * k + 2 * T + id));
    }
}

#ifndef KS_HOST_EMULATION
// ---- rows -------------------------------------------------------------------------------------
// Row tiles of the register kernels: 2 F rows of one loop per warp (fewer at the end of a loop).
struct RgTile {
    int b, n0;
};

// One row tile: pair f of the warp's F is rows n0 + 2 f, n0 + 2 f + 1, lane = id F + f.
// The rows of u between the two row phases lie in the U array as the pairs' values
// [pair][s][id] (u_a, u_b): both phases run with the same tiles and lanes.
template <int MODE, int LGX>
__device__ __forceinline__ void rg_rows(const Dims& d, const Bufs<float>& p, int b, int n0, rgv* xbuf,
                                        const rgv* tw) {
    typedef RgShape<LGX> Sh;
    constexpr int N = Sh::N, T = Sh::T, F = Sh::F, KX = N / 3;
    const int lane = threadIdx.x & 31, id = lane / F, f = lane % F;
    const int ns = p.ns[b];
    const bool on = n0 + 2 * f < ns;
    rgv* x = xbuf + f * Sh::STRIDE;
    const int na = on ? n0 + 2 * f : 0;  // idle lanes repeat the loop's first pair and store nothing
    cpx<float>* const M = p.M + p.moff[b] + na;
    float2* const U = reinterpret_cast<float2*>(p.U + p.goff[b] + (size_t)na * N) + id;
    // the mixed values of x-mode j in rows a and b
    auto load = [&](int j) { return *reinterpret_cast<const float4*>(M + (size_t)j * ns); };
    cpx<float> y[16];
    if constexpr (MODE == ROW_NONLIN) {
        // z = u + i u_x per row: Z_j = (1 - q_j) v_j, Z_{-j} = (1 + q_j) conj(v_j)   (a1, a2)
        cpx<float> za[16], zb[16];
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const int J = id + T * s;
            za[s] = zb[s] = mk<float>(0.f, 0.f);
            if (T * s <= KX && J <= KX) {
                const float4 m = load(J);
                const float g = 1.f - p.qv[J];
                za[s] = rg_scale(mk<float>(m.x, m.y), g);
                zb[s] = rg_scale(mk<float>(m.z, m.w), g);
            } else if (T * s + T - 1 >= N - KX && J >= N - KX) {
                const float4 m = load(N - J);
                const float g = 1.f + p.qv[N - J];
                za[s] = rg_scale(mk<float>(m.x, -m.y), g);
                zb[s] = rg_scale(mk<float>(m.z, -m.w), g);
            }
        }
        rg_fft<LGX, +1>(za, id, x, tw);
        rg_fft<LGX, +1>(zb, id, x, tw);
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            if (on) U[T * s] = make_float2(za[s].x, zb[s].x);
            y[s] = mk<float>(mul_rn(za[s].x, za[s].y), mul_rn(zb[s].x, zb[s].y));  // p = u u_x  (a3)
        }
    } else {
        // r_x rows: z = X_a + i X_b  (a7)
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const int J = id + T * s;
            y[s] = mk<float>(0.f, 0.f);
            if (T * s <= KX && J <= KX) {
                const float4 m = load(J);
                y[s] = mk<float>(m.x, m.y) + mul_i(mk<float>(m.z, m.w), 1);
            } else if (T * s + T - 1 >= N - KX && J >= N - KX) {
                const float4 m = load(N - J);
                y[s] = mk<float>(m.x, -m.y) + mul_i(mk<float>(m.z, -m.w), 1);
            }
        }
        float2 u[16];
#pragma unroll
        for (int s = 0; s < 16; ++s) u[s] = U[T * s];
        rg_fft<LGX, +1>(y, id, x, tw);
#pragma unroll
        for (int s = 0; s < 16; ++s) y[s] = mk<float>(mul_rn(u[s].x, y[s].x), mul_rn(u[s].y, y[s].y));  // w = u r_x  (a8)
    }
    rg_fft<LGX, -1>(y, id, x, tw);
    // split into the rows' half spectra (store_pair_spectra): mode j = id + T s wants Y[N - j] =
    // element (T - id) + T (15 - s) of thread T - id, or, for id = 0, T (16 - s) of its own
    const float h = (float)d.hx;
    const int src = ((T - id) & (T - 1)) * F + f;
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        if (T * s > KX) break;
        const cpx<float> o = y[15 - s], c = s == 0 ? y[0] : y[16 - s];
        cpx<float> ym;
        ym.x = __shfl_sync(0xffffffffu, o.x, src);
        ym.y = __shfl_sync(0xffffffffu, o.y, src);
        if (id == 0) ym = c;
        ym = conj(ym);
        const cpx<float> yj = y[s], sm = yj + ym, df = yj - ym;
        const int j = id + T * s;
        if (on && j <= KX)
            *reinterpret_cast<float4*>(M + (size_t)j * ns) =
                make_float4(sm.x * h, sm.y * h, df.y * h, -df.x * h);
    }
}

template <int MODE, int LGX>
__global__ void __launch_bounds__(RG_THREADS) k_rg_rows(Dims d, Bufs<float> p, const RgTile* tiles, int ntiles,
                                                        const rgv* tab) {
    __shared__ rgv xs[RG_THREADS / 64 * (RG_XBYTES / 8)];
    __shared__ rgv tws[rg_len(LGX)];
    grid_trigger();
    for (int i = threadIdx.x; i < rg_len(LGX); i += RG_THREADS) tws[i] = tab[rg_at(LGX) + i];
    __syncthreads();
    grid_wait();
    const int w = threadIdx.x >> 5;
    rgv* x = xs + w * (RG_XBYTES / 16);
    for (int it = blockIdx.x * (RG_THREADS / 32) + w; it < ntiles; it += gridDim.x * (RG_THREADS / 32)) {
        const RgTile t = tiles[it];
        if (loop_live(p, t.b)) rg_rows<MODE, LGX>(d, p, t.b, t.n0, x, tws);
    }
    // the step scalars of each live loop (see loops_scalars)
    if constexpr (MODE == ROW_ADJ) loops_scalars(d, p, p.par, blockIdx.x, gridDim.x);
}

// ---- columns ----------------------------------------------------------------------------------
// Sums of |r|^2 and k Im(conj(u) r) over a column, in the order of the items: element i in
// accumulator i mod 128, elements of one accumulator in order, then an xor tree over the
// accumulators with distances 16, 8, 4, 2, 1, 64, 32 (warps of 32 accumulators first).
// Accumulators past the column's end hold zeros, which change nothing, so their levels are skipped.
template <int LG>
__device__ __forceinline__ void rg_reduce(ff (&a)[16], ff (&c)[16], int id, ff* xch, ff& ra, ff& rc) {
    constexpr int T = RgShape<LG>::T;
    constexpr int NA = LG < 7 ? 16 : (128 / T);  // accumulators a thread holds (s < NA), after the
                                                 // caller's sums in order
    constexpr int dist[7] = {16, 8, 4, 2, 1, 64, 32};
    bool gone[16] = {};
#pragma unroll
    for (int l = 0; l < 7; ++l) {
        const int D = dist[l];
        if (D >= (1 << LG)) continue;
        if (D >= T) {
            const int ds = D / T;
#pragma unroll
            for (int s = 0; s < NA; ++s)
                if (!gone[s] && !(s & ds)) {
                    a[s] = ff_add(a[s], a[s ^ ds]);
                    c[s] = ff_add(c[s], c[s ^ ds]);
                    gone[s ^ ds] = true;
                }
        } else if (D < 32) {
#pragma unroll
            for (int s = 0; s < NA; ++s)
                if (!gone[s]) {
                    ff o, q;
                    o.hi = __shfl_xor_sync(0xffffffffu, a[s].hi, D);
                    o.lo = __shfl_xor_sync(0xffffffffu, a[s].lo, D);
                    q.hi = __shfl_xor_sync(0xffffffffu, c[s].hi, D);
                    q.lo = __shfl_xor_sync(0xffffffffu, c[s].lo, D);
                    a[s] = ff_add(a[s], o);
                    c[s] = ff_add(c[s], q);
                }
        } else {  // D = 32 = the other warp of a 1024-point column
            rg_sync<LG>();
            if ((id & 31) == 0) {
                xch[2 * (id >> 5)] = a[0];
                xch[2 * (id >> 5) + 1] = c[0];
            }
            rg_sync<LG>();
            a[0] = ff_add(a[0], xch[2 * ((id >> 5) ^ 1)]);
            c[0] = ff_add(c[0], xch[2 * ((id >> 5) ^ 1) + 1]);
        }
    }
    ra = a[0];
    rc = c[0];
}

// F columns j0 .. j0 + F - 1 of loop b: lane = f T + id.  MODE: COL_RESID or COL_UPDATE.
template <int MODE, int LG>
__device__ __forceinline__ void rg_cols(const Dims& d, const Bufs<float>& p, int b, int j0, rgv* xbuf,
                                        const rgv* tw) {
    typedef RgShape<LG> Sh;
    constexpr int N = Sh::N, T = Sh::T, KS = N / 3, NK = 2 * KS + 1;
    const int tt = threadIdx.x & (Sh::TEAM - 1), id = tt & (T - 1), f = tt / T;
    const int j = j0 + f;
    const bool on = j < d.nkx;
    const int jc = on ? j : j0;  // idle lanes repeat the first column and store nothing
    rgv* x = xbuf + f * Sh::STRIDE;
    float2* const col = reinterpret_cast<float2*>(p.M + p.moff[b] + (size_t)jc * N) + id;
    const size_t bo = (size_t)p.boff[b] + (size_t)jc * NK;
    float2* const uh = reinterpret_cast<float2*>(p.uh + bo);
    float2* const rh = reinterpret_cast<float2*>(p.rh + bo);
    cpx<float> v[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const float2 m = col[T * s];
        v[s] = mk<float>(m.x, m.y);
    }
    // the band values the elements need, fetched beside the transform
    float2 us[16], rs[16];
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        if (T * s > KS && T * s + T - 1 < N - KS) continue;
        const int i = id + T * s, k = i < N / 2 ? i : i - N;
        us[s] = rs[s] = make_float2(0.f, 0.f);
        if (k >= -KS && k <= KS) {
            us[s] = uh[k + KS];
            if constexpr (MODE == COL_UPDATE) rs[s] = rh[k + KS];
        }
    }
    const float ins = p.insv[b];
    const float a_lin = p.lin[jc];
    const float w_over_T = (float)p.wT[(size_t)p.par * d.B + b];
    rg_fft<LG, -1>(v, id, x, tw);
    if constexpr (MODE == COL_RESID) {
        const float rq = p.qv[jc];
        ff aJ[16], aL[16];
        constexpr int NA = LG < 7 ? 16 : (128 / T);
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            const int i = id + T * s, k = i < N / 2 ? i : i - N;
            cpx<float> o = mk<float>(0.f, 0.f);
            ColAcc<float> acc;
            const bool fresh = s < NA;
            if (!fresh) {
                acc.J = aJ[s % NA];
                acc.L = aL[s % NA];
            }
            if (!(T * s > KS && T * s + T - 1 < N - KS)) {
                if (k >= -KS && k <= KS) {
                    const cpx<float> ph = scale(v[s], ins);
                    const cpx<float> u = mk<float>(us[s].x, us[s].y);
                    const float bk = -(float)k * w_over_T;  // -omega_k / T
                    const cpx<float> r = symbol_add(a_lin, bk, u, neg(ph));
                    if (on) rh[k + KS] = make_float2(r.x, r.y);
                    acc.add(u, r, k);                       // a6
                    o = mk<float>(-mul_rn(rq, r.y), mul_rn(rq, r.x));  // i q_j r_hat  (a7)
                }
            }
            aJ[s % NA] = acc.J;
            aL[s % NA] = acc.L;
            v[s] = o;
        }
        ff J, L;
        rg_reduce<LG>(aJ, aL, id, reinterpret_cast<ff*>(x), J, L);
        if (on && id == 0) {
            ColAcc<float> acc;
            acc.J = J;
            acc.L = L;
            const double wj = j == 0 ? 1.0 : 2.0;
            p.Jpart[(size_t)b * d.nkx + j] = acc.part_J(wj);
            p.L2part[(size_t)b * d.nkx + j] = acc.part_L(wj);
        }
    } else {
        const float dt = (float)d.dtau, cqj = p.cq[jc], wT2 = w_over_T * w_over_T;
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            cpx<float> o = mk<float>(0.f, 0.f);
            if (!(T * s > KS && T * s + T - 1 < N - KS)) {
                const int i = id + T * s, k = i < N / 2 ? i : i - N;
                if (k >= -KS && k <= KS) {
                    const cpx<float> wh = scale(v[s], ins);
                    const cpx<float> r = mk<float>(rs[s].x, rs[s].y);
                    const float bk = (float)k * w_over_T;
                    // G_hat = (a + i omega/T) r_hat + F[P(u r_x)]                        (a9)
                    const cpx<float> G = symbol_add(a_lin, bk, r, wh);
                    float g = dt;
                    if (d.scheme == 1) g = imex_factor(dt, k, wT2, cqj);                  // (a10)
                    o = step_along(mk<float>(us[s].x, us[s].y), G, g);
                    if (on) uh[k + KS] = make_float2(o.x, o.y);
                }
            }
            v[s] = o;
        }
    }
    rg_fft<LG, +1>(v, id, x, tw);
    if (on) {
#pragma unroll
        for (int s = 0; s < 16; ++s) col[T * s] = make_float2(v[s].x, v[s].y);
    }
}

// Column tiles: F columns of one loop per team, longest loops first.  A loop of 1024 points takes two
// warps, so tiles come in pairs of warps: pair t of a 64-thread half-block takes tiles[t] with both
// warps together or, for shorter loops, two neighbouring tiles (entry b < 0: none).
struct RgCol {
    int b, j0;
};

//
// Three blocks an SM (168 registers, a 48-byte spill in COL_RESID): left at 222 to 231 registers two fit,
// and the 352 blocks of 256 ragged loops or the 344 of eight 256x1024 loops took a second wave for the
// last 40 (120 and 60 steps: 6093 -> 5253 us, 3269 -> 2680 us, ff_add's shorter sum included).  Over 77
// batches that take these kernels the step takes 0.79 to 1.01 of its time with two, below 0.93 where there
// are more than two blocks an SM.
template <int MODE>
__global__ void __launch_bounds__(RG_THREADS, 3) k_rg_cols(Dims d, Bufs<float> p, const RgCol* tiles, int npairs,
                                                        const rgv* tab, int ntab) {
    extern __shared__ __align__(16) unsigned char smem[];
    rgv* tws = reinterpret_cast<rgv*>(smem);
    rgv* xs = tws + ntab;
    grid_trigger();
    for (int i = threadIdx.x; i < ntab; i += RG_THREADS) tws[i] = tab[i];
    __syncthreads();
    grid_wait();
    const int half = threadIdx.x >> 6, w = (threadIdx.x >> 5) & 1;
    for (int it = blockIdx.x * (RG_THREADS / 64) + half; it < npairs; it += gridDim.x * (RG_THREADS / 64)) {
        const bool both = p.lgns[tiles[2 * it].b] == 10;
        const RgCol t = tiles[2 * it + (both ? 0 : w)];
        if (t.b < 0) continue;
        rgv* x = xs + half * (RG_XBYTES / 8) + (both ? 0 : w * (RG_XBYTES / 16));
        if constexpr (MODE == COL_UPDATE) {
            if (p.check_active && p.prec[t.b] != p.myprec) continue;
            if (p.check_active && p.status[t.b] != ST_RUNNING) {
                // a loop frozen before this step carries its period on (a loop that froze in it had
                // that done with its scalars)
                if (t.j0 == 0 && (threadIdx.x & 31) == 0 && !(both && w)) {
                    p.T[(size_t)(p.par ^ 1) * d.B + t.b] = p.T[(size_t)p.par * d.B + t.b];
                    p.wT[(size_t)(p.par ^ 1) * d.B + t.b] = p.wT[(size_t)p.par * d.B + t.b];
                }
                continue;
            }
        } else {
            if (!loop_live(p, t.b)) continue;
        }
        switch (p.lgns[t.b]) {
        case 5: rg_cols<MODE, 5>(d, p, t.b, t.j0, x, tws + rg_at(5)); break;
        case 6: rg_cols<MODE, 6>(d, p, t.b, t.j0, x, tws + rg_at(6)); break;
        case 7: rg_cols<MODE, 7>(d, p, t.b, t.j0, x, tws + rg_at(7)); break;
        case 8: rg_cols<MODE, 8>(d, p, t.b, t.j0, x, tws + rg_at(8)); break;
        case 9: rg_cols<MODE, 9>(d, p, t.b, t.j0, x, tws + rg_at(9)); break;
        default: rg_cols<MODE, 10>(d, p, t.b, t.j0, x, tws + rg_at(10)); break;
        }
    }
}

// the kernels, held by ks_reg.cu: mode ROW_NONLIN or ROW_ADJ and rows of 2^lgnx points; mode COL_RESID or
// COL_UPDATE
using RgRowsFn = void (*)(Dims, Bufs<float>, const RgTile*, int, const rgv*);
using RgColsFn = void (*)(Dims, Bufs<float>, const RgCol*, int, const rgv*, int);
RgRowsFn rg_rows_fn(int mode, int lgnx);
RgColsFn rg_cols_fn(int mode);
#endif  // KS_HOST_EMULATION

}  // namespace ks
