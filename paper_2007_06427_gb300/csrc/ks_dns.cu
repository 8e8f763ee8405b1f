// ks_dns.cu - time integration of the KSE itself, for the initial loops (Sec. 4.3 of the paper).
//
// The paper draws its initial loops from close recurrences of a chaotic solution u(x, t) of
// u_t = -u u_x - u_xx - u_xxxx on [0, L) (Sec. 4.3).  This file integrates that equation on the
// GPU: a Fourier pseudo-spectral discretisation with Nx points, the product dealiased by the 2/3
// rule as in the descent (Sec. 4.2), and fourth-order exponential time differencing (ETDRK4,
// Cox & Matthews, J. Comput. Phys. 176, 2002), whose linear part is the exact diagonal symbol
// q_j^2 - q_j^4.  The phi-function weights are contour averages (Kassam & Trefethen, SIAM
// J. Sci. Comput. 26, 2005) computed in the kernel at launch.  A second kernel cuts a segment
// of a saved trajectory into the Ns instants of a loop by linear interpolation in time.
//
// Layout: one CTA integrates up to DNS_PAIRS_MAX pairs of trajectories for the whole run.  The
// two real fields of a pair share one complex x-transform (u_a + i u_b, and the products
// u_a^2 + i u_b^2); the state of each trajectory is its half spectrum v_j, j = 0..Kx, kept in
// shared memory with the stage values of the scheme.  Global memory is touched at the start
// (u0), at every saved instant (u and ||u||) and at the end.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "ks_items.cuh"
#include "ks_loop.h"

using namespace ks;

void ks_internal_set_error(const char* msg);

namespace {

constexpr int DNS_THREADS = 128;
constexpr int DNS_PAIRS_MAX = 4;
constexpr int DNS_CONTOUR = 32;  // points on the upper half of the contour circle
constexpr int DNS_SPECS = 6;     // v, a, s (stage b then c), Nv, Na, Nb per trajectory
constexpr int DNS_COEFS = 7;     // E, E2, Q, f1, f2, f3, g per x-mode

struct DnsArgs {
    double L, dt;
    int nx, lgnx, kx, nh, batch, pairs;  // pairs per CTA
    int save_every, symmetric;
    long long nsteps, nsave;
    const double* u0;   // [batch][nx]
    double* u_saved;    // [batch][nsave][nx] or null
    double* norms;      // [batch][nsave] or null
    double* u_end;      // [batch][nx] or null
};

// shared-memory plan: twiddles, coefficients, per pair two transform buffers of nx, per
// trajectory DNS_SPECS half spectra of nh values
struct DnsPlan {
    int off_tw, off_coef, off_fft, off_spec, off_red, bytes;
};

__host__ __device__ inline DnsPlan dns_plan(int nx, int nh, int pairs) {
    DnsPlan p;
    int o = 0;
    p.off_tw = o;
    o += nx * (int)sizeof(cpx<double>);
    p.off_coef = o;
    o += DNS_COEFS * nh * (int)sizeof(double);
    o = (o + 15) & ~15;
    p.off_fft = o;
    o += 2 * pairs * nx * (int)sizeof(cpx<double>);
    p.off_spec = o;
    o += 2 * pairs * DNS_SPECS * nh * (int)sizeof(cpx<double>);
    p.off_red = o;
    o += 2 * DNS_PAIRS_MAX * (int)sizeof(double);
    p.bytes = o;
    return p;
}

// complex helpers for the contour averages (double, device)
struct cd {
    double x, y;
};
__device__ __forceinline__ cd cadd(cd a, cd b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cd cmulc(cd a, cd b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ cd cscal(cd a, double s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ cd cdivc(cd a, cd b) {
    const double d = b.x * b.x + b.y * b.y;
    return {(a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d};
}
__device__ __forceinline__ cd cexpc(cd a) {
    double s, c;
    sincos(a.y, &s, &c);
    const double e = exp(a.x);
    return {e * c, e * s};
}

// ETDRK4 weights of x-mode j (Cox & Matthews), z = dt (q^2 - q^4):
//   E = e^z, E2 = e^(z/2), Q = dt (e^(z/2) - 1) / z,
//   f1 = dt (-4 - z + e^z (4 - 3z + z^2)) / z^3, f2 = dt (2 + z + e^z (z - 2)) / z^3,
//   f3 = dt (-4 - 3z - z^2 + e^z (4 - z)) / z^3,
// each evaluated as the mean of the expression over points z + r_k on a circle of radius 1 around
// z (the expressions are entire, so the mean equals the value at z without the cancellation of
// the closed forms near z = 0); for real z the mean over the upper half circle, real part, is the
// mean over the whole circle.  g = -q/2 is the factor of the nonlinear term -(u^2/2)_x.
__device__ void dns_coefficients(double* coef, int nh, double L, double dt) {
    for (int j = threadIdx.x; j < nh; j += blockDim.x) {
        const double q = 2.0 * 3.14159265358979323846 * (double)j / L;
        const double z = dt * (q * q - q * q * q * q);
        cd sQ{0, 0}, s1{0, 0}, s2{0, 0}, s3{0, 0};
        for (int k = 1; k <= DNS_CONTOUR; ++k) {
            double sr, cr;
            sincospi(((double)k - 0.5) / (double)DNS_CONTOUR, &sr, &cr);
            const cd w{z + cr, sr};
            const cd ew = cexpc(w), ew2 = cexpc(cscal(w, 0.5));
            const cd w2 = cmulc(w, w), w3 = cmulc(w2, w);
            sQ = cadd(sQ, cdivc({ew2.x - 1.0, ew2.y}, w));
            // -4 - w + e^w (4 - 3w + w^2)
            const cd a1 = cadd({-4.0 - w.x, -w.y}, cmulc(ew, {4.0 - 3.0 * w.x + w2.x, -3.0 * w.y + w2.y}));
            // 2 + w + e^w (w - 2)
            const cd a2 = cadd({2.0 + w.x, w.y}, cmulc(ew, {w.x - 2.0, w.y}));
            // -4 - 3w - w^2 + e^w (4 - w)
            const cd a3 = cadd({-4.0 - 3.0 * w.x - w2.x, -3.0 * w.y - w2.y}, cmulc(ew, {4.0 - w.x, -w.y}));
            s1 = cadd(s1, cdivc(a1, w3));
            s2 = cadd(s2, cdivc(a2, w3));
            s3 = cadd(s3, cdivc(a3, w3));
        }
        const double im = 1.0 / (double)DNS_CONTOUR;
        coef[0 * nh + j] = exp(z);
        coef[1 * nh + j] = exp(0.5 * z);
        coef[2 * nh + j] = dt * sQ.x * im;
        coef[3 * nh + j] = dt * s1.x * im;
        coef[4 * nh + j] = dt * s2.x * im;
        coef[5 * nh + j] = dt * s3.x * im;
        coef[6 * nh + j] = -0.5 * q;
    }
}

// The x-transforms of the run: transforms of length n = 2^lg in double, radix-2 passes under the
// conventions of fft_batch.  A run is chaotic, so its trajectory after a few hundred time units
// hangs on the rounding of every operation: it keeps this arithmetic, where the descent's double
// transforms are in fixed point.  With the twiddle product fused into the additions (v0 + w v1 as
// four fused multiply-adds, v0 - w v1 as 2 v0 minus that) it costs 3 operations per point and stage.
//
// A run is a chain of dependent passes, and an FP64 warp instruction holds its pipe for 64 clocks
// whatever lanes are active, so a butterfly is shared by two threads, one per component: three
// dependent FP64 instructions a pass where one thread takes six, on twice the warps.  The values
// are the same.
//
// That is where the block has the threads for it (SPLIT). Where a pass has more butterflies, a thread
// takes whole ones: their loads and index arithmetic are shared, and its two chains overlap (us a step
// with one thread a component and a thread a butterfly: 1216 trajectories of 64 modes 33.2 / 26.3, 400 of
// 128 modes 36.9 / 28.9, 64 of 256 modes 40.5 / 31.6).
//
// n butterflies over the block: f(i, c, o) computes component c of the two outputs of butterfly i, which
// go to at(i, 0) and at(i, 1); extra(i, c, o) sees them before.
template <bool SPLIT, typename F, typename A, typename E>
__device__ __forceinline__ void dns_each(int n, F f, A at, E extra) {
    for (int t = threadIdx.x; t < (SPLIT ? 2 * n : n); t += blockDim.x) {
        if constexpr (SPLIT) {
            double o[2];
            f(t >> 1, t & 1, o);
            extra(t >> 1, t & 1, o);
            reinterpret_cast<double*>(at(t >> 1, 0))[t & 1] = o[0];
            reinterpret_cast<double*>(at(t >> 1, 1))[t & 1] = o[1];
        } else {
            double o[2], q[2];
            f(t, 0, o);
            f(t, 1, q);
            extra(t, 0, o);
            extra(t, 1, q);
            *at(t, 0) = mk<double>(o[0], q[0]);
            *at(t, 1) = mk<double>(o[1], q[1]);
        }
    }
}

// One component of a butterfly's outputs (c = 0 real, 1 imaginary).
__device__ __forceinline__ void dns_bfly(cpx<double> v0, cpx<double> v1, cpx<double> w, int c, double& o0,
                                         double& o1) {
    const double z = c ? v0.y : v0.x, a = c ? v1.y : v1.x, b = c ? v1.x : v1.y, s = c ? w.y : -w.y;
    o0 = fma(w.x, a, fma(s, b, z));
    o1 = fma(2.0, z, -o0);
}

// Passes first <= span < last of cnt transforms at a (b scratch); returns where the data is.
template <bool SPLIT>
__device__ __forceinline__ cpx<double>* dns_passes(cpx<double>* a, cpx<double>* b, int lg, int cnt, int dir,
                                                   const cpx<double>* tw, int twsh, int first, int last) {
    const int n = 1 << lg, nb = n >> 1;
    for (int span = first; span < last; span <<= 1) {
        const int tu = NMAX / (span * 2);
        dns_each<SPLIT>(
            cnt << (lg - 1),
            [&](int i, int c, double (&o)[2]) {
                const int f = i >> (lg - 1), j = i & (nb - 1);
                const cpx<double>* s = a + (f << lg);
                if (span > 1) {
                    dns_bfly(s[j], s[j + nb], twid<double, true>(tw, (j & (span - 1)) * tu, dir, twsh), c, o[0], o[1]);
                } else {
                    const double v0 = reinterpret_cast<const double*>(s + j)[c];
                    const double v1 = reinterpret_cast<const double*>(s + j + nb)[c];
                    o[0] = v0 + v1;
                    o[1] = v0 - v1;
                }
            },
            [&](int i, int q) {
                const int f = i >> (lg - 1), j = i & (nb - 1), jm = j & (span - 1);
                return b + (f << lg) + ((j - jm) << 1) + jm + (q ? span : 0);
            },
            [](int, int, double (&)[2]) {});
        __syncthreads();
        cpx<double>* t = a;
        a = b;
        b = t;
    }
    return a;
}

// spectrum `which` of trajectory t (t = 2 * pair + member) in the CTA's spectra block
__device__ __forceinline__ cpx<double>* spec(cpx<double>* base, int nh, int t, int which) {
    return base + ((size_t)t * DNS_SPECS + which) * nh;
}

enum { SV = 0, SA = 1, SS = 2, SNV = 3, SNA = 4, SNB = 5 };

// Sum of y over the nx points of each trajectory of the CTA (component 0: member a, 1: b),
// warp w reduces trajectories w, w + warps, ...; fixed order for a given nx.
__device__ void dns_norms(const cpx<double>* Y, int nx, int ntraj, double* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int t = w; t < ntraj; t += nw) {
        const cpx<double>* y = Y + (size_t)(t >> 1) * nx;
        double s = 0.0;
        for (int m = lane; m < nx; m += 32) s += (t & 1) ? y[m].y : y[m].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[t] = s;
    }
}

// One evaluation for every trajectory of the CTA: the grid field of spectrum `src` (inverse
// x-transform of the pair u_a + i u_b), optionally saved, and, unless `end`, the nonlinear term
// N_j = -(i q_j / 2) F[u^2]_j on the retained modes (forward transform of the pair u_a^2 + i u_b^2,
// split into the two members), handed to use(t, j, c, N): component c of mode j of trajectory t.
// The first pass forms the pair's spectrum as it reads it, the last inverse pass squares what it
// writes, so that neither takes a round trip of its own.
template <bool SPLIT, typename Use>
__device__ __forceinline__ void dns_eval(const DnsArgs& a, int tr0, int ntraj, cpx<double>* fftb,
                                         cpx<double>* specs, const cpx<double>* tw, const double* coef,
                                         double* red, int src, long long isave, bool end, Use use) {
    const int nx = a.nx, lgnx = a.lgnx, kx = a.kx, nh = a.nh;
    const int np = (ntraj + 1) >> 1, nb = nx >> 1;
    const int twsh = LGNMAX - lgnx;
    cpx<double>* A = fftb;
    cpx<double>* Bf = fftb + (size_t)a.pairs * nx;
    dns_each<SPLIT>(
        np * nb,
        [&](int i, int c, double (&o)[2]) {
            const int pr = i >> (lgnx - 1), j = i & (nb - 1);
            const int ta = 2 * pr, tb = ta + 1;
            const bool hb = tb < ntraj;
            const double* sa = reinterpret_cast<const double*>(spec(specs, nh, ta, src));
            const double* sb = reinterpret_cast<const double*>(spec(specs, nh, tb, src));
            auto z = [&](int J) {  // component c of v_a + i v_b, or of conj v_a + i conj v_b
                if (J <= kx) {
                    const double x = sa[2 * J + c], y = hb ? sb[2 * J + 1 - c] : 0.0;
                    return c ? x + y : x - y;
                }
                if (J >= nx - kx) {
                    const double x = sa[2 * (nx - J) + c], y = hb ? sb[2 * (nx - J) + 1 - c] : 0.0;
                    return c ? -x + y : x + y;
                }
                return 0.0;
            };
            const double v0 = z(j), v1 = z(j + nb);
            o[0] = v0 + v1;
            o[1] = v0 - v1;
        },
        [&](int i, int q) { return A + 2 * i + q; }, [](int, int, double (&)[2]) {});
    __syncthreads();
    cpx<double>* Z = dns_passes<SPLIT>(A, Bf, lgnx, np, +1, tw, twsh, 2, nb);
    cpx<double>* Y = Z == A ? Bf : A;
    const double inx = 1.0 / (double)nx;  // exact: nx is a power of two
    const bool save = isave >= 0;
    dns_each<SPLIT>(  // the pass of span nb
        np * nb,
        [&](int i, int c, double (&o)[2]) {
            const int pr = i >> (lgnx - 1), j = i & (nb - 1);
            dns_bfly(Z[(pr << lgnx) + j], Z[(pr << lgnx) + j + nb],
                     twid<double, true>(tw, j * (NMAX / nx), +1, twsh), c, o[0], o[1]);
        },
        [&](int i, int q) { return Y + ((i >> (lgnx - 1)) << lgnx) + (i & (nb - 1)) + (q ? nb : 0); },
        [&](int i, int c, double (&o)[2]) {
            const int pr = i >> (lgnx - 1), j = i & (nb - 1), t = 2 * pr + c;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int m = j + q * nb;
                const double u = o[q] * inx;
                o[q] = u * u;
                if (save && a.u_saved && t < ntraj) a.u_saved[((size_t)(tr0 + t) * a.nsave + isave) * nx + m] = u;
                if (end && a.u_end && t < ntraj) a.u_end[(size_t)(tr0 + t) * nx + m] = u;
            }
        });
    __syncthreads();
    if (save && a.norms) {
        dns_norms(Y, nx, ntraj, red);
        __syncthreads();
        if ((int)threadIdx.x < ntraj)
            a.norms[(size_t)(tr0 + threadIdx.x) * a.nsave + isave] = sqrt(a.L * red[threadIdx.x] * inx);
    }
    if (end) return;
    const cpx<double>* F = dns_passes<SPLIT>(Y, Z, lgnx, np, -1, tw, twsh, 1, nx);
    const double* g = coef + 6 * nh;
    auto give = [&](int t, int j, int c) {
        const cpx<double> P = F[((t >> 1) << lgnx) + j], Q = F[((t >> 1) << lgnx) + ((nx - j) & (nx - 1))];
        // W_a = (P + conj Q) / 2, W_b = (P - conj Q) / (2 i); N = i g W
        const double h = (c ^ (t & 1)) ? P.x : P.y, k = (c ^ (t & 1)) ? Q.x : Q.y;
        // a: W.x = (P.x + Q.x) / 2, W.y = (P.y - Q.y) / 2; b: W.x = (P.y + Q.y) / 2, W.y = -(P.x - Q.x) / 2
        const double W = c ? 0.5 * (h + k) : ((t & 1) ? -0.5 : 0.5) * (h - k);
        use(t, j, c, (c ? g[j] : -g[j]) * W);
    };
    for (int i = threadIdx.x; i < ntraj * nh * (SPLIT ? 2 : 1); i += blockDim.x) {
        const int tj = SPLIT ? i >> 1 : i, t = tj / nh, j = tj - t * nh;
        if constexpr (SPLIT) {
            give(t, j, i & 1);
        } else {
            give(t, j, 0);
            give(t, j, 1);
        }
    }
    __syncthreads();
}

template <bool SPLIT>
__global__ void __launch_bounds__(DNS_THREADS) k_dns(DnsArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const DnsPlan pl = dns_plan(a.nx, a.nh, a.pairs);
    cpx<double>* tw = reinterpret_cast<cpx<double>*>(smem + pl.off_tw);
    double* coef = reinterpret_cast<double*>(smem + pl.off_coef);
    cpx<double>* fftb = reinterpret_cast<cpx<double>*>(smem + pl.off_fft);
    cpx<double>* specs = reinterpret_cast<cpx<double>*>(smem + pl.off_spec);
    double* red = reinterpret_cast<double*>(smem + pl.off_red);
    const int nx = a.nx, lgnx = a.lgnx, nh = a.nh;
    const int tr0 = blockIdx.x * 2 * a.pairs;
    const int ntraj = min(2 * a.pairs, a.batch - tr0);
    if (ntraj <= 0) return;
    const int np = (ntraj + 1) >> 1;
    const int twsh = LGNMAX - lgnx;

    // twiddles e^(2 pi i t / nx) at their swizzled slots of a compact table (see tw_swz)
    for (int t = threadIdx.x; t < nx; t += blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)t / (double)nx, &s, &c);
        tw[tw_swz<double>(t)] = mk<double>(c, s);
    }
    dns_coefficients(coef, nh, a.L, a.dt);
    // analysis of u0: forward transform of the pairs, split, truncated to |j| <= Kx
    cpx<double>* A = fftb;
    cpx<double>* Bf = fftb + (size_t)a.pairs * nx;
    for (int i = threadIdx.x; i < np * nx; i += blockDim.x) {
        const int pr = i >> lgnx, m = i & (nx - 1);
        const double ua = a.u0[(size_t)(tr0 + 2 * pr) * nx + m];
        const double ub = (2 * pr + 1 < ntraj) ? a.u0[(size_t)(tr0 + 2 * pr + 1) * nx + m] : 0.0;
        A[i] = mk<double>(ua, ub);
    }
    __syncthreads();
    {
        cpx<double>* F = dns_passes<SPLIT>(A, Bf, lgnx, np, -1, tw, twsh, 1, nx);
        for (int i = threadIdx.x; i < np * nh; i += blockDim.x) {
            const int pr = i / nh, j = i - pr * nh;
            const cpx<double> P = F[(size_t)pr * nx + j];
            const cpx<double> Pm = conj(F[(size_t)pr * nx + ((nx - j) & (nx - 1))]);
            const cpx<double> sm = P + Pm, df = P - Pm;
            cpx<double> va = mk<double>(0.5 * sm.x, 0.5 * sm.y);
            cpx<double> vb = mk<double>(0.5 * df.y, -0.5 * df.x);
            if (a.symmetric) {
                va.x = 0.0;
                vb.x = 0.0;
            }
            spec(specs, nh, 2 * pr, SV)[j] = va;
            if (2 * pr + 1 < ntraj) spec(specs, nh, 2 * pr + 1, SV)[j] = vb;
        }
        __syncthreads();
    }

    const double* E = coef;
    const double* E2 = coef + nh;
    const double* Q = coef + 2 * nh;
    const double* f1 = coef + 3 * nh;
    const double* f2 = coef + 4 * nh;
    const double* f3 = coef + 5 * nh;
    auto at = [&](int t, int which, int j, int c) -> double& {
        return reinterpret_cast<double*>(spec(specs, nh, t, which) + j)[c];
    };
    for (long long n = 0; n < a.nsteps; ++n) {
        const long long isave = (n % a.save_every == 0) ? n / a.save_every : -1;
        dns_eval<SPLIT>(a, tr0, ntraj, fftb, specs, tw, coef, red, SV, isave, false, [&](int t, int j, int c, double N) {
            at(t, SNV, j, c) = N;
            at(t, SA, j, c) = E2[j] * at(t, SV, j, c) + Q[j] * N;  // a = E2 v + Q Nv
        });
        dns_eval<SPLIT>(a, tr0, ntraj, fftb, specs, tw, coef, red, SA, -1, false, [&](int t, int j, int c, double N) {
            at(t, SNA, j, c) = N;
            at(t, SS, j, c) = E2[j] * at(t, SV, j, c) + Q[j] * N;  // b = E2 v + Q Na
        });
        dns_eval<SPLIT>(a, tr0, ntraj, fftb, specs, tw, coef, red, SS, -1, false, [&](int t, int j, int c, double N) {
            at(t, SNB, j, c) = N;
            const double d2 = 2.0 * N - at(t, SNV, j, c);          // c = E2 a + Q (2 Nb - Nv)
            at(t, SS, j, c) = E2[j] * at(t, SA, j, c) + Q[j] * d2;
        });
        // v' = E v + f1 Nv + 2 f2 (Na + Nb) + f3 Nc; in the subspace the real parts are zeroed
        dns_eval<SPLIT>(a, tr0, ntraj, fftb, specs, tw, coef, red, SS, -1, false, [&](int t, int j, int c, double N) {
            const double w2 = 2.0 * f2[j];
            const double v = at(t, SV, j, c), Nv = at(t, SNV, j, c), Na = at(t, SNA, j, c), Nb = at(t, SNB, j, c);
            const double vn = E[j] * v + f1[j] * Nv + w2 * (Na + Nb) + f3[j] * N;
            at(t, SV, j, c) = a.symmetric && c == 0 ? 0.0 : vn;
        });
    }
    const bool save_last = (a.nsteps % a.save_every == 0);
    if (save_last || a.u_end)
        dns_eval<SPLIT>(a, tr0, ntraj, fftb, specs, tw, coef, red, SV, save_last ? a.nsteps / a.save_every : -1, true,
                 [](int, int, int, double) {});
}

// Loop l of a segment cut: field at instants t_a + T_l n / Ns_l (n = 0..Ns_l - 1) by linear
// interpolation between the saved samples (sample i at time i * dts), written to the loop's
// ragged-packed slot [n][m] at out + off_l.
__global__ void k_dns_segment(const double* us, int nx, double dts, const int* a_idx, const double* T,
                              const int* ns, const long long* off, double* out) {
    const int l = blockIdx.x;
    const int nsl = ns[l], a0 = a_idx[l];
    const double Tl = T[l];
    for (int i = threadIdx.x; i < nsl * nx; i += blockDim.x) {
        const int n = i / nx, m = i - n * nx;
        const double x = (Tl * (double)n / (double)nsl) / dts;  // position in samples after a0
        int i0 = (int)floor(x);
        if (i0 < 0) i0 = 0;
        const double f = x - (double)i0;
        const double y0 = us[(size_t)(a0 + i0) * nx + m];
        const double y1 = us[(size_t)(a0 + i0 + 1) * nx + m];
        out[off[l] + i] = y0 + f * (y1 - y0);
    }
}

int dns_fail(int code, const std::string& msg) {
    ks_internal_set_error(msg.c_str());
    return code;
}

bool dns_is_device(const void* p) {
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// A caller buffer as a device pointer: the buffer itself, or a temporary device copy (filled
// from the host when `in`), released and copied back by finish().
struct Staged {
    void* user = nullptr;
    void* dev = nullptr;
    size_t bytes = 0;
    bool temp = false;
    bool out = false;
    int stage(void* p, size_t n, bool in, bool is_out, cudaStream_t s) {
        user = p;
        bytes = n;
        out = is_out;
        if (!p || n == 0) return KS_OK;
        if (dns_is_device(p)) {
            dev = p;
            return KS_OK;
        }
        if (cudaMalloc(&dev, n) != cudaSuccess) {
            cudaGetLastError();
            dev = nullptr;
            return dns_fail(KS_ERR_OOM, "device allocation for a host buffer failed");
        }
        temp = true;
        if (in && cudaMemcpyAsync(dev, p, n, cudaMemcpyHostToDevice, s) != cudaSuccess)
            return dns_fail(KS_ERR_CUDA, "host to device copy failed");
        return KS_OK;
    }
    int finish(cudaStream_t s) {
        if (!temp) return KS_OK;
        int rc = KS_OK;
        if (out && cudaMemcpyAsync(user, dev, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess)
            rc = dns_fail(KS_ERR_CUDA, "device to host copy failed");
        if (cudaStreamSynchronize(s) != cudaSuccess && rc == KS_OK)
            rc = dns_fail(KS_ERR_CUDA, "stream synchronisation failed");
        cudaFree(dev);
        temp = false;
        return rc;
    }
    ~Staged() {
        if (temp) cudaFree(dev);
    }
};

int ilog2i(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

}  // namespace

extern "C" int ks_dns(double L, int nx, int batch, double dt, long long nsteps, int save_every,
                      int symmetric, const double* u0, double* u_saved, double* norms, double* u_end,
                      void* stream) {
    ks_internal_set_error("");
    if (!(L > 0.0) || !std::isfinite(L)) return dns_fail(KS_ERR_ARG, "L must be finite and > 0");
    if (!(dt > 0.0) || !std::isfinite(dt)) return dns_fail(KS_ERR_ARG, "dt must be finite and > 0");
    if (nx < 8 || nx > NMAX || (nx & (nx - 1))) return dns_fail(KS_ERR_ARG, "nx must be a power of two in [8, 1024]");
    if (batch < 1) return dns_fail(KS_ERR_ARG, "batch must be >= 1");
    if (nsteps < 0) return dns_fail(KS_ERR_ARG, "nsteps must be >= 0");
    if (save_every < 1) return dns_fail(KS_ERR_ARG, "save_every must be >= 1");
    if (!u0) return dns_fail(KS_ERR_ARG, "u0 is required");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        return dns_fail(KS_ERR_CUDA, "no usable CUDA device");
    }
    cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    DnsArgs a{};
    a.L = L;
    a.dt = dt;
    a.nx = nx;
    a.lgnx = ilog2i(nx);
    a.kx = nx / 3;
    a.nh = a.kx + 1;
    a.batch = batch;
    a.save_every = save_every;
    a.symmetric = symmetric ? 1 : 0;
    a.nsteps = nsteps;
    a.nsave = nsteps / save_every + 1;
    // pairs per CTA: no more than spread the batch over the SMs (a pass is a chain of dependent
    // instructions, whatever the pairs; 64 trajectories of 64 modes: 25.9 us a step on 8 CTAs), than
    // give the block's threads two butterfly components each, or than fit its shared memory
    int pairs = std::max(1, std::min(DNS_PAIRS_MAX, (2 * DNS_THREADS) / nx));
    while (pairs > 1 && dns_plan(nx, a.nh, pairs).bytes > 200 * 1024) --pairs;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return dns_fail(KS_ERR_CUDA, "no usable CUDA device");
    }
    const int npairs = (batch + 1) / 2;
    pairs = std::min(pairs, (npairs + sms - 1) / sms);
    a.pairs = pairs;
    const DnsPlan pl = dns_plan(nx, a.nh, pairs);
    if (pl.bytes > 227 * 1024) return dns_fail(KS_ERR_ARG, "nx too large for the shared-memory plan");
    const size_t fb = (size_t)batch * nx * sizeof(double);
    Staged su0, ssv, snm, sue;
    int rc = su0.stage(const_cast<double*>(u0), fb, true, false, s);
    if (rc == KS_OK) rc = ssv.stage(u_saved, fb * (size_t)a.nsave, false, true, s);
    if (rc == KS_OK) rc = snm.stage(norms, (size_t)batch * a.nsave * sizeof(double), false, true, s);
    if (rc == KS_OK) rc = sue.stage(u_end, fb, false, true, s);
    if (rc != KS_OK) return rc;
    a.u0 = static_cast<const double*>(su0.dev);
    a.u_saved = static_cast<double*>(ssv.dev);
    a.norms = static_cast<double*>(snm.dev);
    a.u_end = static_cast<double*>(sue.dev);
    // a thread per butterfly component where the block has one for each
    auto* const kern = pairs * nx <= DNS_THREADS ? k_dns<true> : k_dns<false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, pl.bytes) != cudaSuccess) {
        cudaGetLastError();
        return dns_fail(KS_ERR_CUDA, "shared-memory attribute of the DNS kernel failed");
    }
    const int grid = (batch + 2 * pairs - 1) / (2 * pairs);
    kern<<<grid, DNS_THREADS, pl.bytes, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return dns_fail(KS_ERR_CUDA, cudaGetErrorString(e));
    rc = su0.finish(s);
    int r2 = ssv.finish(s), r3 = snm.finish(s), r4 = sue.finish(s);
    if (rc == KS_OK) rc = r2;
    if (rc == KS_OK) rc = r3;
    if (rc == KS_OK) rc = r4;
    return rc;
}

extern "C" int ks_dns_segments(int nx, long long nsave, double dts, const double* us, int nloops,
                               const int* a_idx, const double* T, const int* ns, double* out,
                               void* stream) {
    ks_internal_set_error("");
    if (nx < 1 || nsave < 2 || !(dts > 0.0) || !std::isfinite(dts))
        return dns_fail(KS_ERR_ARG, "nx >= 1, nsave >= 2 and a finite dts > 0 are required");
    if (nloops < 0) return dns_fail(KS_ERR_ARG, "nloops must be >= 0");
    if (nloops == 0) return KS_OK;
    if (!us || !a_idx || !T || !ns || !out) return dns_fail(KS_ERR_ARG, "null pointer");
    // the per-loop tables are read here on the host
    if (dns_is_device(a_idx) || dns_is_device(T) || dns_is_device(ns))
        return dns_fail(KS_ERR_ARG, "a_idx, T and ns must be host arrays");
    std::vector<long long> off(nloops);
    long long tot = 0;
    for (int l = 0; l < nloops; ++l) {
        if (ns[l] < 1) return dns_fail(KS_ERR_ARG, "every Ns must be >= 1");
        if (!(T[l] > 0.0) || !std::isfinite(T[l])) return dns_fail(KS_ERR_ARG, "every T must be finite and > 0");
        // the last instant, a + T (Ns - 1) / Ns, and its right-hand sample must be saved
        const double last = T[l] * (double)(ns[l] - 1) / (double)ns[l] / dts;
        if (a_idx[l] < 0 || (double)a_idx[l] + std::floor(last) + 1.0 > (double)(nsave - 1))
            return dns_fail(KS_ERR_ARG, "a segment runs past the saved samples");
        off[l] = tot;
        tot += (long long)ns[l] * nx;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        return dns_fail(KS_ERR_CUDA, "no usable CUDA device");
    }
    cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    Staged sus, sout, sa, sT, sn, so;
    int rc = sus.stage(const_cast<double*>(us), (size_t)nsave * nx * sizeof(double), true, false, s);
    if (rc == KS_OK) rc = sout.stage(out, (size_t)tot * sizeof(double), false, true, s);
    // the per-loop tables always travel through a temporary device copy
    if (rc == KS_OK) rc = sa.stage(const_cast<int*>(a_idx), nloops * sizeof(int), true, false, s);
    if (rc == KS_OK) rc = sT.stage(const_cast<double*>(T), nloops * sizeof(double), true, false, s);
    if (rc == KS_OK) rc = sn.stage(const_cast<int*>(ns), nloops * sizeof(int), true, false, s);
    if (rc == KS_OK) rc = so.stage(off.data(), nloops * sizeof(long long), true, false, s);
    if (rc != KS_OK) return rc;
    k_dns_segment<<<nloops, 256, 0, s>>>(static_cast<const double*>(sus.dev), nx, dts,
                                         static_cast<const int*>(sa.dev), static_cast<const double*>(sT.dev),
                                         static_cast<const int*>(sn.dev), static_cast<const long long*>(so.dev),
                                         static_cast<double*>(sout.dev));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return dns_fail(KS_ERR_CUDA, cudaGetErrorString(e));
    rc = sus.finish(s);
    int r2 = sout.finish(s);
    int r3 = sa.finish(s), r4 = sT.finish(s), r5 = sn.finish(s), r6 = so.finish(s);
    for (int r : {r2, r3, r4, r5, r6})
        if (rc == KS_OK) rc = r;
    return rc;
}
