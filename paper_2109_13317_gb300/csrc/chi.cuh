// Correlations and structure factor of FP64 states of the SU(2) and XYZ cores (internal header,
// included by flow.cu after the shared device helpers).  Sec. 3, Eqs. frg:correlation and
// frg:structurefactor; the quadrature is that of k_chi.
//
// k_chi gives every pair (b, j) a block that walks all frequency pairs for one site, reading 8 bytes
// of a 32-byte sector per corner; pairs related by symmetry repeat the same sum.  Here the frequency
// pairs are split over the blocks, whose threads sum whole rows (all irreducible sites and
// components, consecutive lanes), and the last block to finish adds the partial rows in a fixed
// order and maps them onto the pairs.  (-w1, -w2) reads the same corners as (w1, w2) with the sites
// exchanged the same way, as s = w1 + w2 and u = w1 - w2 change their signs together, so half of the
// frequency pairs are taken with doubled weight.  Where |w1| = |w2| one of the two is zero, which
// counts as positive: the pair and its mirror image read one the plain, the other the exchanged entry,
// and the value goes half to each.  k_chi_k had one thread per momentum and a cosine per
// pair: the displacements are merged up to sign (the cosine is even) and a warp shares a momentum.
// Square J1-J2 range 7, 48 frequencies, 64 x 64 momenta (one GB300): k_chi 149 -> 25 us (37
// with a loop over the corners and one group of rows), k_chi_k 110 -> 23 us.  Latency bounds the sum (a chain of
// searches, then the last block), the FP64 pipe's cosines the transform.
#pragma once

namespace chik {

constexpr int kThreads = 128;
constexpr int kMaxBlocks = 256;
constexpr int kPass = 32;      // frequency pairs whose descriptors share a pass

// Doubles of the per-flow scratch: partial rows (plain and exchanged lookups) and on-site values of
// every block.
__host__ __device__ inline size_t part_doubles(int Ns, int nc) { return (size_t)kMaxBlocks * (2 * Ns * nc + nc); }

__host__ __device__ inline int groups(int row) { return row < kThreads ? kThreads / row : 1; }

// Node positions and weights of the correlation quadrature: y[0] = lam, then the mesh points above it;
// W: exact segment weights of G^2 halved between the ends, plus the tail.  Any block size; returns K.
__device__ __forceinline__ int chi_nodes(const Geo& g, const double* __restrict__ w, const double* __restrict__ invh,
                                         const double* __restrict__ gam, double lam, double* y, double* yg, double* W) {
    const int N = g.N;
    int lo = 0, hi = N;   // first mesh point above lam
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (w[m] > lam) hi = m; else lo = m + 1;
    }
    const int K = N - lo + 1;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        y[k] = k == 0 ? lam : w[lo + k - 1];
        yg[k] = y[k] + interp_odd(w, invh, N, gam, y[k]);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        double a = 0.0;
        if (k > 0) a += 0.5 * ((y[k] - y[k - 1]) / (yg[k - 1] * yg[k]));
        if (k + 1 < K) a += 0.5 * ((y[k + 1] - y[k]) / (yg[k] * yg[k + 1]));
        else a += 1.0 / yg[k];
        W[k] = a;
    }
    __syncthreads();
    return K;
}

// chi^{cc}_{b j} of every pair, and S_d = sum over the pairs at +-displacement d of sum_mu chi^{mu mu}.
// counter: zero between launches.  Shared memory: 2 NG Ns NC doubles.
template <int NC>
__global__ void __launch_bounds__(kThreads)
k_chi_sum(Geo g, Tabs tb, const double* __restrict__ w, const double* __restrict__ gam, const double* __restrict__ G, double lam,
          const int2* __restrict__ cmap, const int* __restrict__ onsite, int ntot, int npairs, const int* __restrict__ doff,
          const int* __restrict__ dpair, int nd, double* __restrict__ part, int* __restrict__ counter, double* __restrict__ chi,
          double* __restrict__ Sd) {
    __shared__ double y[kMaxFreq + 1], yg[kMaxFreq + 1], Wn[kMaxFreq + 1];
    __shared__ Desc<double> dsc[kPass], dex[kPass];
    __shared__ bool even[kPass];      // |w1| = |w2|
    __shared__ double on_sum[NC];
    __shared__ int last;
    extern __shared__ double acc[];   // [group][plain, exchanged][c * Ns + r]
    const int tid = threadIdx.x, Ns = g.Ns, row = NC * Ns, NG = groups(row);
    const int K = chi_nodes(g, w, tb.invh, gam, lam, y, yg, Wn);
    for (int e = tid; e < NG * 2 * row; e += kThreads) acc[e] = 0.0;
    double os[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) os[c] = 0.0;
    // frequency pairs (w1 > 0, w2 of either sign) of this block
    const int total = K * 2 * K, per = (total + gridDim.x - 1) / gridDim.x, i0 = blockIdx.x * per, i1 = min(i0 + per, total);
    for (int b0 = i0; b0 < i1; b0 += kPass) {
        const int n = min(kPass, i1 - b0);
        __syncthreads();
        // direct part at (w1 + w2, 0, w1 - w2), exchange part at (w1 + w2, w2 - w1, 0)
        if (tid < 2 * n) {
            const int i = tid < n ? tid : tid - n, idx = b0 + i, p = idx / (2 * K), q = idx - p * 2 * K, qk = q < K ? q : q - K;
            const double xp = y[p], xq = q < K ? y[qk] : -y[qk], W = 2.0 * Wn[p] * Wn[qk];
            Desc<double>& d = tid < n ? dsc[i] : dex[i];
            if (tid < n) {
                make_desc<double, true>(xp + xq, 0.0, xp - xq, 1, 0, tb, g, d, W);
                even[i] = qk == p;
            }
            else make_desc<double, true>(xp + xq, xq - xp, 0.0, 2, 0, tb, g, d, W);
            for (int k = d.n; k < 4; ++k) {   // always four corners: their loads need no loop
                d.off[k] = d.off[0];
                d.wd[k] = d.ws[k] = 0.0;
            }
        }
        __syncthreads();
        // value e of the rows by group gi of the descriptors (rows beyond a block's threads: one group)
        for (int o = tid; o < NG * row; o += kThreads) {
            const int gi = o / row, e = o - gi * row;
            double a = 0.0, x = 0.0;
#pragma unroll 4
            for (int i = gi; i < n; i += NG) {
                const Desc<double>& d = dsc[i];
                const double* wt = e < Ns ? d.wd : d.ws;
                double v = 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) v = fma(wt[k], __ldg(G + d.off[k] + e), v);
                if (even[i]) { a = fma(0.5, v, a); x = fma(0.5, v, x); }
                else if (d.swap) x += v;
                else a += v;
            }
            acc[gi * 2 * row + e] += a;
            acc[(gi * 2 + 1) * row + e] += x;
        }
        if (tid >= kThreads - 32) {   // on-site exchange values (the on-site pair is its own exchange)
            const int i = tid & 31;
            if (i < n)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const double* wt = c == 0 ? dex[i].wd : dex[i].ws;
#pragma unroll
                    for (int k = 0; k < 4; ++k) os[c] = fma(wt[k], __ldg(G + dex[i].off[k] + c * Ns), os[c]);
                }
        }
    }
    __syncthreads();
    if (tid >= kThreads - 32)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            for (int o = 16; o > 0; o >>= 1) os[c] += __shfl_down_sync(0xffffffffu, os[c], o);
            if ((tid & 31) == 0) on_sum[c] = os[c];
        }
    __syncthreads();
    double* mine = part + (size_t)blockIdx.x * (2 * row + NC);
    for (int e = tid; e < 2 * row + NC; e += kThreads) {
        double a = e < 2 * row ? acc[e] : on_sum[e - 2 * row];
        if (e < 2 * row)
            for (int k = 1; k < NG; ++k) a += acc[k * 2 * row + e];
        mine[e] = a;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    // the last block: totals in block order, then every pair
    __threadfence();
    for (int e = tid; e < 2 * row + NC; e += kThreads) {
        double a = 0.0;
#pragma unroll 8
        for (unsigned b = 0; b < gridDim.x; ++b) a += __ldcg(part + (size_t)b * (2 * row + NC) + e);
        if (e < 2 * row) acc[e] = a; else on_sum[e - 2 * row] = a;
    }
    __syncthreads();
    double bub = 0.0;
    for (int k = 0; k < K; ++k) bub += Wn[k];
    bub = bub / (2.0 * kPi);
    for (int o = tid; o < npairs * NC; o += kThreads) {
        const int pi = o / NC, mu = o - pi * NC;
        const int2 pm = cmap[pi];
        const int c = perm_of(pm.y, mu), r = pm.x;
        // plain lookups of the stored entry, and exchanged ones of the entry that it exchanges to
        double F = 4.0 * (acc[c * Ns + r] + acc[row + perm_of(tb.swap_perm[r], c) * Ns + tb.swap_r[r]]);
        const bool on = onsite[pi] != 0;
        if (on) {
            const int2 po = cmap[(pi / ntot) * ntot];
            double e[NC], x;
#pragma unroll
            for (int k = 0; k < NC; ++k) e[k] = on_sum[perm_of(po.y, k)];
            if (NC == 2) x = mu == 0 ? 2.0 * (e[0] + 3.0 * e[1]) : 2.0 * (e[0] - e[1]);
            else {
                x = 0.0;
                for (int k = 0; k < NC; ++k) x += (mu == 0 || k == 0 || k == mu) ? 2.0 * e[k] : -2.0 * e[k];
            }
            F -= x;
        }
        chi[o] = (on ? bub : 0.0) - F / (16.0 * kPi * kPi);
    }
    __syncthreads();
    for (int d = tid; d < nd; d += kThreads) {
        double a = 0.0;
        for (int k = doff[d]; k < doff[d + 1]; ++k) {
            const double* c = chi + (size_t)dpair[k] * NC;
            a += NC == 2 ? 3.0 * c[1] : c[1] + c[2] + c[NC - 1];
        }
        Sd[d] = a;
    }
    if (tid == 0) *counter = 0;
}

// chi(k) = (1/N_b) sum_d cos(k d) S_d, a warp per momentum.
__global__ void __launch_bounds__(kThreads) k_chi_fourier(int nk, const double* __restrict__ kp, const double* __restrict__ dr,
                                                          const double* __restrict__ Sd, int nd, int nb, double* __restrict__ out) {
    const int i = (blockIdx.x * kThreads + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= nk) return;
    const double kx = kp[3 * i], ky = kp[3 * i + 1], kz = kp[3 * i + 2];
    double a = 0.0;
    for (int d = lane; d < nd; d += 32) a = fma(cos(kx * dr[3 * d] + ky * dr[3 * d + 1] + kz * dr[3 * d + 2]), Sd[d], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (lane == 0) out[i] = a / (double)nb;
}

// ---- host side: displacements merged up to sign, and their pairs
struct Displacements {
    std::vector<double> dr;       // nd x 3
    std::vector<int> off, pair;   // nd + 1, npairs
};

inline Displacements merge(const std::vector<double>& chi_dr) {
    const int n = (int)chi_dr.size() / 3;
    std::vector<std::array<long long, 3>> key(n);
    for (int i = 0; i < n; ++i) {
        long long s = 0;
        for (int k = 0; k < 3; ++k) {
            key[i][k] = std::llround(chi_dr[3 * i + k] * 1e8);
            if (s == 0 && key[i][k] != 0) s = key[i][k] > 0 ? 1 : -1;
        }
        if (s < 0)
            for (int k = 0; k < 3; ++k) key[i][k] = -key[i][k];
    }
    Displacements D;
    D.pair.resize(n);
    for (int i = 0; i < n; ++i) D.pair[i] = i;
    std::stable_sort(D.pair.begin(), D.pair.end(), [&](int a, int b) { return key[a] < key[b]; });
    for (int i = 0; i < n; ++i) {
        const int p = D.pair[i];
        if (i == 0 || key[p] != key[D.pair[i - 1]]) {
            D.off.push_back(i);
            for (int k = 0; k < 3; ++k) D.dr.push_back(chi_dr[3 * p + k]);
        }
    }
    D.off.push_back(n);
    return D;
}

}  // namespace chik
