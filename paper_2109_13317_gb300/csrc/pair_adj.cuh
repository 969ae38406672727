// Reverse-mode vertex flow of the SU(2) and XYZ cores on the packed state (internal header, included
// by flow.cu after pair.cuh and adjoint.cuh): the vector-Jacobian product of k_gamma_rhs_pair's
// arithmetic, in place of k_gamma_adj where the tables fit.
//
// k_gamma_adj was bound by the FP64 pipe (86 % busy), most of it work beside the flow equations: the
// products and their derivatives component by component, and compare-and-swap loops of double
// additions in shared memory.  Here
//   * s and u channels keep a site's components in the registers of one thread: with the output's
//     adjoint o (constants of the thread) the row adjoints are W O(o) B and W O(o) A, O the symmetric
//     matrix of the component products of pair.cuh, and the weight adjoint is A O(o) B;
//   * the on-site factors' adjoints are summed once per node and component instead of by atomic
//     additions from every site;
//   * the adjoint of a node weight is summed from shared memory in a fixed order;
//   * the transposed lookups of all channels add to accumulators in the layout of the t rows (and the
//     same of the exchanged pairs), so lanes add to consecutive addresses; k_pair_fold maps them onto
//     the state.  (FP64 rows of both layouts have the same stride, so a packed offset serves both.)
// Heisenberg-Kitaev, range 5, 32 frequencies (one GB300, a step's adjoint): 15.9 -> 9.4 ms, bound by the
// FP64 pipe: 8 + 8 operations per value and node for the interpolation and its transpose, 2 x 16 per
// site and node for the products, two per product and node for the lattice sum.  Lists sorted by length
// (a warp runs as long as its longest): 10.9 -> 10.0 ms at that stage; registers capped for six CTAs
// instead of four: 10.0 -> 9.8; one accumulator layout for all channels: 9.9 -> 9.4.
#pragma once

namespace pairk {

struct AdjTab {
    const int* out_off;   // nprod + 1: outputs of every product
    const int* out_idx;   // c * Ns + r
    const int2* list;     // [entry][slot]: (product, offset of the other row's value)
    const int2* items;    // slot: (item, entries); items are the row A values c * Ns + r, then the row B
                          // values, in order of falling length, so that the lanes of a warp end together
};

constexpr int kAN = 64;   // nodes whose descriptors share a pass
constexpr int kAQ = 8;    // t-channel nodes per block of rows

template <int NC>
__host__ __device__ inline size_t adj_smem(int N, int Ns, int nst, int nprod) {
    const int CH = units<double, NC>(Ns), rt = NC * nst;
    const size_t su = (2 * 16 + 2 * 32 + 8) * (size_t)kAN + sizeof(double) * kAN * CH;
    const size_t t = (4 * 48 + 8) * (size_t)kAN + sizeof(double) * (kAQ * 2 * rt + kAQ * 4 * NC + kAQ * 2 * NC * Ns);
    return r16(sizeof(double) * 2 * N) + r16(sizeof(double) * NC * Ns) + r16(sizeof(double) * nprod) + (su > t ? su : t) + 64;
}

// t = O(f) v: derivative of f . product(a, v) with respect to a (and, O being symmetric, the same for
// the other row) of the s (S_CH) or u channel.
template <bool S_CH, int NC>
__device__ __forceinline__ void product_adjoint(const double* f, const double* v, double* t) {
    if constexpr (NC == 2) {
        t[0] = fma(f[0], v[0], f[1] * v[1]);
        t[1] = fma(f[1], v[0], fma(3.0, f[0], S_CH ? -2.0 * f[1] : 2.0 * f[1]) * v[1]);
    } else {
        t[0] = fma(f[0], v[0], fma(f[1], v[1], fma(f[2], v[2], f[3] * v[3])));
#pragma unroll
        for (int c = 1; c < 4; ++c) {
            const int e = c % 3 + 1, g = e % 3 + 1;
            t[c] = fma(f[0], v[c], f[c] * v[0]);
            t[c] = fma(S_CH ? -f[e] : f[e], v[g], fma(S_CH ? -f[g] : f[g], v[e], t[c]));
        }
    }
}

// Transposed lookup of a unit: corner weights w (density signs in the offsets), values t, component
// rows nst apart.
template <int NC>
__device__ __forceinline__ void red_unit(double* q, const int4 o, const double* wt, const double* t, int nst) {
    double w[4];
    lds_w(wt, w);
    const int of[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if ((__double_as_longlong(w[k]) & 0x7fffffffffffffffLL) == 0) continue;   // w == 0 (uniform in a group)
        double* p = q + (long)(of[k] & ~kNeg) * 2;
#pragma unroll
        for (int c = 0; c < NC; ++c) atomicAdd(p + c * nst, (c == 0 ? flip_sign(w[k], of[k]) : w[k]) * t[c]);
    }
}

// Abar += (d dGamma / d Gamma)^T fbar in the layout of the t rows, Wbar += d dGamma / d W . fbar; one CTA per
// stored triple.
template <int NC>
__global__ void __launch_bounds__(128, 6)
k_gamma_adj_pair(Geo g, Tabs tb, Tab td, AdjTab at, const double* __restrict__ P, const double* __restrict__ nx,
                 const double* __restrict__ nW, const int* __restrict__ ncount, const double* __restrict__ fbar,
                 double* __restrict__ Pbar, double* __restrict__ Wbar) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, nth = blockDim.x, N = g.N, Ns = g.Ns, rc = td.rv / 2, nst = td.nst, rt = NC * nst;
    const int row = NC * Ns;
    double* wm = reinterpret_cast<double*>(smem);
    double* ih = wm + N;
    double* ob = reinterpret_cast<double*>(smem + r16(sizeof(double) * 2 * N));   // fbar of the triple, c * Ns + r
    double* pbar = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(ob) + r16(sizeof(double) * row));
    unsigned char* work = reinterpret_cast<unsigned char*>(pbar) + r16(sizeof(double) * td.nprod);
    const int ti = blockIdx.x % N, p = blockIdx.x / N;
    int si = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((si + 1) * (si + 2) / 2 <= p) ++si;
    while (si * (si + 1) / 2 > p) --si;
    const int ui = p - si * (si + 1) / 2;
    for (int i = tid; i < N; i += nth) { wm[i] = tb.w[i]; ih[i] = i + 1 < N ? tb.invh[i] : 0.0; }
    for (int e = tid; e < row; e += nth) ob[e] = fbar[(size_t)(p * N + ti) * row + e];
    __syncthreads();
    // out = ... - 2 sum of products: adjoint of every product's node integral
    for (int o = tid; o < td.nprod; o += nth) {
        double a = 0.0;
        for (int k = at.out_off[o]; k < at.out_off[o + 1]; ++k) a += ob[at.out_idx[k]];
        pbar[o] = -2.0 * a;
    }
    const double s = wm[si], t = wm[ti], u = wm[ui];
    const double w1p = (s + t + u) * 0.5, w2p = (s - t - u) * 0.5, w1 = (s - t + u) * 0.5, w2 = (s + t - u) * 0.5;

    // ---- s and u channels: thread (site, node group)
    {
        const int CH = units<double, NC>(Ns), NG = nth / CH, my_g = tid / CH, my_c = tid - my_g * CH;
        int4* offs = reinterpret_cast<int4*>(work);                                 // [row][node]
        double* wts = reinterpret_cast<double*>(work + 2 * 16 * kAN);               // [row][node][corner]
        double* Wq = wts + 2 * 4 * kAN;                                             // [node]
        double* z = Wq + kAN;                                                       // [node][site]: A O(o) B
        double o[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) o[c] = my_g < NG ? ob[c * Ns + my_c] : 0.0;
        auto channel = [&](auto s_channel) {
            constexpr bool is_s = decltype(s_channel)::value;
            const int cidx = is_s ? si : 2 * N + ui, nq = ncount[cidx];
            for (int n0 = 0; n0 < nq; n0 += kAN) {
                const int nn = min(kAN, nq - n0);
                __syncthreads();
                for (int idx = tid; idx < 2 * nn; idx += nth) {
                    const int r = idx >= nn ? 1 : 0, i = idx - r * nn;
                    const double x = nx[(size_t)cidx * g.nmax + n0 + i];
                    if (r == 0) Wq[i] = nW[(size_t)cidx * g.nmax + n0 + i];
                    const double y0 = r ? (is_s ? x - w1 : w1p + x) : (is_s ? w1p - x : w1 + x);
                    const double y1 = r ? (is_s ? x - w2 : w2 - x) : x - w2p;
                    const double m0 = mag(y0), m1 = mag(y1);
                    const auto c0 = axis_of(wm, ih, g, m0), c1 = axis_of(wm, ih, g, m1);
                    const bool swap = is_s ? is_neg(y1) : is_neg(y0);
                    const int so = swap ? td.ex_su : 0;
                    const bool flip = is_s ? less(s, m1) : less(m0, u);
                    int off[4];
                    double wt[4];
                    bool neg[4];
                    corners<false>(is_s ? 0 : 2, c0, c1, is_s ? si : ui, flip, N, rc, off, wt, neg);
#pragma unroll
                    for (int k = 0; k < 4; ++k) off[k] += so + (neg[k] ? kNeg : 0);
                    offs[r * kAN + i] = make_int4(off[0], off[1], off[2], off[3]);
                    st_w(wts + 4 * (r * kAN + i), wt);
                }
                __syncthreads();
                if (my_g < NG)
                    for (int i = my_g; i < nn; i += NG) {
                        double a[NC], b[NC], ta[NC], tb_[NC];
                        const int4 oa = offs[i], obb = offs[kAN + i];
                        interp_unit<double, NC>(P + NC * my_c, oa, wts + 4 * i, 0, a);
                        interp_unit<double, NC>(P + NC * my_c, obb, wts + 4 * (kAN + i), 0, b);
                        product_adjoint<is_s, NC>(o, b, ta);
                        product_adjoint<is_s, NC>(o, a, tb_);
                        const double W = Wq[i];
                        double zz = 0.0;
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            zz = fma(a[c], ta[c], zz);
                            ta[c] *= W;
                            tb_[c] *= W;
                        }
                        z[i * CH + my_c] = zz;
                        red_unit<NC>(Pbar + my_c, oa, wts + 4 * i, ta, nst);
                        red_unit<NC>(Pbar + my_c, obb, wts + 4 * (kAN + i), tb_, nst);
                    }
                __syncthreads();
                for (int i = tid; i < nn; i += nth) {
                    double a = 0.0;
                    for (int c = 0; c < CH; ++c) a += z[i * CH + c];
                    atomicAdd(&Wbar[(size_t)cidx * g.nmax + n0 + i], a);
                }
            }
        };
        channel(std::true_type{});
        channel(std::false_type{});
    }
    __syncthreads();

    // ---- t channel
    int4* offs = reinterpret_cast<int4*>(work);                                   // [A, B, C, D][node]
    double* wts = reinterpret_cast<double*>(work + 4 * 16 * kAN);                 // [A, B, C, D][node][corner]: density
    double* Wn = wts + 4 * 4 * kAN;                                               // [node]
    double* rows = Wn + kAN;                                                      // [q][A, B][rt]
    double* fac = rows + kAQ * 2 * rt;                                            // [q][C, D][factor, adjoint][component]
    double* z = fac + kAQ * 4 * NC;                                               // [q][2 row]
    const double* Pt = P + td.su_t;
    const int cidx = N + ti, nq = ncount[cidx];
    for (int n0 = 0; n0 < nq; n0 += kAN) {
        const int nn = min(kAN, nq - n0);
        __syncthreads();
        for (int idx = tid; idx < 2 * nn; idx += nth) {
            const int r = idx >= nn ? 1 : 0, i = idx - r * nn;
            const double x = nx[(size_t)cidx * g.nmax + n0 + i];
            if (r == 0) Wn[i] = nW[(size_t)cidx * g.nmax + n0 + i];
            const double y0 = r ? x + w2p : w1 + x, y1 = r ? x - w2 : w1p - x, m0 = mag(y0), m1 = mag(y1);
            const auto c0 = axis_of(wm, ih, g, m0), c1 = axis_of(wm, ih, g, m1);
            const int so = is_neg(y0) != is_neg(y1) ? td.ex_t : 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {   // the row itself, then the on-site row of the same searches
                int off[4];
                double wt[4];
                bool neg[4];
                corners<false>(h ? 2 : 1, c0, c1, ti, h ? less(m0, t) : less(m0, m1), N, rc, off, wt, neg);
                const int slot = h ? 3 - r : r, add = h ? 0 : so;
#pragma unroll
                for (int k = 0; k < 4; ++k) wt[k] = neg[k] ? -wt[k] : wt[k];
                offs[slot * kAN + i] = make_int4(off[0] + add, off[1] + add, off[2] + add, off[3] + add);
                st_w(wts + 4 * (slot * kAN + i), wt);
            }
        }
        __syncthreads();
        for (int q0 = 0; q0 < nn; q0 += kAQ) {
            const int qn = min(kAQ, nn - q0);
            if (q0 > 0) __syncthreads();
            // rows A, B over all sites, and the on-site rows C, D (site 0)
            for (int idx = tid; idx < qn * (2 * row + 2 * NC); idx += nth) {
                const int q = idx / (2 * row + 2 * NC), rem = idx - q * (2 * row + 2 * NC);
                const bool on = rem >= 2 * row;
                const int e = on ? rem - 2 * row : rem, n = on ? NC : row, rw = e >= n ? 1 : 0, v = e - rw * n;
                const int c = on ? v : v / Ns, at_ = on ? c * nst : c * nst + (v - c * Ns), slot = on ? 2 + rw : rw;
                const int4 of = offs[slot * kAN + q0 + q];
                double w[4];
                lds_w(wts + 4 * (slot * kAN + q0 + q), w);
                if (c > 0)
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = mag(w[k]);
                auto at = [&](int o) { return __ldg(Pt + at_ + (long)o * 2); };
                const double val = fma(w[3], at(of.w), fma(w[2], at(of.z), fma(w[1], at(of.y), w[0] * at(of.x))));
                if (on) fac[(q * 4 + 2 * rw + 1) * NC + c] = val;   // raw row, replaced by its adjoint below
                else rows[(q * 2 + rw) * rt + at_] = val;
            }
            __syncthreads();
            for (int idx = tid; idx < qn * 2; idx += nth) {
                double v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) v[c] = fac[(idx * 2 + 1) * NC + c];
#pragma unroll
                for (int c = 0; c < NC; ++c) fac[(idx * 2) * NC + c] = onsite_factor<double, NC>(v, c);
            }
            __syncthreads();
            // adjoint of the on-site factors: F_C gets sum o A over the sites (through the site's
            // component permutation), F_D gets sum o B
            for (int idx = tid; idx < qn * 2 * NC; idx += nth) {
                const int q = idx / (2 * NC), rw = (idx / NC) & 1, f = idx % NC;
                const double* R = rows + (q * 2 + rw) * rt;
                double a = 0.0;
                for (int r = 0; r < Ns; ++r) {
                    int c = f;
                    if (NC == 4 && rw == 0) {
                        const int pon = tb.onsite_perm[r];
#pragma unroll
                        for (int k = 0; k < NC; ++k)
                            if (perm_of(pon, k) == f) c = k;
                    }
                    a = fma(ob[c * Ns + r], R[c * nst + r], a);
                }
                fac[(q * 4 + 2 * rw + 1) * NC + f] = a;
            }
            // row adjoints: on-site and lattice sum, all nodes of the block at once per value
            for (int slot = tid; slot < 2 * row; slot += nth) {
                const int2 item = at.items[slot];
                const int it = item.x;
                const int rw = it >= row ? 1 : 0, v = it - rw * row, c = v / Ns, r = v - c * Ns;
                double la[kAQ];
#pragma unroll
                for (int q = 0; q < kAQ; ++q) la[q] = 0.0;
                const double* other = rows + (1 - rw) * rt;
                for (int j = 0; j < item.y; ++j) {
                    const int2 e = at.list[(size_t)j * 2 * row + slot];
                    const double pb = pbar[e.x];
#pragma unroll
                    for (int q = 0; q < kAQ; ++q)
                        if (q < qn) la[q] = fma(pb, other[2 * q * rt + e.y], la[q]);
                }
                const double oc = ob[v];
                const int fc = (NC == 4 && rw == 0) ? perm_of(tb.onsite_perm[r], c) : c;
#pragma unroll
                for (int q = 0; q < kAQ; ++q)
                    if (q < qn) {
                        const double on = oc * fac[(q * 4 + 2 * rw) * NC + fc], mine = rows[(q * 2 + rw) * rt + c * nst + r];
                        // weight adjoint: the lattice sum counts once (with row A)
                        z[q * 2 * row + it] = mine * (rw == 0 ? on + la[q] : on);
                        const double vb = Wn[q0 + q] * (on + la[q]);
                        const int4 of = offs[rw * kAN + q0 + q];
                        double w[4];
                        lds_w(wts + 4 * (rw * kAN + q0 + q), w);
                        double* b = Pbar + c * nst + r;
                        const int o4[4] = {of.x, of.y, of.z, of.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if ((__double_as_longlong(w[k]) & 0x7fffffffffffffffLL) != 0) atomicAdd(b + (long)o4[k] * 2, (c > 0 ? mag(w[k]) : w[k]) * vb);
                    }
            }
            __syncthreads();
            // on-site rows: components from the factors' adjoints (transpose of onsite_factor), scattered
            for (int idx = tid; idx < qn * 2 * NC; idx += nth) {
                const int q = idx / (2 * NC), rw = (idx / NC) & 1, c = idx % NC;
                const double* fb = fac + (q * 4 + 2 * rw + 1) * NC;
                double a = 0.0;
                if (NC == 2) a = c == 0 ? fb[0] + fb[1] : 3.0 * fb[0] - fb[1];
                else
#pragma unroll
                    for (int k = 0; k < NC; ++k) a += (c == 0 || k == 0 || k == c) ? fb[k] : -fb[k];
                a *= Wn[q0 + q];
                const int4 of = offs[(2 + rw) * kAN + q0 + q];
                const double* w = wts + 4 * ((2 + rw) * kAN + q0 + q);
                const int o4[4] = {of.x, of.y, of.z, of.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (w[k] != 0.0) atomicAdd(Pbar + (long)o4[k] * 2 + c * nst, (c > 0 ? mag(w[k]) : w[k]) * a);
            }
            // weight adjoints: 16 lanes per node, fixed order
            for (int base = tid >> 4; base < qn; base += nth >> 4) {
                const int l = tid & 15;
                double a = 0.0;
                for (int e = l; e < 2 * row; e += 16) a += z[base * 2 * row + e];
                for (int o = 8; o > 0; o >>= 1) a += __shfl_down_sync(0xffffu << (tid & 16), a, o, 16);
                if (l == 0) atomicAdd(&Wbar[(size_t)cidx * g.nmax + n0 + q0 + base], a);
            }
        }
    }
}

// Gammabar from the accumulators: transpose of the exchange in pack_rows, a block per stored triple
// (shared memory: NC * Ns doubles).
template <int NC>
__global__ void k_pair_fold(Geo g, Tabs tb, Tab td, const double* __restrict__ Pbar, double* __restrict__ Gbar) {
    extern __shared__ double acc[];
    const int Ns = g.Ns;
    for (int row = blockIdx.x; row < td.nrow; row += gridDim.x) {
        for (int x = 0; x < (td.ex_t ? 2 : 1); ++x) {
            for (int r = threadIdx.x; r < Ns; r += blockDim.x) {
                const double* bt = Pbar + (x ? (size_t)td.ex_t * 2 : 0) + (size_t)row * NC * td.nst + r;
                // (the exchange permutes the stored entries: no two threads meet)
                const int rs = x ? tb.swap_r[r] : r, pm = x ? tb.swap_perm[r] : 0xe4;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    double& a = acc[perm_of(pm, c) * Ns + rs];
                    const double v = bt[c * td.nst];
                    a = x ? a + v : v;
                }
            }
            __syncthreads();
        }
        for (int e = threadIdx.x; e < NC * Ns; e += blockDim.x) Gbar[(size_t)row * NC * Ns + e] = acc[e];
        __syncthreads();
    }
}

}  // namespace pairk
