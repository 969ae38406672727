// TRI vertex flow with the lattice sum as a dense contraction (internal header, included by
// flow.cu after tri.cuh).
//
// The t-channel lattice sum of a stored triple is, over the integration nodes q and every table
// entry (rA, rB) of an output site, the 4 x 4 spin-matrix product sum_l A^{mu l}_j B^{l nu}_j of
// rows read through signed permutations of the spin indices.  The permutations of the outer indices
// and all signs can wait until the nodes are summed, so the kernel integrates
//     C_{k}[(rA, mu)][(rB, nu)] = sum_q A_q[rA]^{mu kappa} B_q[rB]^{kappa' nu}
// once for every inner pair k = (kappa, kappa') the table uses -- a plain matrix product with the
// nodes as the inner dimension, kept in register tiles across the t channel -- and the outputs
// gather their signed terms from C at the end of the triple.  Entries that differ only in the
// images of the outer indices or in signs share one product (kagome with Dzyaloshinskii-Moriya
// couplings, range 7: 2543 entries, 1156 pairs of sites).
//
// Graded flows (GR): a lattice whose component maps all preserve the parity of a spin axis (the
// number of indices among the two other axes, even or odd) keeps a vertex without odd components
// free of them: every product of the flow equations has an even number of odd factors.  Then only
// 8 of the 16 functions take part, in two 2 x 2 blocks {0, z} and {x, y} (the axis relabelled z).
// Whether the state at hand has odd components is read off the state itself when it is packed
// (k_tri_pack sets a flag, which the kernels of both forms test), so any state is served.
//
// The s and u channels need no shared memory: a thread interpolates both rows of its site and
// multiplies them in registers (4 + 4 corner rows per node; consecutive lanes read consecutive sites).
//
// Measured against the general kernel (whole right-hand side, one GB300):
//   kagome Dzyaloshinskii-Moriya, range 7, 32 frequencies, FP32   27.2 -> 2.9 ms
//   the same model, range 4, 24 frequencies, FP64                 24.8 -> 3.3 ms
//   honeycomb Kitaev-Gamma, range 4, 24 frequencies, FP32          2.5 -> 0.65 ms
// What bounds it now: FP32, the L1 / shared-memory data path (75 % busy at range 7: corner rows, and
// three 16-byte operand loads per 32 multiply-adds of a tile); FP64, the FP64 pipe (2 per clock and
// SM): 1.7 G multiply-adds take 2.8 ms of the 3.3.
#pragma once

namespace trid {

constexpr int kMaxPairs = 16;

// Tables of the dense form (device pointers).
struct Tab {
    const int2* pack;      // 16 Ns: packed position of a state entry (plain; exchanged | sign << 30),
                           // x = -1 for an odd component of a graded flow
    const unsigned* fmap;  // Ns * NCm / 4: a byte per component of the on-site factor (index | sign << 4)
    const int* ent;        // GR: entries of every output site by class: offset of the block (rA, rB) in C_k
    const int2* runs;      // GR: (begin, end) of every run of equal class
    const int* run_pair;   // GR: run * 4 + l: inner pair k of the inner index l
    const int* n_terms;    // Ns: terms of every output of a site
    const int* terms;      // [term][m * Ns + r]: offset into the run sums (GR) or into C | sign << 30
    int n_runs, nk;        // runs, inner pairs
    int kap[kMaxPairs];    // kappa | kappa' << 4
    int spin[4];           // stored spin index of the internal one (cyclic relabelling)
    int nrow;              // packed rows (stored triples): the exchanged rows start nrow * NCm * Ns later
    unsigned div_half;     // ceil(2^32 / (NCm Ns / 8))
};

template <typename R>
struct __align__(16) DescD {
    int off[4];
    R wd[4];   // corner weights of functions whose second spin index (as read) is 0
    R ws[4];   // of the others
};

template <bool GR> __host__ __device__ constexpr int ncomp() { return GR ? 8 : 16; }
template <bool GR> __host__ __device__ constexpr int nmu() { return GR ? 2 : 4; }

// internal component m of a packed site: graded 2 x 2 blocks {0, 3} then {1, 2}, else mu * 4 + nu
__host__ __device__ constexpr int mu_of(bool gr, int m) { return !gr ? m >> 2 : (m < 4 ? ((m >> 1) ? 3 : 0) : ((m >> 1) & 1 ? 2 : 1)); }
__host__ __device__ constexpr int nu_of(bool gr, int m) { return !gr ? m & 3 : (m < 4 ? ((m & 1) ? 3 : 0) : ((m & 1) ? 2 : 1)); }
__host__ __device__ constexpr bool same_block(int a, int b) { return ((a == 0) || (a == 3)) == ((b == 0) || (b == 3)); }
// position of a spin index inside its block (graded) / itself
__host__ __device__ constexpr int in_block(bool gr, int a) { return !gr ? a : (a == 3 || a == 2 ? 1 : 0); }
__host__ __device__ constexpr int idx_of(bool gr, int mu, int nu) {
    return !gr ? mu * 4 + nu : ((mu == 0 || mu == 3) ? 0 : 4) + in_block(true, mu) * 2 + in_block(true, nu);
}

// The on-site terms factorise like the lattice sum: out^{mu nu} += sum_l A^{mu l} F2^{l nu} and
// sum_m F3^{mu m} B^{m nu} with node factors that do not depend on the site, F2^{l nu} = sum_m
// phi2 C^{m (m^l^nu)} and F3^{mu m} = sum_l phi3 D^{(mu^l^m) l} (64 products instead of 256 each).
__host__ __device__ constexpr int phi2(int l, int nu, int m) {
    using namespace sr::tri;
    return sgn_of(pexp(m, l) + pexp(m ^ l, m ^ l ^ nu) + iota(m, m ^ l ^ nu) - iota(l, nu));
}
__host__ __device__ constexpr int phi3(int mu, int m, int l) {
    using namespace sr::tri;
    return sgn_of(pexp(l, m) + pexp(l ^ m, mu ^ l ^ m) + iota(mu ^ l ^ m, l) - iota(mu, m));
}
__host__ __device__ constexpr bool factors_ok() {
    using namespace sr::tri;
    for (int mu = 0; mu < 4; ++mu)
        for (int nu = 0; nu < 4; ++nu)
            for (int l = 0; l < 4; ++l)
                for (int m = 0; m < 4; ++m) {
                    if (coef_o2(mu, nu, l, m) != coef_t(mu, nu, l) * phi2(l, nu, m)) return false;
                    if (coef_o3(mu, nu, l, m) != coef_t(mu, nu, m) * phi3(mu, m, l)) return false;
                }
    return true;
}
static_assert(factors_ok(), "on-site coefficients factorise");

template <typename R> __host__ __device__ constexpr int qblock() { return sizeof(R) == 4 ? 32 : 16; }   // nodes per shared-memory block

// Row length of one kappa vector (nm Ns entries): FP32 padded to the 8 x 4 tiles and, for full rows,
// to 8 modulo 32 words so that the four mu of a site's row store to different banks; FP64 tiles
// divide nm Ns.
template <typename R, bool GR>
__host__ __device__ inline int row_ld(int Ns) {
    const int n = nmu<GR>() * Ns;
    if (sizeof(R) == 8) return n;
    int ld = (n + 7) & ~7;
    if (!GR)
        while ((ld & 31) != 8) ld += 8;
    return ld;
}

template <bool GR, int TM, int TN>
__host__ __device__ inline int tiles(int Ns, int nk) {
    const int n = nmu<GR>() * Ns;
    return nk * ((n + TM - 1) / TM) * ((n + TN - 1) / TN);
}

template <typename R, bool GR>
__host__ __device__ inline size_t smem_bytes(int N, int Ns, int nk, int n_runs, int threads) {
    constexpr int NCm = ncomp<GR>(), QB = qblock<R>();
    auto rnd = [](size_t b) { return (b + 15) & ~size_t(15); };
    const size_t ld = row_ld<R, GR>(Ns), LM = (size_t)nmu<GR>() * Ns, nmax = 2 * (size_t)N + 8;   // nodes of a channel
    const int NG = threads / Ns;
    const size_t blk = rnd(sizeof(R) * QB * 2 * 4 * ld), on = rnd(sizeof(R) * nmax * 2 * NCm), rows = blk > on ? blk : on;
    const size_t fin = rnd(sizeof(R) * nk * LM * LM) + rnd(sizeof(R) * NG * Ns * NCm) +
                       (GR ? rnd(sizeof(R) * n_runs * 16) : 0);
    return rnd(sizeof(DescD<R>) * nmax * 4) + rnd(sizeof(int) * nmax * 4) + rnd(sizeof(R) * nmax * 2 * NCm) +
           (rows > fin ? rows : fin);
}

// Corner pair of one axis: axis_weights with a single corner repeated under weight zero.
template <typename R>
__device__ __forceinline__ void axis_pair(const Tabs& tb, const Geo& g, double x, int* ix, R* wx) {
    int n;
    axis_weights<R>(tb, g, x, n, ix, wx);
    if (n == 1) { ix[1] = ix[0]; wx[1] = R(0); }
}

// Descriptor of Gamma(s, t, u) with the exact argument ex_slot = w[ex_idx]: the folding of
// make_desc, the exact axis selected arithmetically (lanes take one path).
template <typename R>
__device__ __forceinline__ int make_desc_d(double s, double t, double u, int ex_slot, int ex_idx, const Tabs& tb, const Geo& g,
                                           int rowp, int swap_off, R scale, DescD<R>* dst) {
    constexpr long long kMag = 0x7fffffffffffffffLL;
    auto negative = [](double x) { const long long b = __double_as_longlong(x); return b < 0 && (b & kMag) != 0; };
    auto mag = [](double x) { return __longlong_as_double(__double_as_longlong(x) & kMag); };
    const bool ns = negative(s), nt = negative(t), nu = negative(u);
    const bool swap = ns != nu;
    s = mag(s); t = mag(t); u = mag(u);
    const bool flip = __double_as_longlong(s) < __double_as_longlong(u);
    const double sh = flip ? u : s, uh = flip ? s : u;
    const int ea = (flip && ex_slot != 1) ? 2 - ex_slot : ex_slot;
    int i0[2], i1[2];
    R v0[2], v1[2];
    axis_pair<R>(tb, g, ea == 0 ? t : sh, i0, v0);
    axis_pair<R>(tb, g, ea == 2 ? t : uh, i1, v1);
    v0[0] *= scale;
    v0[1] *= scale;
    const int so = swap ? swap_off : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int a = i0[k & 1], b = i1[k >> 1];
        const int js = ea == 0 ? ex_idx : a;
        const int jt = ea == 1 ? ex_idx : (ea == 0 ? a : b);
        const int ju = ea == 2 ? ex_idx : b;
        const R wt = v0[k & 1] * v1[k >> 1];
        const bool below = js < ju;
        dst->off[k] = (pair_index(below ? ju : js, below ? js : ju) * g.N + jt) * rowp + so;
        dst->wd[k] = (flip != below) ? -wt : wt;
        dst->ws[k] = wt;
    }
    return (swap ? 1 : 0) | ((nt != nu) ? 2 : 0);
}

__device__ __forceinline__ void load4(const float* p, float* v) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void load4(const double* p, double* v) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
// N consecutive values of a shared-memory vector (N a power of two, suitably aligned)
template <int N>
__device__ __forceinline__ void lds(const float* p, float* v) {
    if constexpr (N >= 4) {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 a = *reinterpret_cast<const float4*>(p + i);
            v[i] = a.x; v[i + 1] = a.y; v[i + 2] = a.z; v[i + 3] = a.w;
        }
    } else {
        const float2 a = *reinterpret_cast<const float2*>(p);
        v[0] = a.x; v[1] = a.y;
    }
}
template <int N>
__device__ __forceinline__ void lds(const double* p, double* v) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const double2 a = *reinterpret_cast<const double2*>(p + i);
        v[i] = a.x; v[i + 1] = a.y;
    }
}

__device__ __forceinline__ void sts2(float* p, float a, float b) { *reinterpret_cast<float2*>(p) = make_float2(a, b); }
__device__ __forceinline__ void sts2(double* p, double a, double b) { *reinterpret_cast<double2*>(p) = make_double2(a, b); }
__device__ __forceinline__ void sts4(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void sts4(double* p, const double* v) {
    sts2(p, v[0], v[1]);
    sts2(p + 2, v[2], v[3]);
}

// One packed 4-value chunk of a row (element 4 (kind Ns + r)): four corners, weights by the type of
// each function, sign of t -> -t / u -> -u for the imaginary class.  Graded: kind 0 = (00, 03, 30, 33),
// 1 = block {1, 2}; full: row mu = kind of the 4 x 4 matrix.  The weight set goes by the second spin index of the function
// as stored, which for an exchanged lookup is the first one of the function read.
template <typename R, bool GR>
__device__ __forceinline__ void chunk_value(const R* __restrict__ P, const DescD<R>& d, int flags, int elem, int kind, R* v) {
    R c[4][4], wd[4], ws[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        load4(P + d.off[k] + elem, c[k]);
        wd[k] = d.wd[k];
        ws[k] = d.ws[k];
    }
    const bool sw = flags & 1, mn = flags & 2;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        bool dens;   // weight set
        bool mixed;  // imaginary class
        if (GR) {
            dens = kind == 0 && (j == 0 || (j == 1 && sw) || (j == 2 && !sw));
            mixed = kind == 0 && (j == 1 || j == 2);
        } else {
            dens = sw ? kind == 0 : j == 0;
            mixed = (kind == 0) != (j == 0);
        }
        R a = (dens ? wd[0] : ws[0]) * c[0][j];
#pragma unroll
        for (int k = 1; k < 4; ++k) a = fmadd(dens ? wd[k] : ws[k], c[k][j], a);
        v[j] = (mixed && mn) ? -a : a;
    }
}

// Site-local product of the s (CH = 0) or u (CH = 2) channel on internal components.
template <int CH, bool GR, typename R>
__device__ __forceinline__ void su_acc(const R* a, const R* b, R* o) {
#pragma unroll
    for (int m = 0; m < ncomp<GR>(); ++m) {
        const int mu = mu_of(GR, m), nu = nu_of(GR, m);
#pragma unroll
        for (int n = 0; n < ncomp<GR>(); ++n) {
            const int x = mu_of(GR, n), y = nu_of(GR, n);
            const int cf = CH == 0 ? sr::tri::coef_s(mu, nu, x, y) : sr::tri::coef_u(mu, nu, x, y);
            const R p = b[idx_of(GR, x ^ mu, y ^ nu)];
            o[m] = fmadd(cf > 0 ? a[n] : -a[n], p, o[m]);
        }
    }
}

// dGamma/dLambda of one stored triple per CTA.  P: packed state (plain rows, then exchanged rows).
// use: nullptr, or the flag of k_tri_pack (zero: this form serves the state).
template <typename R, bool GR, int TM, int TN, int NT, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
k_gamma_rhs_trid(Geo g, Tabs tb, Tab td, const double* __restrict__ w, const R* __restrict__ P, const double* __restrict__ nx,
                 const double* __restrict__ nW, const int* __restrict__ ncount, double* __restrict__ dG, int p0,
                 const int* __restrict__ use) {
    if (use && *use != 0) return;   // the general kernel serves this state
    constexpr int NCm = ncomp<GR>(), NM = nmu<GR>(), QB = qblock<R>();
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, nth = blockDim.x, Ns = g.Ns;
    const int ld = row_ld<R, GR>(Ns), LM = NM * Ns, rowq = 4 * ld;   // one row (A or B) of a node: 4 kappa vectors
    const int rowp = NCm * Ns, half = rowp / 8;
    size_t so = 0;
    auto take = [&](size_t bytes) { unsigned char* q = smem + so; so += (bytes + 15) & ~size_t(15); return q; };
    DescD<R>* desc = (DescD<R>*)take(sizeof(DescD<R>) * g.nmax * 4);   // of a whole channel
    int* flags = (int*)take(sizeof(int) * g.nmax * 4);
    R* onf = (R*)take(sizeof(R) * g.nmax * 2 * NCm);
    R* rows = (R*)take(0);
    const int ti = blockIdx.x % g.N;
    const int p = p0 + (int)(blockIdx.x / g.N);
    int si = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((si + 1) * (si + 2) / 2 <= p) ++si;
    while (si * (si + 1) / 2 > p) --si;
    const int ui = p - si * (si + 1) / 2;
    const double s = w[si], t = w[ti], u = w[ui];
    const double w1p = (s + t + u) / 2, w2p = (s - t - u) / 2, w1 = (s - t + u) / 2, w2 = (s + t - u) / 2;
    const int swap_off = td.nrow * rowp;

    // site-local products: thread (site my_r, node group my_g), sums in registers for the triple
    // (the host launches at least Ns threads)
    const int NG = nth / Ns;
    const int my_g = tid / Ns, my_r = tid - my_g * Ns;
    const bool site_on = my_g < NG;
    R so_acc[NCm];
#pragma unroll
    for (int m = 0; m < NCm; ++m) so_acc[m] = R(0);

    // descriptors of all nodes of a channel at once (one search chain per thread); the node weight
    // rides on the first row and the second on-site row
    auto descriptors = [&](int ch, int first) {
        const int vi = ch == 0 ? si : (ch == 1 ? ti : ui), cidx = ch * g.N + vi, nq = ncount[cidx], nrow = ch == 1 ? 4 : 2;
        for (int idx = tid; idx < nq * nrow; idx += nth) {
            const int rw = idx / nq, q = idx - rw * nq;
            double a, b, c;
            node_args(ch, rw, nx[(size_t)cidx * g.nmax + q], s, t, u, w1p, w2p, w1, w2, a, b, c);
            const int exs = ch == 0 ? 0 : (ch == 2 ? 2 : (rw < 2 ? 1 : 2)), at = first + q * nrow + rw;
            flags[at] = make_desc_d<R>(a, b, c, exs, vi, tb, g, rowp, swap_off,
                                       (rw == 0 || rw == 3) ? (R)nW[(size_t)cidx * g.nmax + q] : R(1), &desc[at]);
        }
        return nq;
    };

    // s and u channels: a thread interpolates both rows of its site and multiplies them in
    // registers; consecutive lanes read consecutive sites of a corner row
    const int nqs = descriptors(0, 0), nqu = descriptors(2, 2 * g.nmax);
    __syncthreads();
    if (site_on) {
        auto channel = [&](auto ch, int nq, int first) {
            for (int q = my_g; q < nq; q += NG) {
                R a[NCm], b[NCm];
#pragma unroll
                for (int h = 0; h < NCm / 4; ++h) {
                    chunk_value<R, GR>(P, desc[first + 2 * q], flags[first + 2 * q], 4 * (h * Ns + my_r), h, a + 4 * h);
                    chunk_value<R, GR>(P, desc[first + 2 * q + 1], flags[first + 2 * q + 1], 4 * (h * Ns + my_r), h, b + 4 * h);
                }
                su_acc<decltype(ch)::value, GR, R>(a, b, so_acc);
            }
        };
        channel(std::integral_constant<int, 0>{}, nqs, 0);
        channel(std::integral_constant<int, 2>{}, nqu, 2 * g.nmax);
    }
    __syncthreads();

    // t channel: descriptors, the on-site rows (site 0) and the node factors of the on-site terms
    const int nq = descriptors(1, 0);
    __syncthreads();
    {
        R* onrow = rows;   // [node][C, D][m]
        constexpr int NCk = NCm / 4;
        for (int idx = tid; idx < nq * 2 * NCk; idx += nth) {
            const int q = idx / (2 * NCk), rr = (idx / NCk) & 1, h = idx % NCk;
            R v[4];
            chunk_value<R, GR>(P, desc[q * 4 + 2 + rr], flags[q * 4 + 2 + rr], h * 4 * Ns, h, v);
            sts4(onrow + (q * 2 + rr) * NCm + 4 * h, v);
        }
        __syncthreads();
        for (int idx = tid; idx < nq * 2; idx += nth) {
            R cv[NCm];
#pragma unroll
            for (int m = 0; m < NCm; ++m) cv[m] = onrow[idx * NCm + m];
#pragma unroll
            for (int m = 0; m < NCm; ++m) {
                const int a = mu_of(GR, m), b = nu_of(GR, m);
                R f2 = R(0), f3 = R(0);
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    const R x2 = cv[idx_of(GR, l, l ^ a ^ b)], x3 = cv[idx_of(GR, a ^ l ^ b, l)];
                    f2 = phi2(a, b, l) > 0 ? f2 + x2 : f2 - x2;
                    f3 = phi3(a, b, l) > 0 ? f3 + x3 : f3 - x3;
                }
                onf[idx * NCm + m] = (idx & 1) ? f3 : f2;
            }
        }
        __syncthreads();
    }
    unsigned fcode[NCm / 4];   // on-site component map of the thread's site, a byte per component
#pragma unroll
    for (int i = 0; i < NCm / 4; ++i) fcode[i] = td.fmap[my_r * (NCm / 4) + i];

    // contraction tiles of this thread (padding entries of the rows are read by the tiles but never
    // used: they start out finite)
    if (ld > LM)
        for (int i = tid; i < QB * 8 * (ld - LM); i += nth) rows[(i / (ld - LM)) * ld + LM + i % (ld - LM)] = R(0);
    const int tm = (LM + TM - 1) / TM, tn = (LM + TN - 1) / TN, ntile = td.nk * tm * tn;
    int ta[NT], tbo[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int id = tid + j * nth;
        ta[j] = -1;
        tbo[j] = 0;
        if (id < ntile) {
            const int k = id / (tm * tn), rem = id - k * (tm * tn), a = rem / tn, b = rem - a * tn;
            ta[j] = (td.kap[k] & 15) * ld + a * TM;
            tbo[j] = rowq + (td.kap[k] >> 4) * ld + b * TN;
        }
    }
    R acc[NT][TM][TN];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int b = 0; b < TN; ++b) acc[j][a][b] = R(0);
    {
        for (int q0 = 0; q0 < nq; q0 += QB) {
            const int qn = min(QB, nq - q0);
            if (q0 > 0) __syncthreads();   // the previous block's rows are consumed
            // rows: an item is two packed chunks of a (node, row)
            for (int idx = tid; idx < qn * 2 * half; idx += nth) {
                const int qr = half > 1 ? (int)__umulhi((unsigned)idx, td.div_half) : idx;
                const int x = idx - qr * half;
                const int dq = (q0 + (qr >> 1)) * 4 + (qr & 1);
                const DescD<R>& d = desc[dq];
                const int fl = flags[dq];
                R* dst = rows + (size_t)qr * rowq;
                const bool ra = (qr & 1) == 0;   // row A keeps its kappa (second index) vectors, B its kappa' (first)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    R v[4];
                    if constexpr (GR) {
                        chunk_value<R, true>(P, d, fl, 4 * (x + h * half), h, v);
                        sts2(dst + (h ? 1 : 0) * ld + 2 * x, v[0], ra ? v[2] : v[1]);
                        sts2(dst + (h ? 2 : 3) * ld + 2 * x, ra ? v[1] : v[2], v[3]);
                    } else {
                        const int mu = (x >= Ns ? 1 : 0) + 2 * h, r = x >= Ns ? x - Ns : x;
                        chunk_value<R, false>(P, d, fl, 4 * (x + h * half), mu, v);
                        if (ra) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) dst[j * ld + 4 * r + mu] = v[j];
                        } else {
                            sts4(dst + mu * ld + 4 * r, v);
                        }
                    }
                }
            }
            __syncthreads();
            // on-site terms
            if (site_on)
                for (int q = my_g; q < qn; q += NG) {
                    const int r = my_r;
                    const R* A = rows + (size_t)(2 * q) * rowq + NM * r;
                    R a[NCm], b[NCm];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        R va[NM], vb[NM];
                        lds<NM>(A + k * ld, va);
                        lds<NM>(A + rowq + k * ld, vb);
#pragma unroll
                        for (int i = 0; i < NM; ++i) {
                            const int o = GR ? ((k == 0 || k == 3) ? (i ? 3 : 0) : (i ? 2 : 1)) : i;
                            a[idx_of(GR, o, k)] = va[i];
                            b[idx_of(GR, k, o)] = vb[i];
                        }
                    }
                    {
                        R f2[NCm], f3[NCm];
#pragma unroll
                        for (int m = 0; m < NCm; ++m) {
                            const unsigned code = (fcode[m >> 2] >> (8 * (m & 3))) & 255u;
                            const R x = onf[(2 * (q0 + q)) * NCm + (code & 15u)];
                            f2[m] = (code & 16u) ? -x : x;
                            f3[m] = onf[(2 * (q0 + q) + 1) * NCm + m];
                        }
#pragma unroll
                        for (int m = 0; m < NCm; ++m) {
                            const int mu = mu_of(GR, m), nu = nu_of(GR, m);
#pragma unroll
                            for (int l = 0; l < 4; ++l)
                                if (!GR || same_block(l, mu)) {
                                    const int ma = idx_of(GR, mu, l), mb = idx_of(GR, l, nu);
                                    const bool pos = sr::tri::coef_t(mu, nu, l) > 0;
                                    so_acc[m] = fmadd(pos ? a[ma] : -a[ma], f2[mb], so_acc[m]);
                                    so_acc[m] = fmadd(pos ? f3[ma] : -f3[ma], b[mb], so_acc[m]);
                                }
                        }
                    }
                }
            // lattice sum: register tiles over the block's nodes
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    if (ta[j] >= 0) {
                        const R* A = rows + ta[j];
                        const R* B = rows + tbo[j];
#pragma unroll 2
                        for (int q = 0; q < qn; ++q) {
                            R a[TM], b[TN];
                            lds<TM>(A + (size_t)(2 * q) * rowq, a);
                            lds<TN>(B + (size_t)(2 * q) * rowq, b);
#pragma unroll
                            for (int x = 0; x < TM; ++x)
#pragma unroll
                                for (int y = 0; y < TN; ++y) acc[j][x][y] = fmadd(a[x], b[y], acc[j][x][y]);
                        }
                    }
        }
    }
    // end of the triple: C and the site partials to shared memory
    __syncthreads();
    R* C = rows;
    R* part = (R*)((unsigned char*)rows + ((sizeof(R) * td.nk * LM * LM + 15) & ~size_t(15)));   // [group][site][m]
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int id = tid + j * nth;
        if (id < ntile) {
            const int k = id / (tm * tn), rem = id - k * (tm * tn), a0 = (rem / tn) * TM, b0 = (rem % tn) * TN;
            if constexpr (GR) {   // 2 x 2 blocks [k][rA][rB]
#pragma unroll
                for (int x = 0; x < TM; x += 2)
#pragma unroll
                    for (int y = 0; y < TN; y += 2)
                        if (a0 + x < LM && b0 + y < LM) {
                            const R v[4] = {acc[j][x][y], acc[j][x][y + 1], acc[j][x + 1][y], acc[j][x + 1][y + 1]};
                            sts4(C + (size_t)((k * Ns + (a0 + x) / 2) * Ns + (b0 + y) / 2) * 4, v);
                        }
            } else {              // rows [k][(rA, mu)][(rB, nu)]
#pragma unroll
                for (int x = 0; x < TM; ++x)
                    if (a0 + x < LM && b0 < LM) sts4(C + (size_t)(k * LM + a0 + x) * LM + b0, acc[j][x]);
            }
        }
    }
    if (site_on)
#pragma unroll
        for (int m = 0; m < NCm; ++m) part[((size_t)my_g * Ns + my_r) * NCm + m] = so_acc[m];
    __syncthreads();
    // outputs, gathered in a fixed order.  Graded lattices have few classes of entries (equal
    // component maps) and long runs of each class at a site: the blocks of every (run, inner index)
    // are summed first, a thread each, and the outputs pick their signed terms from these sums.
    // Otherwise every output sums its own terms.
    R* src = C;
    if constexpr (GR) {
        R* raw = part + (size_t)NG * Ns * NCm;   // [run][l][4]
        for (int o = tid; o < td.n_runs * 4; o += nth) {
            const int ru = o >> 2, k = td.run_pair[o];
            const int2 run = td.runs[ru];
            const R* base = C + (size_t)k * Ns * Ns * 4;
            R x[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll 4
            for (int e = run.x; e < run.y; ++e) {
                R v[4];
                lds<4>(base + td.ent[e], v);
#pragma unroll
                for (int j = 0; j < 4; ++j) x[j] += v[j];
            }
            sts4(raw + (size_t)o * 4, x);
        }
        __syncthreads();
        src = raw;
    }
    double* out = dG + (size_t)(p * g.N + ti) * 16 * Ns;
    for (int o = tid; o < Ns * NCm; o += nth) {
        const int m = o / Ns, r = o - m * Ns;
        R a = R(0), l = R(0);
        for (int k = 0; k < NG; ++k) a += part[((size_t)k * Ns + r) * NCm + m];
        // (four partial sums: independent loads, and a smaller rounding error of the long FP32 lists)
        const int nt = td.n_terms[r];
        R lp[4] = {R(0), R(0), R(0), R(0)};
        for (int j = 0; j < nt; j += 4)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (j + i < nt) {
                    const int c = td.terms[(size_t)(j + i) * Ns * NCm + o];
                    const R v = src[c & 0x3fffffff];
                    lp[i] += (c >> 30) & 1 ? -v : v;
                }
        l = (lp[0] + lp[1]) + (lp[2] + lp[3]);
        const int mu = mu_of(GR, m), nu = nu_of(GR, m);
        out[(td.spin[mu] * 4 + td.spin[nu]) * Ns + r] = (double)a - 2.0 * (double)l;
    }
    if (GR)
        for (int o = tid; o < Ns * 8; o += nth) {
            const int m = o / Ns, r = o - m * Ns, mu = m >> 1;   // odd components: mu and nu in different blocks
            const int nu = (mu == 0 || mu == 3) ? ((m & 1) ? 2 : 1) : ((m & 1) ? 3 : 0);
            out[(td.spin[mu] * 4 + td.spin[nu]) * Ns + r] = 0.0;
        }
}

// Packed copy of the FP64 state, plain and exchanged rows; one block per stored triple.  Graded:
// *flag is set when the state has an odd component or a value that is not finite.
template <typename R, bool GR>
__global__ void k_tri_pack(Geo g, Tab td, const double* __restrict__ G, R* __restrict__ P, int* __restrict__ flag) {
    const int rowp = ncomp<GR>() * g.Ns;
    const size_t ex = (size_t)td.nrow * rowp;
    bool bad = false;
    for (int pt = blockIdx.x; pt < td.nrow; pt += gridDim.x) {
        const double* src = G + (size_t)pt * 16 * g.Ns;
        R* dst = P + (size_t)pt * rowp;
        for (int e = threadIdx.x; e < 16 * g.Ns; e += blockDim.x) {
            const double v = src[e];
            const int2 c = td.pack[e];
            if (c.x < 0) bad |= v != 0.0;   // also true for NaN
            else {
                bad |= !isfinite(v);
                dst[c.x] = (R)v;
                dst[ex + (c.y & 0x3fffffff)] = (c.y >> 30) & 1 ? (R)-v : (R)v;
            }
        }
    }
    if (GR && bad) *flag = 1;
}

// FP32 copy in the state's own layout, made only when *flag says that the graded form does not apply.
__global__ void k_shadow_if(long n, const double* __restrict__ G, float* __restrict__ Gf, const int* __restrict__ flag) {
    if (*flag == 0) return;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) Gf[i] = (float)G[i];
}

// ---- host side

template <typename R>
using Kernel = void (*)(Geo, Tabs, Tab, const double*, const R*, const double*, const double*, const int*, double*, int,
                        const int*);

template <typename R>
struct Variant {
    Kernel<R> fn;
    int tm, tn, nt, max_threads;
};

// Kernel variants in order of preference (tiles of tm x tn, nt per thread, registers capped for the
// resident CTAs named).  Measured with kagome Dzyaloshinskii-Moriya range 7 (612 tiles, FP32): 2 tiles
// on 320 threads, two CTAs per SM, 2.9 ms; 3 on 224, two CTAs, 3.4; 2 on 320, one CTA, 3.5; 3 on 224,
// one CTA, 4.0 (without the cap on registers nothing spills, but a lone CTA waits at its barriers).
// Full rows need the registers: honeycomb Kitaev-Gamma range 4 (320 tiles), 3 tiles on 128 threads
// 0.65 ms, 2 on 160 with the cap 0.86, 1 on 320 0.75.
template <typename R, bool GR>
inline std::vector<Variant<R>> variants() {
    if constexpr (sizeof(R) == 4 && GR)
        return {{k_gamma_rhs_trid<R, GR, 8, 4, 2, 320, 2>, 8, 4, 2, 320},
                {k_gamma_rhs_trid<R, GR, 8, 4, 1, 256, 3>, 8, 4, 1, 256},
                {k_gamma_rhs_trid<R, GR, 8, 4, 3, 384, 1>, 8, 4, 3, 384}};
    else if constexpr (sizeof(R) == 4)
        return {{k_gamma_rhs_trid<R, GR, 8, 4, 3, 384, 1>, 8, 4, 3, 384}, {k_gamma_rhs_trid<R, GR, 8, 4, 1, 256, 2>, 8, 4, 1, 256}};
    else if constexpr (GR)
        return {{k_gamma_rhs_trid<R, GR, 2, 2, 6, 512, 1>, 2, 2, 6, 512}, {k_gamma_rhs_trid<R, GR, 2, 2, 12, 448, 1>, 2, 2, 12, 448}};
    else
        return {{k_gamma_rhs_trid<R, GR, 4, 4, 1, 512, 1>, 4, 4, 1, 512}, {k_gamma_rhs_trid<R, GR, 4, 4, 3, 384, 1>, 4, 4, 3, 384}};
}

template <typename R>
struct Choice {
    Kernel<R> fn = nullptr;
    int threads = 0;
    size_t smem = 0;
};

// The first variant that fits a CTA and fills at least three warps with tiles; where none fills them
// (lattices of a few sites), the first that fits; none when the tiles or the shared memory exceed one CTA.
template <typename R, bool GR>
inline Choice<R> choose(int N, int Ns, int nk, int n_runs) {
    Choice<R> c;
    for (const Variant<R>& v : variants<R, GR>()) {
        const int n = nmu<GR>() * Ns, T = nk * ((n + v.tm - 1) / v.tm) * ((n + v.tn - 1) / v.tn);
        const int need = std::max((T + v.nt - 1) / v.nt, Ns), th = std::max(128, (need + 31) / 32 * 32);
        const size_t sm = smem_bytes<R, GR>(N, Ns, nk, n_runs, th);
        if (th > v.max_threads || sm > 227 * 1024) continue;
        if (c.fn && need < 96) continue;   // too few tiles to use more of them per thread
        c.fn = v.fn;
        c.threads = th;
        c.smem = sm;
        if (need >= 96) break;
    }
    return c;
}

// Host tables of the dense form.
struct Plan {
    bool graded = false;
    int axis = 0;
    int nk = 0;
    int kap[kMaxPairs] = {};
    int spin[4] = {0, 1, 2, 3};
    std::vector<int2> pack;
    std::vector<unsigned> fmap;
    std::vector<int> ent, run_pair, n_terms, terms;
    std::vector<int2> runs;
};

inline bool even_comp(int c, int axis) { return ((c >> 2) == 0 || (c >> 2) == axis) == ((c & 3) == 0 || (c & 3) == axis); }

// Tables for a lattice; false when the maps do not fit (the general kernel serves it then).
inline bool build_tables(const sr_lattice* lat, Plan* pl) {
    const int Ns = lat->Ns;
    // graded about axis a: every component map keeps even functions even, and the bare vertex is even
    auto keeps = [&](const sr::Map16& m, int a) {
        for (int c = 0; c < 16; ++c)
            if (even_comp(c, a) != even_comp(m[c] & 15, a)) return false;
        return true;
    };
    for (int a = 3; a >= 1 && !pl->graded; --a) {
        bool ok = true;
        for (int r = 0; r < Ns && ok; ++r) {
            ok = keeps(lat->swap_map16[r], a) && keeps(lat->onsite_map16[r], a);
            for (int c = 0; c < 16 && ok; ++c) ok = even_comp(c, a) || lat->init_gamma[(size_t)r * 16 + c] == 0.0;
        }
        for (size_t e = 0; e < lat->rpa16.size() && ok; ++e) ok = keeps(lat->rpa16[e].mA, a) && keeps(lat->rpa16[e].mB, a);
        if (ok) { pl->graded = true; pl->axis = a; }
    }
    const bool gr = pl->graded;
    if (gr) { pl->spin[3] = pl->axis; pl->spin[1] = pl->axis % 3 + 1; pl->spin[2] = (pl->axis + 1) % 3 + 1; }
    int inv[4];
    for (int i = 0; i < 4; ++i) inv[pl->spin[i]] = i;
    const int NCm = gr ? 8 : 16, NM = gr ? 2 : 4, LM = NM * Ns;
    auto internal = [&](int c) { return idx_of(gr, inv[c >> 2], inv[c & 3]); };          // stored -> internal component
    auto position = [&](int r, int m) { return ((m >> 2) * Ns + r) * 4 + (m & 3); };
    auto used = [&](int c) { return !gr || even_comp(c, pl->axis); };
    pl->pack.assign((size_t)16 * Ns, make_int2(-1, -1));
    for (int c = 0; c < 16; ++c)
        for (int r = 0; r < Ns; ++r) {
            if (!used(c)) continue;
            pl->pack[c * Ns + r].x = position(r, internal(c));
            const int m = lat->swap_map16[r][c];
            int2& src = pl->pack[(m & 15) * Ns + lat->swap_r[r]];
            if (src.y >= 0) return false;   // the exchange is a permutation of the stored entries
            src.y = position(r, internal(c)) | ((m & 16) ? 1 << 30 : 0);
        }
    for (const int2& s : pl->pack)
        if ((s.x < 0) != (s.y < 0)) return false;
    pl->fmap.assign((size_t)Ns * NCm / 4, 0u);
    for (int r = 0; r < Ns; ++r)
        for (int c = 0; c < 16; ++c)
            if (used(c)) {
                const int m = lat->onsite_map16[r][c];
                const int to = internal(c);
                pl->fmap[(r * NCm + to) / 4] |= (unsigned)(internal(m & 15) | (m & 16)) << (8 * (to & 3));
            }
    // entries of every site by class (their two component maps); per class, component and inner index
    // the inner pair and the signed block entry
    int pair_id[16];
    for (int& x : pair_id) x = -1;
    struct Term { int k, at, sg; };
    using Maps = std::pair<sr::Map16, sr::Map16>;
    auto term = [&](const Maps& c, int mu, int nu, int l) {
        const int ma = c.first[pl->spin[mu] * 4 + pl->spin[l]], mb = c.second[pl->spin[l] * 4 + pl->spin[nu]];
        const int a = inv[(ma & 15) >> 2], ka = inv[ma & 3], kb = inv[(mb & 15) >> 2], b = inv[mb & 3];
        int& id = pair_id[ka * 4 + kb];
        if (id < 0) {
            pl->kap[pl->nk] = ka | (kb << 4);
            id = pl->nk++;
        }
        const int sg = sr::tri::coef_t(mu, nu, l) * ((ma & 16) ? -1 : 1) * ((mb & 16) ? -1 : 1);
        return Term{id, gr ? in_block(gr, a) * 2 + in_block(gr, b) : a * LM + b, sg};
    };
    std::vector<std::vector<std::vector<int>>> lists((size_t)Ns, std::vector<std::vector<int>>(NCm));
    for (int r = 0; r < Ns; ++r) {
        std::map<Maps, std::vector<std::pair<int, int>>> by;
        for (int e = lat->rpa_off[r]; e < lat->rpa_off[r + 1]; ++e)
            by[Maps(lat->rpa16[e].mA, lat->rpa16[e].mB)].push_back({lat->rpa16[e].rA, lat->rpa16[e].rB});
        for (auto& kv : by) {
            const int run = (int)pl->runs.size(), b = (int)pl->ent.size();
            if (gr) {
                for (auto& ab : kv.second) pl->ent.push_back((ab.first * Ns + ab.second) * 4);
                pl->runs.push_back(make_int2(b, (int)pl->ent.size()));
                for (int l = 0; l < 4; ++l) pl->run_pair.push_back(term(kv.first, l, l, l).k);
            }
            for (int m = 0; m < NCm; ++m)
                for (int l = 0; l < 4; ++l) {
                    const int mu = mu_of(gr, m), nu = nu_of(gr, m);
                    if (gr && !same_block(l, mu)) continue;
                    const Term t = term(kv.first, mu, nu, l);
                    const int neg = t.sg < 0 ? 1 << 30 : 0;
                    if (gr) lists[r][m].push_back(((run * 4 + l) * 4 + t.at) | neg);
                    else
                        for (auto& ab : kv.second)
                            lists[r][m].push_back((t.k * LM * LM + ab.first * 4 * LM + ab.second * 4 + t.at) | neg);
                }
        }
    }
    size_t most = 0;
    pl->n_terms.assign(Ns, 0);
    for (int r = 0; r < Ns; ++r) {
        pl->n_terms[r] = (int)lists[r][0].size();
        most = std::max(most, lists[r][0].size());
    }
    if (most * Ns * NCm > (size_t)1 << 28 || (size_t)16 * LM * LM >= (size_t)1 << 30) return false;
    pl->terms.assign(most * Ns * NCm, 0);
    for (int r = 0; r < Ns; ++r)
        for (int m = 0; m < NCm; ++m)
            for (size_t j = 0; j < lists[r][m].size(); ++j) pl->terms[(j * NCm + m) * Ns + r] = lists[r][m][j];
    return true;
}

inline bool build_plan(const sr_lattice* lat, Plan* pl) {
    try {
        return build_tables(lat, pl);
    } catch (...) {   // no memory for the lists: the general kernel needs none of them
        return false;
    }
}

}  // namespace trid
