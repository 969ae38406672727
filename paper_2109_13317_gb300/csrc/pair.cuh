// Vertex flow of the SU(2) and XYZ cores, FP64 and FP32-mixed (internal header, included by flow.cu
// after the shared device helpers).  Eq. frg:flowexplicit:2particle, one CTA per stored (s, u, t)
// triple.
//
// s and u channels.  A thread interpolates both rows of a site and multiplies them in registers,
// component by component: no shared memory but the descriptors, no barrier between nodes.  With
// A, B the rows and a, b, c the three spin components in turn, the projected products are
//     SU2  d: dA dB + 3 sA sB                    s: dA sB + sA dB -/+ 2 sA sB         (s / u channel)
//     XYZ  0: sum_c Ac Bc                        a: A0 Ba + Aa B0 -/+ (Ab Bc + Ac Bb)
// SU2 keeps sum dd, sum (ds + sd) and sum ss of each channel (four multiply-adds per node), XYZ the
// four components.  (The products are diagonal in the common eigenbasis of sigma^c sigma^c, one
// multiply-add per value; but a component is then a difference of eigenvalues, and one that is a
// factor smaller than the others loses that factor in precision.  Whole right-hand side in that form
// and in this one: square range 7 FP64 10.5 / 10.8 ms, pyrochlore range 6 FP32 8.2 / 8.4, Heisenberg-
// Kitaev range 5 FP64 2.9 / 3.1.)
// Their rows are stored site by site, so that a site's components come in one load; a row and its
// s <-> u image, which flips the sign of the density, share the storage (a weight set each for the
// density and the spin components).
// t channel.  Interpolated component rows go to shared memory for the lattice sum: register tiles of
// the dense contraction over pairs of sites (FP32; FP64 with many products) or a list of the
// distinct products (FP64, whose pipe allows no padding); on-site terms in registers.
// Lookups.  The arguments of the rows of a node are sums of x and four frequencies of the triple, so
// a node needs four interval searches per channel for its two to four rows.
//
// Measured (packing and vertex kernel, one GB300; before: the general FP64 kernel and the FP32 kernels on
// the stored state): square J1-J2 range 7, 48 frequencies, FP64 13.2 -> 10.7 ms, FP32 1.56 -> 1.02 ms;
// pyrochlore range 6, 64 frequencies, FP32 12.6 -> 8.3 ms; honeycomb Heisenberg-Kitaev range 5,
// 32 frequencies, FP64 3.65 -> 3.10 ms, FP32 0.60 -> 0.36 ms.
// What bounds it: FP64, the FP64 pipe (94 % busy on the square and the honeycomb lattice); FP32, the L1
// data path (87 % busy on the square lattice, 73 % on the pyrochlore: a corner chunk is one 16-byte load
// per 4 multiply-adds, and a row of 160 bytes touches two 128-byte lines).  Tried and dropped in FP32:
// corner chunks kept in registers over a run of nodes per group (1.69 ms against 1.27 at that stage:
// adjacent nodes no longer share their loads, the L1 hit rate falls from 62 to 14 %).  Taken: corners in
// parity slots with adjacent nodes in adjacent groups and descriptors stored as arrays (1.27 -> 1.03),
// on-site rows with both t corners in one load and lattice-sum terms merged with multiplicities (1.03 ->
// 0.98).  The t rows are packed apart from the s / u rows, component by component: read from the latter
// they would halve the packed state but cost FP32 2 % (a second weight set per row; pyrochlore 8.36 ->
// 8.56 ms), and the density's sign in the offset instead of that set costs the long rows more (8.65).
#pragma once

namespace pairk {

// Tables of one lattice and flow (device pointers).  The rows of a kind are addressed in chunks of 16
// bytes, so that 31 bits reach every mesh and lattice whose state's entries 31 bits count.
struct Tab {
    int nk;             // component pairs (row A, row B) of the lattice sum
    const int* kap;     // nk: cA | cB << 4
    const int* terms;   // [term][c * Ns + r]: offset into C (TILE) or product index (LIST) | multiplicity << 20
    const int* n_terms; // Ns
    const double* mult; // FP64: multiplicity as a value
    const int2* prod;   // LIST: offsets (row A, row B) of every product
    int nprod;
    long su_t;          // offset of the t rows [component][site]; the s / u rows [site][component] start the packed state
    long on;            // on-site rows, each with its successor in t: [triple][2][component]
    int ex_su, ex_t;    // distance of the exchanged rows in 16-byte chunks (0: the exchange is trivial)
    int rv, nst;        // stride of the s / u rows, sites of a t row (both padded)
    int nrow;           // stored triples
};

template <typename R> __host__ __device__ constexpr int vec() { return 16 / (int)sizeof(R); }   // values of a 16-byte chunk
template <typename R> __host__ __device__ constexpr int qrows() { return sizeof(R) == 4 ? 32 : 16; }   // t-channel nodes per block of rows
constexpr int kSU = 128;   // s and u nodes whose descriptors share a pass
constexpr int kT = 64;     // t nodes whose descriptors share a pass


// Unit of an s / u row: the values a thread takes, whole sites and whole 16-byte chunks.
template <typename R, int NC> __host__ __device__ constexpr int unit_values() { return vec<R>() > NC ? vec<R>() : NC; }
template <typename R, int NC> __host__ __device__ constexpr int unit_sites() { return unit_values<R, NC>() / NC; }
template <typename R, int NC> __host__ __device__ constexpr int units(int Ns) { return (Ns + unit_sites<R, NC>() - 1) / unit_sites<R, NC>(); }
constexpr int kAcc = 4;    // partial sums of a site in the s and u channels

// Descriptors in shared memory: arrays over the nodes of a pass (consecutive threads write
// consecutive nodes) of corner offsets and corner weights, per row, with a weight set for the density
// and one for the spin components.  The s / u rows in FP64 have the latter alone and the density's
// sign in bit 31 of the offset: its integer operations are free beside the FP64 pipe, and the shared
// memory decides how many CTAs of a small lattice are resident.
template <typename R> __host__ __device__ constexpr bool sign_in_offset() { return sizeof(R) == 8; }
template <typename R> __host__ __device__ constexpr size_t su_bytes() { return 2 * (16 + (sign_in_offset<R>() ? 4 : 8) * sizeof(R)) * kSU; }
template <typename R> __host__ __device__ constexpr size_t t_bytes() { return 2 * (16 + 8 * sizeof(R)) * kT; }

__host__ __device__ inline size_t r16(size_t b) { return (b + 15) & ~size_t(15); }

// Shared memory of a triple: mesh, then a region for descriptors and rows, reused at the end for the
// contraction's result and the threads' partial sums.
template <typename R, int NC>
__host__ __device__ inline size_t smem_bytes(int N, int Ns, int nst, size_t nC, int threads) {
    const int CH = units<R, NC>(Ns), NG = threads / CH, U = 2 * NC * nst / vec<R>(), S = threads / U;
    const size_t dsu = su_bytes<R>(), dt = t_bytes<R>() + sizeof(R) * 2 * NC * kT;
    const size_t work = r16(dt) + sizeof(R) * qrows<R>() * 2 * NC * nst;
    const size_t fin = r16(sizeof(R) * nC) + r16(sizeof(R) * NG * kAcc * CH * unit_sites<R, NC>()) + r16(sizeof(R) * 2 * S * NC * nst);
    const size_t a = work > dsu ? work : dsu;
    return r16(sizeof(R) * 2 * N) + (a > fin ? a : fin);
}

// Interval and weights of an argument x >= 0 (constant extrapolation outside the mesh).
// (step 0: a single corner, repeated under weight zero)
struct Axis32 { int k, step; float lo, hi; };
struct Axis64 { int k, step; double lo, hi; };
__device__ __forceinline__ Axis32 axis_of(const float* w, const float* ih, const Geo& g, float x) {
    const int N = g.N;
    const float xc = fminf(fmaxf(x, w[0]), w[N - 1]);
    int k = interval_guess(g, xc);
    while (k > 0 && xc < w[k]) --k;
    while (k < N - 2 && xc >= w[k + 1]) ++k;
    Axis32 a{k, 1, (w[k + 1] - xc) * ih[k], (xc - w[k]) * ih[k]};
    if (!(x < w[N - 1])) { a.k = N - 1; a.step = 0; a.lo = 1.0f; a.hi = 0.0f; }
    if (a.hi == 0.0f) { a.step = 0; a.lo = 1.0f; }
    return a;
}
// (comparisons on the bit patterns of non-negative values: the FP64 pipe is what bounds this kernel)
__device__ __forceinline__ Axis64 axis_of(const double* w, const double* ih, const Geo& g, double x) {
    const int N = g.N;
    const long long xb = __double_as_longlong(x);
    auto below = [&](int i) { return xb < __double_as_longlong(w[i]); };
    if (below(0) || xb == __double_as_longlong(w[0])) return {0, 0, 1.0, 0.0};
    if (!below(N - 1)) return {N - 1, 0, 1.0, 0.0};
    int k = interval_guess(g, (float)x);
    while (k > 0 && below(k)) --k;
    while (k < N - 2 && !below(k + 1)) ++k;
    const double hi = (x - w[k]) * ih[k];
    return {k, (__double_as_longlong(hi) & 0x7fffffffffffffffLL) != 0 ? 1 : 0, (w[k + 1] - x) * ih[k], hi};
}

__device__ __forceinline__ bool is_neg(float x) { return x < 0.0f; }
__device__ __forceinline__ bool is_neg(double x) {
    const long long b = __double_as_longlong(x);
    return b < 0 && (b & 0x7fffffffffffffffLL) != 0;
}
__device__ __forceinline__ float mag(float x) { return fabsf(x); }
__device__ __forceinline__ double mag(double x) { return __longlong_as_double(__double_as_longlong(x) & 0x7fffffffffffffffLL); }
__device__ __forceinline__ bool less(float a, float b) { return a < b; }
__device__ __forceinline__ bool less(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }   // a, b >= 0

// Four corners of a row: cells a, b along the two free axes, the third index exact.  EA: the exact
// axis (0 s, 1 t, 2 u); a, b are (t, u), (s, u) or (s, t).  flip: |s| < |u|.  Corner (i_s, j_t, k_u) is
// stored at the pair (max, min) of i_s, k_u; below the diagonal (and on it for a flipped lookup) the
// s <-> u relation flips the density's sign.  row: stride of a row in chunks.
// SLOTS (FP32, bound by the L1 path): a corner goes to the slot of its index parities.  Consecutive
// nodes share about half of their corners; in its slot a shared corner is read by the same load
// instruction for the adjacent nodes that a warp handles, as one access to its lines.
template <bool SLOTS, typename A, typename R>
__device__ __forceinline__ void corners(const int EA, const A& a, const A& b, int ex, bool flip, int N, int row, int (&off)[4],
                                        R (&w)[4], bool (&neg)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int ia = a.k + (k & 1) * a.step, ib = b.k + (k >> 1) * b.step;
        const int i = EA == 0 ? ex : ia, j = EA == 0 ? ia : (EA == 1 ? ex : ib), u = EA == 2 ? ex : ib;
        const int hi = max(i, u), lo = min(i, u);
        neg[k] = i < u || (i == u && flip);
        off[k] = ((hi * (hi + 1) / 2 + lo) * N + j) * row;
        w[k] = ((k & 1) ? a.hi : a.lo) * ((k >> 1) ? b.hi : b.lo);
    }
    if (SLOTS) {
        const bool qa = a.k & 1, qb = b.k & 1;
        auto swap2 = [](auto& x, auto& y) { const auto t = x; x = y; y = t; };
#pragma unroll
        for (int h = 0; h < 4; h += 2)
            if (qa) { swap2(off[h], off[h + 1]); swap2(w[h], w[h + 1]); swap2(neg[h], neg[h + 1]); }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (qb) { swap2(off[h], off[h + 2]); swap2(w[h], w[h + 2]); swap2(neg[h], neg[h + 2]); }
    }
}

__device__ __forceinline__ void ld16(const float* p, float* v) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void ld16(const double* p, double* v) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p));
    v[0] = a.x; v[1] = a.y;
}
__device__ __forceinline__ void lds16(const float* p, float* v) {
    const float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void lds16(const double* p, double* v) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    v[0] = a.x; v[1] = a.y;
}
__device__ __forceinline__ void st16(float* p, const float* v) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st16(double* p, const double* v) { *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]); }
// N consecutive values (a multiple of 16 bytes)
template <int N, typename R>
__device__ __forceinline__ void ld_n(const R* p, R* v) {
#pragma unroll
    for (int i = 0; i < N; i += vec<R>()) ld16(p + i, v + i);
}
__device__ __forceinline__ void lds_w(const float* p, float* v) { lds16(p, v); }
__device__ __forceinline__ void lds_w(const double* p, double* v) { lds16(p, v); lds16(p + 2, v + 2); }

__device__ __forceinline__ void st_w(float* p, const float* v) { st16(p, v); }
__device__ __forceinline__ void st_w(double* p, const double* v) { st16(p, v); st16(p + 2, v + 2); }

// Interpolated chunk: four corner chunks at o with the weights wt.
template <typename R>
__device__ __forceinline__ void interp(const R* __restrict__ P, const int4 o, const R* wt, R* v) {
    constexpr int V = vec<R>();
    R w[4], c[4][V];
    lds_w(wt, w);
    ld16(P + (long)o.x * V, c[0]);
    ld16(P + (long)o.y * V, c[1]);
    ld16(P + (long)o.z * V, c[2]);
    ld16(P + (long)o.w * V, c[3]);
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = fmadd(w[3], c[3][i], fmadd(w[2], c[2][i], fmadd(w[1], c[1][i], w[0] * c[0][i])));
}

// x with its sign changed where bit 31 of o is set
constexpr int kNeg = (int)0x80000000;
__device__ __forceinline__ float flip_sign(float x, int o) { return __int_as_float(__float_as_int(x) ^ (o & kNeg)); }
__device__ __forceinline__ double flip_sign(double x, int o) {
    return __hiloint2double(__double2hiint(x) ^ (o & kNeg), __double2loint(x));
}

// Interpolated unit of an s / u row; wt: weights of the spin components, wt + dens those of the density
// (FP64: their signs in the offsets).
template <typename R, int NC>
__device__ __forceinline__ void interp_unit(const R* __restrict__ P, const int4 o, const R* wt, int dens, R* v) {
    constexpr int VS = unit_values<R, NC>();
    R ws[4], wd[4], c[4][VS];
    const int of[4] = {o.x, o.y, o.z, o.w};
    lds_w(wt, ws);
    if constexpr (!sign_in_offset<R>()) lds_w(wt + dens, wd);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if constexpr (sign_in_offset<R>()) wd[k] = flip_sign(ws[k], of[k]);
        ld_n<VS>(P + (long)(sign_in_offset<R>() ? of[k] & ~kNeg : of[k]) * vec<R>(), c[k]);
    }
#pragma unroll
    for (int i = 0; i < VS; ++i) {
        const R* w = i % NC == 0 ? wd : ws;
        v[i] = fmadd(w[3], c[3][i], fmadd(w[2], c[2][i], fmadd(w[1], c[1][i], w[0] * c[0][i])));
    }
}

// Partial sums of a site plus the product of its rows a, b: SU2 sum dd, sum (ds + sd), sum ss of the s
// channel, sum ss of the u channel; XYZ the components.
template <bool S_CH, int NC, typename R>
__device__ __forceinline__ void su_products(const R* a, const R* b, R* acc) {
    if constexpr (NC == 2) {
        acc[0] = fmadd(a[0], b[0], acc[0]);
        acc[1] = fmadd(a[0], b[1], fmadd(a[1], b[0], acc[1]));
        acc[S_CH ? 2 : 3] = fmadd(a[1], b[1], acc[S_CH ? 2 : 3]);
    } else {
        acc[0] = fmadd(a[0], b[0], fmadd(a[1], b[1], fmadd(a[2], b[2], fmadd(a[3], b[3], acc[0]))));
#pragma unroll
        for (int c = 1; c < 4; ++c) {
            const int e = c % 3 + 1, f = e % 3 + 1;
            acc[c] = fmadd(a[0], b[c], fmadd(a[c], b[0], acc[c]));
            acc[c] = fmadd(S_CH ? -a[e] : a[e], b[f], fmadd(S_CH ? -a[f] : a[f], b[e], acc[c]));
        }
    }
}
// Component c from a site's partial sums.
template <int NC, typename R>
__device__ __forceinline__ R su_component(const R* acc, int c) {
    if constexpr (NC == 2) return c == 0 ? fmadd(R(3), acc[2] + acc[3], acc[0]) : fmadd(R(2), acc[3] - acc[2], acc[1]);
    else return acc[c];
}

// One stored frequency triple, all sites and components, written to dG (FP64).
// TILE: register tiles TM x TN of the dense contraction, NT per thread; LIST (TM = 1): NT products
// per thread.  Needs blockDim.x >= units(Ns) and >= 2 NC nst / V.
template <typename R, int NC, int TM, int TN, int NT>
__device__ __forceinline__ void triple(const Geo& g, const Tabs& tb, const Tab& td, const R* __restrict__ P,
                                       const R* __restrict__ nx, const R* __restrict__ nW, const int* __restrict__ ncount,
                                       double* __restrict__ dG, const int p, const int ti, unsigned char* smem) {
    constexpr int V = vec<R>(), QB = qrows<R>();
    constexpr bool LIST = TM == 1;
    const int tid = threadIdx.x, nth = blockDim.x, N = g.N, Ns = g.Ns;
    const int nst = td.nst, rt = NC * nst;
    R* wm = reinterpret_cast<R*>(smem);
    R* ih = wm + N;
    unsigned char* work = smem + r16(sizeof(R) * 2 * N);
    int si = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);   // guess, corrected below
    while ((si + 1) * (si + 2) / 2 <= p) ++si;
    while (si * (si + 1) / 2 > p) --si;
    const int ui = p - si * (si + 1) / 2;
    __syncthreads();   // shared memory of a previous triple (persistent callers) is consumed
    for (int i = tid; i < N; i += nth) {
        if constexpr (sizeof(R) == 4) { wm[i] = tb.wf[i]; ih[i] = i + 1 < N ? tb.invhf[i] : R(0); }
        else { wm[i] = tb.w[i]; ih[i] = i + 1 < N ? tb.invh[i] : R(0); }
    }
    __syncthreads();
    const R s = wm[si], t = wm[ti], u = wm[ui];
    const R w1p = (s + t + u) * R(0.5), w2p = (s - t - u) * R(0.5), w1 = (s - t + u) * R(0.5), w2 = (s + t - u) * R(0.5);

    // ---- s and u channels
    constexpr int VS = unit_values<R, NC>(), SPU = unit_sites<R, NC>();
    const int CH = units<R, NC>(Ns), NG = nth / CH, my_g = tid / CH, my_c = tid - my_g * CH;
    R psu[kAcc * SPU];
#pragma unroll
    for (int i = 0; i < kAcc * SPU; ++i) psu[i] = R(0);
    {
        int4* offs = reinterpret_cast<int4*>(work);                     // [row][node]
        R* wts = reinterpret_cast<R*>(work + 2 * 16 * kSU);             // [spin, density][row][node][corner]
        constexpr int kDens = 2 * 4 * kSU;
        const int cs = si, cu = 2 * N + ui, ns = ncount[cs], n_all = ns + ncount[cu];
        for (int n0 = 0; n0 < n_all; n0 += kSU) {
            const int nn = min(kSU, n_all - n0);
            if (n0 > 0) __syncthreads();
            for (int i = tid; i < nn; i += nth) {
                const bool is_s = n0 + i < ns;
                const size_t at = is_s ? (size_t)cs * g.nmax + n0 + i : (size_t)cu * g.nmax + (n0 + i - ns);
                const R x = nx[at], W = nW[at];
                // row A: (s, w1p - x, x - w2p), B: (s, x - w1, x - w2);  u: (w1 + x, x - w2p, u), (w1p + x, w2 - x, u)
                const R a0 = is_s ? w1p - x : w1 + x, a1 = x - w2p, b0 = is_s ? x - w1 : w1p + x, b1 = is_s ? x - w2 : w2 - x;
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    const R y0 = r ? b0 : a0, y1 = r ? b1 : a1, m0 = mag(y0), m1 = mag(y1);
                    auto c0 = axis_of(wm, ih, g, m0);
                    const auto c1 = axis_of(wm, ih, g, m1);
                    if (r == 0) { c0.lo *= W; c0.hi *= W; }   // the node weight rides on row A
                    const bool swap = is_s ? is_neg(y1) : is_neg(y0);
                    const int so = swap ? td.ex_su : 0;
                    const bool flip = is_s ? less(s, m1) : less(m0, u);
                    int off[4];
                    R wt[4];
                    bool neg[4];
                    corners<sizeof(R) == 4>(is_s ? 0 : 2, c0, c1, is_s ? si : ui, flip, N, td.rv / V, off, wt, neg);
                    if constexpr (!sign_in_offset<R>()) {
                        R wd[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) wd[k] = neg[k] ? -wt[k] : wt[k];
                        st_w(wts + kDens + 4 * (r * kSU + i), wd);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) off[k] += so + (sign_in_offset<R>() && neg[k] ? kNeg : 0);
                    offs[r * kSU + i] = make_int4(off[0], off[1], off[2], off[3]);
                    st_w(wts + 4 * (r * kSU + i), wt);
                }
            }
            __syncthreads();
            if (my_g < NG) {
                // adjacent groups, in one warp, take adjacent nodes
                const R* Pc = P + my_c * VS;
                const int e = min(max(ns - n0, 0), nn);
                auto channel = [&](auto is_s, int i0, int i1) {
                    for (int i = i0 + my_g; i < i1; i += NG) {
                        R a[VS], b[VS];
                        interp_unit<R, NC>(Pc, offs[i], wts + 4 * i, kDens, a);
                        interp_unit<R, NC>(Pc, offs[kSU + i], wts + 4 * (kSU + i), kDens, b);
#pragma unroll
                        for (int j = 0; j < SPU; ++j) su_products<decltype(is_s)::value, NC>(a + j * NC, b + j * NC, psu + j * kAcc);
                    }
                };
                channel(std::true_type{}, 0, e);
                channel(std::false_type{}, e, nn);
            }
        }
    }
    __syncthreads();

    // ---- t channel: unit (row, chunk of 16 bytes) of a stream of nodes
    const int CT = rt / V, U = 2 * CT, S = nth / U, stream = tid / U, unit = tid - stream * U;
    const int rw = unit / CT, ct = unit - rw * CT, comp = ct * V / nst, site0 = ct * V - comp * nst;
    const bool in_stream = stream < S;
    int4* offs = reinterpret_cast<int4*>(work);                     // [row][node]
    R* wts = reinterpret_cast<R*>(work + 2 * 16 * kT);              // [row][density, spin][node][corner]
    R* fac = reinterpret_cast<R*>(work + t_bytes<R>());             // [node][C, D][component]
    R* rows = reinterpret_cast<R*>(work + r16(t_bytes<R>() + sizeof(R) * 2 * NC * kT));
    R pt[V];
    int pon[V];   // component of the on-site factor of the unit's sites
#pragma unroll
    for (int i = 0; i < V; ++i) {
        pt[i] = R(0);
        pon[i] = (NC == 4 && rw == 0 && site0 + i < Ns) ? perm_of(tb.onsite_perm[site0 + i], comp) : comp;
    }
    // contraction tiles / products of this thread
    const int tm = nst / (LIST ? 1 : TM), tn = nst / (LIST ? 1 : TN), ntile = LIST ? td.nprod : td.nk * tm * tn;
    int ta[NT], tbo[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int id = tid + j * nth;
        ta[j] = -1;
        tbo[j] = 0;
        if (id < ntile) {
            if (LIST) {
                const int2 pr = td.prod[id];
                ta[j] = pr.x;
                tbo[j] = rt + pr.y;
            } else {
                const int k = id / (tm * tn), rem = id - k * (tm * tn), a = rem / tn, b = rem - a * tn;
                ta[j] = (td.kap[k] & 15) * nst + a * TM;
                tbo[j] = rt + (td.kap[k] >> 4) * nst + b * TN;
            }
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
        const R* Pt = P + td.su_t;
        const int cidx = N + ti, nq = ncount[cidx];
        for (int n0 = 0; n0 < nq; n0 += kT) {
            const int nn = min(kT, nq - n0);
            if (n0 > 0) __syncthreads();
            for (int i = tid; i < nn; i += nth) {
                const size_t at = (size_t)cidx * g.nmax + n0 + i;
                const R x = nx[at], W = nW[at];
                // A: (w1 + x, t, w1p - x), B: (x + w2p, t, x - w2); on-site C: (w2p + x, w2 - x, -t) and
                // D: (w1 + x, x - w1p, -t) search the same magnitudes
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    const R y0 = r ? x + w2p : w1 + x, y1 = r ? x - w2 : w1p - x, m0 = mag(y0), m1 = mag(y1);
                    const auto c0 = axis_of(wm, ih, g, m0), c1 = axis_of(wm, ih, g, m1);
                    const bool swap = is_neg(y0) != is_neg(y1);
                    const int so = swap ? td.ex_t : 0;
                    auto cw = c0;
                    if (r == 0) { cw.lo *= W; cw.hi *= W; }   // the node weight rides on row A
                    int off[4];
                    R wt[4], wd[4];
                    bool neg[4];
                    corners<sizeof(R) == 4>(1, cw, c1, ti, less(m0, m1), N, rt / V, off, wt, neg);
#pragma unroll
                    for (int k = 0; k < 4; ++k) wd[k] = neg[k] ? -wt[k] : wt[k];
                    offs[r * kT + i] = make_int4(off[0] + so, off[1] + so, off[2] + so, off[3] + so);
                    st_w(wts + 4 * ((2 * r) * kT + i), wd);
                    st_w(wts + 4 * ((2 * r + 1) * kT + i), wt);
                    // on-site row at (m0, m1, t) (its own exchange): C from row B's searches, D from
                    // row A's, with the node weight; stored as its factor sum_k s(k, c) X_k
                    // (one load gives both t corners: the table holds each row with its successor in t)
                    R v[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[c] = R(0);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int is = cw.k + k * cw.step, hi = max(is, ti), lo = min(is, ti);
                        const bool dneg = is < ti || (is == ti && less(m0, t));
                        R x2[2 * NC];
                        ld_n<2 * NC>(P + td.on + (size_t)((hi * (hi + 1) / 2 + lo) * N + c1.k) * 2 * NC, x2);
                        const R ws = k ? cw.hi : cw.lo, wl = ws * c1.lo, wh = ws * c1.hi;
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            const R y = c1.step ? x2[NC + c] : x2[c];
                            v[c] = fmadd(c == 0 && dneg ? -wl : wl, x2[c], v[c]);
                            v[c] = fmadd(c == 0 && dneg ? -wh : wh, y, v[c]);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < NC; ++c) fac[(2 * i + (r ^ 1)) * NC + c] = onsite_factor<R, NC>(v, c);
                }
            }
            __syncthreads();
            for (int q0 = 0; q0 < nn; q0 += QB) {
                const int qn = min(QB, nn - q0);
                if (q0 > 0) __syncthreads();
                if (in_stream) {
                    const R* Pc = Pt + ct * V;
                    const R* wr = wts + 4 * (2 * rw + (comp == 0 ? 0 : 1)) * kT;
                    for (int q = stream; q < qn; q += S) {
                        R v[V];
                        interp(Pc, offs[rw * kT + q0 + q], wr + 4 * (q0 + q), v);
                        // on-site terms: A_c F_c(C) (row A), F_c(D) B_c (row B)
                        const R* f = fac + (2 * (q0 + q) + rw) * NC;
#pragma unroll
                        for (int j = 0; j < V; ++j) pt[j] = fmadd(v[j], f[pon[j]], pt[j]);
                        st16(rows + (q * 2 + rw) * rt + ct * V, v);
                    }
                }
                __syncthreads();
                // lattice sum
                if constexpr (LIST) {
#pragma unroll 1
                    for (int q = 0; q < qn; ++q) {
                        const R* r = rows + 2 * q * rt;
#pragma unroll
                        for (int j = 0; j < NT; ++j)
                            if (ta[j] >= 0) acc[j][0][0] = fmadd(r[ta[j]], r[tbo[j]], acc[j][0][0]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < NT; ++j)
                        if (ta[j] >= 0) {
                            const R* A = rows + ta[j];
                            const R* B = rows + tbo[j];
#pragma unroll 2
                            for (int q = 0; q < qn; ++q) {
                                R a[TM], b[TN];
#pragma unroll
                                for (int x = 0; x < TM; x += V) lds16(A + 2 * q * rt + x, a + x);
#pragma unroll
                                for (int x = 0; x < TN; x += V) lds16(B + 2 * q * rt + x, b + x);
#pragma unroll
                                for (int x = 0; x < TM; ++x)
#pragma unroll
                                    for (int y = 0; y < TN; ++y) acc[j][x][y] = fmadd(a[x], b[y], acc[j][x][y]);
                            }
                        }
                }
            }
        }
    }
    // ---- outputs: partial sums and the contraction's result through shared memory, fixed order
    __syncthreads();
    const size_t nC = LIST ? (size_t)td.nprod : (size_t)td.nk * nst * nst;
    R* C = reinterpret_cast<R*>(work);
    const int nsu = kAcc * SPU * CH;
    R* su = reinterpret_cast<R*>(work + r16(sizeof(R) * nC));                              // [group][site][kAcc]
    R* tt = reinterpret_cast<R*>(work + r16(sizeof(R) * nC) + r16(sizeof(R) * NG * nsu));     // [stream][row][rt]
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int id = tid + j * nth;
        if (id < ntile) {
            if constexpr (LIST) C[id] = acc[j][0][0];
            else {
                const int k = id / (tm * tn), rem = id - k * (tm * tn), a = (rem / tn) * TM, b = (rem % tn) * TN;
#pragma unroll
                for (int x = 0; x < TM; ++x)
#pragma unroll
                    for (int y = 0; y < TN; y += V) st16(C + (k * nst + a + x) * nst + b + y, &acc[j][x][y]);
            }
        }
    }
    if (my_g < NG) {
#pragma unroll
        for (int i = 0; i < kAcc * SPU; i += V) st16(su + my_g * nsu + my_c * kAcc * SPU + i, psu + i);
    }
    if (in_stream) st16(tt + (2 * stream + rw) * rt + ct * V, pt);
    __syncthreads();
    // FP64 and long rows: the sums over groups and streams first, a value each (into the slots of the
    // first group and stream), instead of every output summing the values it mixes (with eigenvalue rows:
    // square range 7 FP64 11.85 -> 11.70 ms, pyrochlore FP32 8.39 -> 8.18; the short FP32 rows lose 3 % by
    // the barrier)
    constexpr bool kStage = sizeof(R) == 8 || TM == 8;
    if constexpr (kStage) {
        for (int v = tid; v < nsu + rt; v += nth) {
            if (v < nsu) {
                R a = su[v];
                for (int k = 1; k < NG; ++k) a += su[k * nsu + v];
                su[v] = a;
            } else {
                R a = tt[v - nsu];
                for (int k = 1; k < 2 * S; ++k) a += tt[k * rt + v - nsu];
                tt[v - nsu] = a;
            }
        }
        __syncthreads();
    }
    for (int o = tid; o < NC * Ns; o += nth) {
        const int c = o / Ns, r = o - c * Ns;
        R x[kAcc], a = tt[c * nst + r], l = R(0);
#pragma unroll
        for (int e = 0; e < kAcc; ++e) x[e] = su[r * kAcc + e];
        if constexpr (!kStage)
            for (int k = 1; k < NG; ++k)
#pragma unroll
                for (int e = 0; e < kAcc; ++e) x[e] += su[k * nsu + r * kAcc + e];
        if constexpr (!kStage)
            for (int k = 1; k < 2 * S; ++k) a += tt[k * rt + c * nst + r];
        const int nt = td.n_terms[r];
#pragma unroll 4
        for (int k = 0; k < nt; ++k) {
            const int code = td.terms[k * NC * Ns + o];
            R m;
            if constexpr (sizeof(R) == 8) m = __ldg(td.mult + (code >> 20));   // (a conversion would run on the FP64 pipe)
            else m = (R)(code >> 20);
            l = fmadd(m, C[code & 0xfffff], l);
        }
        a += su_component<NC, R>(x, c);
        dG[((size_t)(p * N + ti) * NC + c) * Ns + r] = (double)a - 2.0 * (double)l;
    }
}

template <typename R, int NC, int TM, int TN, int NT, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
k_gamma_rhs_pair(Geo g, Tabs tb, Tab td, const R* __restrict__ P, const R* __restrict__ nx, const R* __restrict__ nW,
                 const int* __restrict__ ncount, double* __restrict__ dG, int p0) {
    extern __shared__ __align__(16) unsigned char smem[];
    triple<R, NC, TM, TN, NT>(g, tb, td, P, nx, nW, ncount, dG, p0 + (int)(blockIdx.x / g.N), blockIdx.x % g.N, smem);
}

// Packed state: s / u rows and t rows of every stored triple, and the same of the exchanged pairs when
// the site exchange is not trivial (the padding stays zero).  A block takes whole rows, staged in
// shared memory, so that a component is read and converted once; kPackThreads threads, grid-stride
// over the rows.
constexpr int kPackThreads = 256;
template <typename R, int NC> __host__ __device__ constexpr size_t pack_smem(int Ns) {
    return sizeof(R) * NC * (kPackThreads > Ns ? kPackThreads : Ns);
}

template <typename R, int NC>
__device__ __forceinline__ void pack_rows(const Geo& g, const Tabs& tb, const Tab& td, const double* __restrict__ G,
                                          R* __restrict__ P, unsigned char* smem) {
    const int Ns = g.Ns, RB = max(1, kPackThreads / Ns), cap = RB * Ns;   // rows of a block, their sites
    R* sh = reinterpret_cast<R*>(smem);                                   // [component][site]
    const bool small = Ns <= kPackThreads;
    const int my_row = small ? (int)threadIdx.x / Ns : 0, first = small ? (int)threadIdx.x - my_row * Ns : (int)threadIdx.x;
    for (int row0 = blockIdx.x * RB; row0 < td.nrow; row0 += gridDim.x * RB) {
        const int row = row0 + my_row;
        const bool on = my_row < RB && row < td.nrow;
        const double* src = G + (size_t)row * NC * Ns;
        for (int r = first; on && r < Ns; r += kPackThreads)
#pragma unroll
            for (int c = 0; c < NC; ++c) sh[c * cap + my_row * Ns + r] = (R)src[c * Ns + r];
        __syncthreads();
        for (int r = first; on && r < Ns; r += kPackThreads)
            for (int x = 0; x < (td.ex_t ? 2 : 1); ++x) {
                const int rs = my_row * Ns + (x ? tb.swap_r[r] : r), pm = x ? tb.swap_perm[r] : 0xe4;
                R v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) v[c] = sh[perm_of(pm, c) * cap + rs];
                R* ps = P + (size_t)(x ? td.ex_su : 0) * vec<R>() + (size_t)row * td.rv + r * NC;
                R* pt = P + td.su_t + (size_t)(x ? td.ex_t : 0) * vec<R>() + (size_t)row * NC * td.nst + r;
                if constexpr (NC * sizeof(R) >= 16) {
#pragma unroll
                    for (int c = 0; c < NC; c += vec<R>()) st16(ps + c, v + c);
                } else {
                    *reinterpret_cast<float2*>(ps) = make_float2(v[0], v[1]);
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    pt[c * td.nst] = v[c];
                    if (x == 0 && r == 0) {
                        R* o = P + td.on + (size_t)row * 2 * NC + c;
                        const int ti = row % g.N;
                        o[0] = v[c];
                        if (ti > 0) o[-NC] = v[c];
                        if (ti == g.N - 1) o[NC] = v[c];
                    }
                }
            }
        __syncthreads();
    }
}

template <typename R, int NC>
__global__ void __launch_bounds__(kPackThreads) k_pair_pack(Geo g, Tabs tb, Tab td, const double* __restrict__ G, R* __restrict__ P) {
    extern __shared__ __align__(16) unsigned char smem[];
    pack_rows<R, NC>(g, tb, td, G, P, smem);
}

// ---- host side

template <typename R>
using Kernel = void (*)(Geo, Tabs, Tab, const R*, const R*, const R*, const int*, double*, int);

// Kernel variants: X(id, NC, TM, TN, NT, largest CTA, resident CTAs of that size its registers allow,
// multiple the sites of a t row are padded to).  FP32 tiles of 8 x 4 instead of 4 x 4 save
// operand loads once the rows are long (pyrochlore: one tile on 160 threads 8.0 ms, two on 96 9.7 ms);
// up to 20 sites 4 x 4 tiles fill 64 threads.  FP64 lists have no padding, tiles take over where the
// products exceed eight per thread; their registers are capped for six CTAs of 128 threads (square range
// 7: five 11.7 ms, six 10.5, seven and eight 10.5; 13 products on 64 threads 11.3; 160 threads 12.8).
// (These times are of the eigenvalue form named above, 2 % faster throughout.)
#define PAIR_F32_VARIANTS(X)     \
    X(0, 2, 4, 4, 1, 64, 12, 4)  \
    X(1, 2, 8, 4, 1, 160, 5, 8)  \
    X(2, 2, 8, 4, 2, 192, 3, 8)  \
    X(3, 2, 8, 4, 4, 384, 1, 8)  \
    X(4, 4, 4, 4, 1, 96, 8, 4)   \
    X(5, 4, 4, 4, 2, 192, 3, 4)  \
    X(6, 4, 4, 4, 4, 384, 1, 4)
#define PAIR_F64_VARIANTS(X)     \
    X(0, 2, 1, 1, 2, 64, 12, 2)  \
    X(1, 2, 1, 1, 8, 128, 6, 2)  \
    X(2, 2, 2, 2, 5, 256, 2, 2)  \
    X(3, 2, 2, 2, 10, 256, 2, 2) \
    X(4, 4, 1, 1, 2, 64, 10, 2)  \
    X(5, 4, 1, 1, 8, 256, 2, 2)

struct Variant { int nc, tm, tn, nt, max_threads, pad; };
#define PAIR_ROW(id, NC, TM, TN, NT, MAXT, MINB, PAD) {NC, TM, TN, NT, MAXT, PAD},
inline const Variant kF32[] = {PAIR_F32_VARIANTS(PAIR_ROW)};
inline const Variant kF64[] = {PAIR_F64_VARIANTS(PAIR_ROW)};
#undef PAIR_ROW

inline Kernel<float> kernel_f32(int id) {
#define PAIR_CASE(id, NC, TM, TN, NT, MAXT, MINB, PAD) \
    case id: return k_gamma_rhs_pair<float, NC, TM, TN, NT, MAXT, MINB>;
    switch (id) { PAIR_F32_VARIANTS(PAIR_CASE) }
#undef PAIR_CASE
    return nullptr;
}
inline Kernel<double> kernel_f64(int id) {
#define PAIR_CASE(id, NC, TM, TN, NT, MAXT, MINB, PAD) \
    case id: return k_gamma_rhs_pair<double, NC, TM, TN, NT, MAXT, MINB>;
    switch (id) { PAIR_F64_VARIANTS(PAIR_CASE) }
#undef PAIR_CASE
    return nullptr;
}

// Host tables and the kernel variant of a flow.
struct Plan {
    int variant = -1, threads = 0;
    size_t smem = 0;
    long size = 0;   // values of the packed state
    Tab td{};
    std::vector<int> terms, n_terms, kap;
    std::vector<int2> prod;
    std::vector<double> mult;
};

// The first variant of the core whose tiles (or products) and rows fit its CTA.
template <typename R>
inline bool choose(const Variant* v, int count, int N, int Ns, int nc, int nk, int nprod, Plan* pl) {
    constexpr int V = vec<R>();
    for (int i = 0; i < count; ++i) {
        if (v[i].nc != nc) continue;
        const int nst = (Ns + v[i].pad - 1) / v[i].pad * v[i].pad;
        // (FP64: the rows of both layouts have one stride, see pair_adj.cuh)
        const int CH = nc == 2 ? units<R, 2>(Ns) : units<R, 4>(Ns);
        const int rv = sizeof(R) == 8 ? nc * nst : CH * (nc == 2 ? unit_values<R, 2>() : unit_values<R, 4>());
        const bool list = v[i].tm == 1;
        const long T = list ? nprod : (long)nk * (nst / v[i].tm) * (nst / v[i].tn);
        const long need = std::max(std::max((T + v[i].nt - 1) / v[i].nt, (long)CH), 2L * nc * nst / V);
        const int th = (int)std::max(64L, (need + 31) / 32 * 32);
        if (th > v[i].max_threads) continue;
        const size_t nC = list ? (size_t)nprod : (size_t)nk * nst * nst;
        const size_t sm = nc == 2 ? smem_bytes<R, 2>(N, Ns, nst, nC, th) : smem_bytes<R, 4>(N, Ns, nst, nC, th);
        if (sm > 227 * 1024) continue;
        pl->variant = i;
        pl->threads = th;
        pl->smem = sm;
        pl->td.rv = rv;
        pl->td.nst = nst;
        return true;
    }
    return false;
}

// Tables of a lattice (SU2 / XYZ) for FP32 (fp32) or FP64 rows; false when no variant fits.
inline bool build_tables(const sr_lattice* lat, int N, bool fp32, bool has_swap, const std::vector<int2>& prods,
                         const std::vector<int>& goff, const std::vector<int>& gidx, Plan* pl) {
    const int nc = lat->nc, Ns = lat->Ns;
    Tab& td = pl->td;
    int pair_id[16];
    for (int& x : pair_id) x = -1;
    for (const int2& p : prods) {
        int& id = pair_id[(p.x % nc) * 4 + p.y % nc];
        if (id >= 0) continue;
        if (td.nk == 10) return false;
        pl->kap.push_back((p.x % nc) | ((p.y % nc) << 4));
        id = td.nk++;
    }
    td.nprod = (int)prods.size();
    const bool ok = fp32 ? choose<float>(kF32, sizeof(kF32) / sizeof(kF32[0]), N, Ns, nc, td.nk, td.nprod, pl)
                         : choose<double>(kF64, sizeof(kF64) / sizeof(kF64[0]), N, Ns, nc, td.nk, td.nprod, pl);
    if (!ok) return false;
    const Variant& v = fp32 ? kF32[pl->variant] : kF64[pl->variant];
    const long nrow = (long)N * (N + 1) / 2 * N, ex = has_swap ? 2 : 1;
    const long V = fp32 ? vec<float>() : vec<double>(), rt = (long)nc * td.nst;
    if (ex * nrow * std::max((long)td.rv, rt) / V >= (1L << 31)) return false;   // 31-bit chunk offsets
    pl->size = ex * nrow * (td.rv + rt) + 2 * nc * nrow;
    td.nrow = (int)nrow;
    td.ex_su = has_swap ? (int)(nrow * td.rv / V) : 0;
    td.ex_t = has_swap ? (int)(nrow * rt / V) : 0;
    td.su_t = ex * nrow * td.rv;
    td.on = ex * nrow * (td.rv + rt);
    if (v.tm == 1)
        for (const int2& p : prods)
            pl->prod.push_back(make_int2(p.x % nc * td.nst + p.x / nc, p.y % nc * td.nst + p.y / nc));
    // terms of every output: its distinct products with their multiplicities
    std::vector<std::vector<int>> lists((size_t)nc * Ns);
    std::vector<int> at;
    size_t most = 0;
    int top = 0;
    pl->n_terms.assign(Ns, 0);
    for (int r = 0; r < Ns; ++r)
        for (int c = 0; c < nc; ++c) {
            at.clear();
            for (int k = goff[r * nc + c]; k < goff[r * nc + c + 1]; ++k) {
                const int2 p = prods[gidx[k]];
                at.push_back(v.tm == 1 ? gidx[k] : (pair_id[(p.x % nc) * 4 + p.y % nc] * td.nst + p.x / nc) * td.nst + p.y / nc);
            }
            std::sort(at.begin(), at.end());
            std::vector<int>& l = lists[(size_t)c * Ns + r];
            for (size_t i = 0, j; i < at.size(); i = j) {
                for (j = i; j < at.size() && at[j] == at[i]; ++j) {}
                if (at[i] >= 1 << 20 || j - i > 2047) return false;
                l.push_back(at[i] | (int)(j - i) << 20);
                top = std::max(top, (int)(j - i));
            }
            pl->n_terms[r] = std::max(pl->n_terms[r], (int)l.size());
            most = std::max(most, l.size());
        }
    for (int i = 0; i <= top; ++i) pl->mult.push_back(i);
    pl->terms.assign(most * nc * Ns, 0);   // (multiplicity 0 where a component has fewer)
    for (size_t o = 0; o < lists.size(); ++o)
        for (size_t j = 0; j < lists[o].size(); ++j) pl->terms[j * nc * Ns + o] = lists[o][j];
    return true;
}

inline bool build_plan(const sr_lattice* lat, int N, bool fp32, bool has_swap, const std::vector<int2>& prods,
                       const std::vector<int>& goff, const std::vector<int>& gidx, Plan* pl) {
    try {
        return build_tables(lat, N, fp32, has_swap, prods, goff, gidx, pl);
    } catch (...) {   // no memory for the lists: the general kernel needs none of them
        return false;
    }
}

}  // namespace pairk
