// The coarse end of the V-cycle in one launch (included by cfp_mg.cu, inside
// its namespaces): every level from the first of at most kCoarseMaxNodes nodes
// down to the coarsest and back up -- smoothing, red residual, restriction,
// the coarsest level's 16 sweeps, prolongation, smoothing -- on one
// thread-block cluster, with the levels in shared memory.
// Where a level's share, with the rows copied from either side, is more than
// kCoarseSmem (FP64, some flat levels: 68 x 54 x 17, 87 x 65 x 9; 0.5 % of the
// grids of 33 to 449 nodes per axis) the list begins one level further down and
// that level runs one launch per pass (V(2,2) of 135 x 107 x 33 217 us, 345 x
// 254 x 33 551; 757 and 1010 when only its smoothing was a cluster's).
//
// These levels hold too few nodes to fill the GPU: a pass over one costs its
// latency, one launch per pass or a CTA working in L2 alike.  Shared memory
// and one launch cut that latency: below 257^3 (33^3, 17^3 and 9^3, V(2,2),
// FP32) eleven launches took 95 us and this one takes 60; below 33^3 in FP64
// a V-cycle of 258 us takes 117.
//
// A level's rows (row R = k n_y + j) are dealt to the CTAs in equal runs of
// rpc > n_y rows.  A CTA keeps copies of the n_y + 1 rows on either side of
// its run, so that every neighbour is a local shared load; whoever updates a node
// of those rows stores it into the neighbour's copy as well (distributed
// shared memory), and a cluster barrier ends each pass.  A level of at most
// kCoarseSolo nodes, for which the barrier would cost more than the
// arithmetic, belongs to CTA 0 alone (fewer nodes in FP64, whose issue rate
// per SM is 1/64 of FP32's).  Per row and colour: the iterate, b and the
// reciprocal diagonal (0 off the unknowns: it stands for the type).  The red
// residual takes the place of the red iterate, which the next red half-sweep
// overwrites without reading.  A thread's nodes are the same in every pass;
// their indices are worked out once (integer divisions cost more than the
// update itself).
// The arithmetic is that of the kernels below (rb_rest, times_rcp / times_rd,
// restrict_sum, prolong_value), so the result is bitwise theirs.
constexpr int kCoarseThreads = 512;
constexpr int64_t kCoarseMaxNodes = int64_t(1) << 16;  // 33^3, 40^3; 65^3 does not fit 16 SMs' shared memory
constexpr int kCoarseLevels = 4;
constexpr int kCoarseSmem = 216 * 1024;
template <class T>
constexpr int64_t kCoarseSolo = sizeof(T) == 4 ? 6000 : 1500;

template <class T>
struct CoarseLevel {
    SLev<T> L;       // the level's global arrays and tables
    Transfer<T> X;   // transfers with the next level of the list
    int hps, mp;     // entries per row of one colour in shared memory; pairs with an interior node
    int rows, rpc;   // rows in all, rows per CTA (solo: all)
    int halo;        // shared: n_y + 1 rows either side; solo: 0
    int dist;        // 0: CTA 0 alone
    float inv_hps, inv_mp, inv_ny, inv_rpc;
    unsigned vec;    // e0 e1 ((rpc + 2 halo) x hps each) b0 b1 rd0 rd1 (rpc x hps), in elements of T from the start
    unsigned cof;    // packed coefficients x, y, z, in PkT<T> from the start
    unsigned itm;    // the pairs' indices (CoarseItem), in 8 bytes from the start
};
template <class T>
struct CoarseArgs {
    CoarseLevel<T> V[kCoarseLevels];
    int nl, ndist, pre, post;
};
struct __align__(8) CoarseItem {  // a pair: its entry in the CTA's rows, m, and its row's j, k
    unsigned short o, m, j, k;
};

// n / d for 0 <= n < 2^20 with inv = 1.0f / d: (n + 1/2) / d is at least 1 / (2 d)
// from an integer, far more than its rounding
__device__ __forceinline__ int fast_div(int n, float inv) { return (int)(((float)n + 0.5f) * inv); }

// This CTA's part of a level, every address and count worked out once (a
// pass must not go back to the kernel's parameters: their loads, indexed by
// the level, cost more than the pass).
template <class T>
struct CoarseView {
    T *e[2], *b[2], *rd[2];            // entry 0 of the CTA's own rows
    const PkT<T>*cx, *cy, *cz;
    CoarseItem* items;
    int n;                             // pairs this CTA updates: of its rows; a solo level's interior rows only
    int R0, cnt, rpc, dist;            // its rows; rows per CTA
    int nx, ny, nz, hps, mp;
    int olo, ohi;                      // entries below olo / from ohi on are copied by the CTA before / after
    T *lo[2], *hi[2];                  // e there, so that the entry index is the same (null: none)
    float inv_ny, inv_rpc;
    // row R of one of the vectors above, in whichever CTA owns it
    __device__ __forceinline__ T* row(T* v, int R) const {
        const int q = R - R0;
        if ((unsigned)q < (unsigned)cnt) return v + q * hps;
        const int own = dist ? fast_div(R, inv_rpc) : 0;
        return cooperative_groups::this_cluster().map_shared_rank(v, own) + (R - own * rpc) * hps;
    }
    // stores v at entry o of e[c], and into the neighbours' copies of that row
    template <bool DIST>
    __device__ __forceinline__ void put(int c, int o, T v) const {
        e[c][o] = v;
        if (DIST && o < olo && lo[c]) lo[c][o] = v;
        if (DIST && o >= ohi && hi[c]) hi[c][o] = v;
    }
};

template <class T>
__device__ __forceinline__ CoarseView<T> coarse_view(const CoarseLevel<T>& V, unsigned char* raw, int rank) {
    CoarseView<T> C;
    C.nx = V.L.nx;
    C.ny = V.L.ny;
    C.nz = V.L.nz;
    C.hps = V.hps;
    C.mp = V.mp;
    C.rpc = V.rpc;
    C.dist = V.dist;
    C.inv_ny = V.inv_ny;
    C.inv_rpc = V.inv_rpc;
    C.R0 = V.dist ? rank * V.rpc : 0;
    C.cnt = V.dist ? max(0, min(V.rpc, V.rows - C.R0)) : (rank == 0 ? V.rows : 0);
    C.n = V.dist ? C.cnt * V.mp : C.cnt ? (C.ny - 2) * (C.nz - 2) * V.mp : 0;
    const int run = V.rpc * V.hps, es = run + 2 * V.halo * V.hps;
    T* vec = reinterpret_cast<T*>(raw) + V.vec;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        C.e[c] = vec + c * es + V.halo * V.hps;
        C.b[c] = vec + 2 * es + c * run;
        C.rd[c] = vec + 2 * es + (2 + c) * run;
        C.lo[c] = C.hi[c] = nullptr;
        if (V.dist) {
            if (rank > 0) C.lo[c] = cooperative_groups::this_cluster().map_shared_rank(C.e[c], rank - 1) + run;
            if (C.R0 + V.rpc < V.rows)
                C.hi[c] = cooperative_groups::this_cluster().map_shared_rank(C.e[c], rank + 1) - run;
        }
    }
    C.olo = V.halo * V.hps;
    C.ohi = run - V.halo * V.hps;
    C.cx = reinterpret_cast<const PkT<T>*>(raw) + V.cof;
    C.cy = C.cx + C.nx;
    C.cz = C.cy + C.ny;
    C.items = reinterpret_cast<CoarseItem*>(raw) + V.itm;
    return C;
}

// barrier between passes over a level
template <bool DIST>
__device__ __forceinline__ void coarse_sync() {
    if (DIST) cooperative_groups::this_cluster().sync();
    else __syncthreads();
}

// one half-sweep of COLOUR (from_zero: the other colour is zero), or, RESID,
// the red residual into the red iterate's place
template <class T, bool DIST, int COLOUR, bool RESID>
__device__ __forceinline__ void coarse_pass(const CoarseView<T>& C, bool from_zero) {
    const int hps = C.hps, hpz = hps * C.ny;
    const T* eoth = C.e[1 - COLOUR];
#pragma unroll 2
    for (int it = threadIdx.x; it < C.n; it += kCoarseThreads) {
        const CoarseItem w = C.items[it];
        const int o = w.o, par = (COLOUR + w.j + w.k) & 1;
        const T d = C.rd[COLOUR][o];  // 0: not an unknown; every load below is within the vectors all the same
        T v = C.b[COLOUR][o];
        const PkT<T> ckx = C.cx[2 * w.m + par], cky = C.cy[w.j], ckz = C.cz[w.k];
        if (RESID || !from_zero) {
            const T* x = eoth + o;
            v = rb_rest(v, ckx.x, ckx.z, cky.x, cky.z, ckz.x, ckz.z, x[par - 1], x[par], x[-hps], x[hps], x[-hpz],
                        x[hpz]);
        }
        T val;
        if constexpr (RESID) val = mg_fma(-(ckx.y + (cky.y + ckz.y)), C.e[COLOUR][o], v);
        else if constexpr (sizeof(T) == 8) val = times_rd(v, d);
        else val = v * d;  // times_rcp with the reciprocal kept
        if (d != T(0)) C.template put<DIST>(COLOUR, o, val);
    }
}

template <class T, bool DIST>
__device__ __forceinline__ void coarse_smooth(const CoarseView<T>& C, int sweeps, bool from_zero) {
    for (int q = 0; q < sweeps; ++q) {
        coarse_pass<T, DIST, 0, false>(C, from_zero && q == 0);
        coarse_sync<DIST>();
        coarse_pass<T, DIST, 1, false>(C, false);
        coarse_sync<DIST>();
    }
}

// the red residual of F (in its red iterate's place) to b of W; the CTA that
// owns a coarse row's fine centre row computes it
template <class T>
__device__ __forceinline__ void coarse_restrict(const Transfer<T>& X, const CoarseView<T>& F, const CoarseView<T>& W) {
    const int ny = F.ny, hps = F.hps, ncx = W.nx, ncy = W.ny, ncz = W.nz;
    const T* r0 = F.e[0];
    const int per = ncx - 2;
    const float inv = 1.0f / (float)per;
    const RwPk<T>*rwx = X.rw[0], *rwy = X.rw[1], *rwz = X.rw[2];
    for (int it = threadIdx.x; it < F.cnt * per; it += kCoarseThreads) {
        const int r = fast_div(it, inv), I = 1 + it - r * per, R = F.R0 + r;
        const int k = fast_div(R, F.inv_ny), j = R - k * ny, J = j >> 1, K = k >> 1;
        if ((j & 1) || (k & 1) || J < 1 || J > ncy - 2 || K < 1 || K > ncz - 2) continue;
        const T v = restrict_sum(rwx[I], rwy[J], rwz[K], [&](int a, int b, int c) {
            return r0[(r + (c - 1) * ny + (b - 1)) * hps + ((2 * I - 1 + a) >> 1)];
        });
        W.row((I + J + K) & 1 ? W.b[1] : W.b[0], K * ncy + J)[I >> 1] = v;
    }
}

// F's black unknowns += the interpolated iterate of W
template <class T, bool DIST>
__device__ __forceinline__ void coarse_prolong(const Transfer<T>& X, const CoarseView<T>& F, const CoarseView<T>& W) {
    const int ncy = W.ny;
    const IpPk<T>*ipx = X.ip[0], *ipy = X.ip[1], *ipz = X.ip[2];
    for (int it = threadIdx.x; it < F.n; it += kCoarseThreads) {
        const CoarseItem w = F.items[it];
        const int o = w.o, i = 2 * w.m + ((1 + w.j + w.k) & 1);
        if (F.rd[1][o] == T(0)) continue;
        const IpPk<T> px = ipx[i], py = ipy[w.j], pz = ipz[w.k];
        const int I = px.ilo, J = py.ilo, K = pz.ilo, x0 = I >> 1, x1 = (I + 1) >> 1;
        T* ea = (I + J + K) & 1 ? W.e[1] : W.e[0];
        T* eb = (I + J + K) & 1 ? W.e[0] : W.e[1];
        const int r00 = K * ncy + J, r01 = r00 + 1, r10 = r00 + ncy, r11 = r10 + 1;
        F.template put<DIST>(1, o,
                             prolong_value(F.e[1][o], px, py, pz, W.row(ea, r00)[x0], W.row(eb, r00)[x1],
                                           W.row(eb, r01)[x0], W.row(ea, r01)[x1], W.row(eb, r10)[x0],
                                           W.row(ea, r10)[x1], W.row(ea, r11)[x0], W.row(eb, r11)[x1]));
    }
}

template <class T>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse(const __grid_constant__ CoarseArgs<T> A) {
    extern __shared__ __align__(32) unsigned char coarse_smem[];
    auto cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank();
    // the levels' coefficients and pairs, b of the first level, zero
    // iterates, reciprocal diagonals
    for (int l = 0; l < A.nl; ++l) {
        const CoarseLevel<T>& V = A.V[l];
        const CoarseView<T> C = coarse_view(V, coarse_smem, rank);
        const SLev<T>& L = V.L;
        if (C.cnt == 0) continue;
        PkT<T>* cof = const_cast<PkT<T>*>(C.cx);
        for (int q = threadIdx.x; q < C.nx + C.ny + C.nz; q += kCoarseThreads) cof[q] = L.cx[q];
        T* vec = reinterpret_cast<T*>(coarse_smem) + V.vec;
        for (int q = threadIdx.x; q < 2 * (V.rpc + 2 * V.halo) * V.hps; q += kCoarseThreads) vec[q] = T(0);
        const int own = C.cnt * C.hps;
        for (int c = 0; c < 2; ++c) {
            const T* gb = L.b[c];
            const T* grd = L.rd[c];
            const uint8_t* gty = L.ty[c];
            T* b = c ? C.b[1] : C.b[0];
            T* rd = c ? C.rd[1] : C.rd[0];
#pragma unroll 4
            for (int o = threadIdx.x; o < own; o += kCoarseThreads) {
                const int r = fast_div(o, V.inv_hps), m = o - r * C.hps, R = C.R0 + r;
                const unsigned g = (unsigned)R * (unsigned)L.hp + (unsigned)m;
                b[o] = l == 0 ? gb[g] : T(0);
                T d = T(0);
                if constexpr (sizeof(T) == 8) {
                    d = grd[g];
                } else {
                    const int k = fast_div(R, C.inv_ny), j = R - k * C.ny, i = min(2 * m + ((c + j + k) & 1), C.nx - 1);
                    const float q = times_rcp(1.f, L.cx[i].y + (L.cy[j].y + L.cz[k].y));
                    if (is_unknown(gty[g])) d = q;
                }
                rd[o] = d;
            }
        }
        for (int it = threadIdx.x; it < C.n; it += kCoarseThreads) {  // read back by the same thread
            int q = fast_div(it, V.inv_mp);
            const int m = it - q * C.mp;
            if (!C.dist) {  // interior rows only
                const int k1 = fast_div(q, 1.0f / (float)(C.ny - 2));
                q = (k1 + 1) * C.ny + 1 + q - k1 * (C.ny - 2);
            }
            const int R = C.R0 + q, k = fast_div(R, C.inv_ny), j = R - k * C.ny;
            C.items[it] = CoarseItem{(unsigned short)(q * C.hps + m), (unsigned short)m, (unsigned short)j,
                                     (unsigned short)k};
        }
    }
    cluster.sync();
    // downward on the shared levels, the solo levels' part of the cycle on
    // CTA 0, upward on the shared levels
    const int last = A.nl - 1;
    for (int l = 0; l < A.ndist; ++l) {
        const CoarseView<T> C = coarse_view(A.V[l], coarse_smem, rank);
        coarse_smooth<T, true>(C, l == last ? 16 : A.pre, true);
        if (l == last) break;
        coarse_pass<T, true, 0, true>(C, false);
        cluster.sync();
        coarse_restrict(A.V[l].X, C, coarse_view(A.V[l + 1], coarse_smem, rank));
        cluster.sync();
    }
    if (rank == 0) {
        for (int l = A.ndist; l <= last; ++l) {
            const CoarseView<T> C = coarse_view(A.V[l], coarse_smem, rank);
            coarse_smooth<T, false>(C, l == last ? 16 : A.pre, true);
            if (l == last) break;
            coarse_pass<T, false, 0, true>(C, false);
            __syncthreads();
            coarse_restrict(A.V[l].X, C, coarse_view(A.V[l + 1], coarse_smem, rank));
            __syncthreads();
        }
        for (int l = last - 1; l >= A.ndist; --l) {
            const CoarseView<T> C = coarse_view(A.V[l], coarse_smem, rank);
            coarse_prolong<T, false>(A.V[l].X, C, coarse_view(A.V[l + 1], coarse_smem, rank));
            __syncthreads();
            coarse_smooth<T, false>(C, A.post, false);
        }
    }
    cluster.sync();
    for (int l = min(A.ndist, last) - 1; l >= 0; --l) {
        const CoarseView<T> C = coarse_view(A.V[l], coarse_smem, rank);
        coarse_prolong<T, true>(A.V[l].X, C, coarse_view(A.V[l + 1], coarse_smem, rank));
        cluster.sync();
        coarse_smooth<T, true>(C, A.post, false);
    }
    // the first level's iterate back to its global arrays
    const CoarseView<T> C = coarse_view(A.V[0], coarse_smem, rank);
    for (int c = 0; c < 2; ++c) {
        T* ge = A.V[0].L.e[c];
        const T* e = c ? C.e[1] : C.e[0];
        for (int o = threadIdx.x; o < C.cnt * C.hps; o += kCoarseThreads) {
            const int r = fast_div(o, A.V[0].inv_hps), m = o - r * C.hps;
            ge[(unsigned)(C.R0 + r) * (unsigned)A.V[0].L.hp + (unsigned)m] = e[o];
        }
    }
    cluster.sync();  // no CTA ends while another reads its shared memory
}
