// Real-space sample M_r^{1/2} z1 by Lanczos (Sec. II B 1; Chow & Saad),
// sm_103a.
//
// Vectors live in cell-sorted order as 16-byte (x, y, z, pad) records.  The
// basis is kept unnormalised: q_1 = z1 and q_{j+1} = w_j, with
// beta_j = ||q_{j+1}||, v_j = q_j / beta_{j-1}.  Per iteration j:
//   matvec  u = M_r q_j                       (+ deterministic q_j . u)
//   update  alpha_j = q_j.u / beta_{j-1}^2,
//           q_{j+1} = u/beta_{j-1} - alpha_j q_j/beta_{j-1} - beta_{j-1} q_{j-1}/beta_{j-2}
//                                               (+ deterministic ||q_{j+1}||^2)
//           and, in one more block of the same launch, y_j = T_j^{1/2} e_1 in
//           FP64 (one warp; T_j needs alpha_j but not beta_j, so it runs beside
//           the vector update), stop test ||y_j - [y_{j-1}; 0]|| / ||y_j|| < tol
//           (= ||x_j - x_{j-1}|| / ||x_j|| for an orthonormal basis)
// and finally x = beta_0 sum_i y_i q_i / beta_{i-1}.  Scalars are FP64; the
// reducing kernels run persistent grids (a fixed multiple of the SM count)
// and their per-block partial sums are added in block order by the last
// block to arrive, so results do not depend on scheduling.
#include <type_traits>

#include "lanczos_tj.cuh"
#include "pse_internal.cuh"

namespace pse {

template <typename T> __device__ __forceinline__ T sqrt_hd(T x) {
    if constexpr (sizeof(T) == 4) return sqrtf(x);
    else return sqrt(x);
}
template <typename T> __device__ __forceinline__ T floor_hd(T x) {
    if constexpr (sizeof(T) == 4) return floorf(x);
    else return floor(x);
}

template <typename T> __device__ __forceinline__ long long w_bits_r(T w) {
    if constexpr (sizeof(T) == 4) return (long long)__float_as_int(w);
    else return __double_as_longlong(w);
}

// per-thread partial: float for the float path (summed per warp in float,
// then in double), double for the FP64 path
template <typename T> struct Part { using type = float; };
template <> struct Part<double> { using type = double; };

template <typename T> __device__ __forceinline__ double block_total(typename Part<T>::type v, double *sh) {
    if constexpr (sizeof(T) == 4) return block_sum_fw(v, sh);
    else return block_sum(v, sh);
}

// ------------------------------------------------------------------ init: q_1 = z1, beta_0
template <typename T>
__device__ __forceinline__ void lz_init_body(int64_t N, const SampleArgs<T> *args, int system,
                                             const V4<T> *pos_sorted, V4<T> *q1, Rec<T> *rec, double *partials,
                                             LzState *lz, const float *__restrict__ pc, int bidx, int nblk,
                                             double *sh) {
    typename Part<T>::type part = 0;
    for (int64_t s = bidx * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)nblk * blockDim.x) {
        const uint32_t orig = (uint32_t)w_bits_r(pos_sorted[s].w);
        const Normals4<T> z = normals4<T>(orig, 2u * system, args->seed, args->sample);
        V4<T> v;
        v.x = z.v[0]; v.y = z.v[1]; v.z = z.v[2]; v.w = T(0);
        q1[s] = v;
        if constexpr (sizeof(T) == 4) {
            if (pc) {  // matvec input is S q
                V4<T> p;
                sym3_apply(pc + s * 16, v.x, v.y, v.z, p.x, p.y, p.z);
                p.w = T(0);
                rec[s].q = p;
            } else if (rec) {
                rec[s].q = v;
            }
        } else if (rec) {
            rec[s].q = v;
        }
        part += v.x * v.x + v.y * v.y + v.z * v.z;
    }
    const double bsum = block_total<T>(part, sh);
    double total;
    if (grid_sum_last(bsum, partials, &lz->counter_init, sh, &total, bidx, nblk) && threadIdx.x == 0) {
        const double bi = total > 0.0 ? rsqrt_f64(total) : 0.0;
        lz->beta[0] = total * bi;
        lz->binv[0] = bi;
        lz->tmax = 0.0;
        lz->iter = 1;
        lz->J = 0;
        lz->converged = 0;
        lz->cont = 1;
        lz->active = 1;
        lz->num = 0.0;
        lz->den = 0.0;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_lz_init(int64_t N, const SampleArgs<T> *args, int system,
                                                 const V4<T> *pos_sorted, V4<T> *q1, Rec<T> *rec, double *partials,
                                                 LzState *lz, const float *__restrict__ pc) {
    __shared__ double sh[32];
    lz_init_body<T>(N, args, system, pos_sorted, q1, rec, partials, lz, pc, blockIdx.x, gridDim.x, sh);
}

__global__ void __launch_bounds__(256) k_lz_init_batch(const BSys *__restrict__ sys, const int *__restrict__ tab) {
    __shared__ double sh[32];
    const BSys &S = sys[tab[blockIdx.x]];
    lz_init_body<float>(S.N, S.d.args, S.system, S.d.pos_sorted, S.d.basis, rec_q(S.d), S.d.partials, S.d.lz, S.d.pc_on,
                        (int)blockIdx.x - S.b0[BK_INIT], S.nb[BK_INIT], sh);
}

// alpha_j = q_j.u / beta_{j-1}^2 and the coefficients of the update, by
// multiplications with the stored 1/beta (an FP64 division costs about as much
// as the rest of this tail).  beta_{j-1} = 0 (binv = 0): the Krylov space is
// invariant and the loop has stopped.  What thread 0 of the last block will
// need is fetched by thread 0 of every block before its rows.
struct LzPrev {
    double bi, cp;
};
__device__ __forceinline__ void lz_prev(const LzState *lz, int j, LzPrev *sp) {
    if (threadIdx.x) return;
    sp->bi = lz->binv[j - 1];
    sp->cp = j >= 2 ? lz->beta[j - 1] * lz->binv[j - 2] : 0.0;
}
__device__ __forceinline__ void lz_alpha(LzState *lz, int j, double total, const LzPrev &sp) {
    const double bi = sp.bi, cu = total * bi, alpha = cu * bi;
    lz->alpha[j] = alpha;
    lz->c_u = bi;
    lz->c_q = alpha * bi;
    lz->c_p = sp.cp;
}

// ------------------------------------------------------------------ near-field matvec
// u_s = self q_s + sum_t [F (I - rr) + G rr] q_t over the ELL list of s, F and
// G linearly interpolated from the FP64-built table (stored / 6 pi a).  A
// group of TPP consecutive threads shares one particle: thread g of the
// group takes entries g, g + TPP, ... and the group sums by shuffles.  Each
// neighbour costs one 4-byte list entry and one 32-byte record; a thread
// issues ILP list loads, then ILP record loads, before any arithmetic, so
// that many independent gathers are in flight.  The first round's list
// loads do not wait for the particle's count: entries up to the ELL
// capacity K are always in the array, and those past the count are dropped.

template <typename T>
__device__ __forceinline__ void pair_fg(T r, const Geom<T> &g, const V4<T> *__restrict__ table, T &F, T &GmF) {
    if (sizeof(T) == 8 && r >= T(0.2) * g.a) {
        // FP64 context: Appendix A evaluated exactly instead of interpolated
        double Fd, Gd;
        fg_closed_hd((double)r, (double)g.xi, (double)g.a, &Fd, &Gd);
        const double sc = 1.0 / (6.0 * 3.14159265358979323846 * (double)g.a);
        F = (T)(Fd * sc);
        GmF = (T)((Gd - Fd) * sc);
    } else {
        const T uu = r * g.tab_inv_dr;
        int it = (int)uu;
        it = it > PSE_TABLE_N - 2 ? PSE_TABLE_N - 2 : it;
        const T f = uu - T(it);
        const V4<T> tb = table[it];
        F = tb.x + f * tb.z;
        GmF = tb.y + f * tb.w;
    }
}

// One matvec record, read-only for the kernel's lifetime: a single 256-bit
// load for float records (one L1 request per neighbour instead of two).
template <typename T> __device__ __forceinline__ Rec<T> load_rec(const Rec<T> *__restrict__ p) {
    if constexpr (sizeof(T) == 4) {
        Rec<T> r;
        asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(r.l.x), "=f"(r.l.y), "=f"(r.l.z), "=f"(r.l.w), "=f"(r.q.x), "=f"(r.q.y), "=f"(r.q.z), "=f"(r.q.w)
            : "l"(p));
        return r;
    } else {
        return *p;
    }
}

// Compact-table lookup (two uniform segments, knot at min(2a, r_cut)); `tab`
// is normally the block's shared-memory copy.
template <typename T>
__device__ __forceinline__ void pair_fg_c(T r, const Geom<T> &g, const V4<T> *tab, T &F, T &GmF) {
    const T u = r < g.tc_split ? r * g.tc_invA : T(PSE_TABLEC_A) + (r - g.tc_split) * g.tc_invB;
    int it = (int)u;
    it = it > PSE_TABLEC_N - 2 ? PSE_TABLEC_N - 2 : it;
    const T f = u - T(it);
    const V4<T> tb = tab[it];
    F = tb.x + f * tb.z;
    GmF = tb.y + f * tb.w;
}

// Species index of a cell record (polydisperse contexts).
template <typename T> __device__ __forceinline__ int spec_of(const V4<T> &l) {
    return (int)((w_bits_r(l.w) >> PSE_SPECIES_SHIFT) & 3);
}
// Self mobility of species sp (selects, so that the parameter array is not
// copied to local memory for a dynamic index).
template <typename T> __device__ __forceinline__ T self_of(const Geom<T> &g, int sp) {
    return sp == 0 ? g.self_s[0] : (sp == 1 ? g.self_s[1] : (sp == 2 ? g.self_s[2] : g.self_s[3]));
}

// Row s of M_r q without the self term, summed over the TPP-thread group.
// CT: `table` is the compact table (pair_fg_c), else the uniform one.
// POLY: the uniform table holds one block per species pair (polydisperse).
template <typename T, int TPP, int ILP, bool CT = false, bool POLY = false>
__device__ __forceinline__ void mr_row_part(int64_t N, int64_t s, int lane_g, bool active, int K, const Geom<T> &g,
                                            const Rec<T> *__restrict__ rec, const int *__restrict__ count,
                                            const int *__restrict__ nbr, const V4<T> *__restrict__ table,
                                            V4<T> &li, V4<T> &qi, T &ax, T &ay, T &az) {
    ax = ay = az = T(0);
    if (active) {
        const int cnt = count[s];
        int ent[ILP];
#pragma unroll
        for (int u = 0; u < ILP; ++u) {
            const int k = lane_g + u * TPP;
            ent[u] = k < K ? __ldg(nbr + (int64_t)k * N + s) : -1;
        }
        const Rec<T> ri = load_rec(rec + s);
        li = ri.l;
        qi = ri.q;
        for (int k0 = lane_g; k0 < cnt; k0 += ILP * TPP) {
            if (k0 != lane_g) {
#pragma unroll
                for (int u = 0; u < ILP; ++u) {
                    const int k = k0 + u * TPP;
                    ent[u] = k < K ? __ldg(nbr + (int64_t)k * N + s) : -1;
                }
            }
#pragma unroll
            for (int u = 0; u < ILP; ++u)
                if (k0 + u * TPP >= cnt) ent[u] = -1;
            Rec<T> rt[ILP];
#pragma unroll
            for (int u = 0; u < ILP; ++u) rt[u] = load_rec(rec + (ent[u] >= 0 ? (ent[u] >> 6) : s));
#pragma unroll
            for (int u = 0; u < ILP; ++u) {
                if (ent[u] < 0) continue;
                const int e = ent[u];
                const int ox = ((e >> 4) & 3) - 1, oy = ((e >> 2) & 3) - 1, oz = (e & 3) - 1;
                const T dx = (li.x - rt[u].l.x) - (T(ox) * g.cs + T(ox) * g.cs_lo);
                const T dy = (li.y - rt[u].l.y) - (T(oy) * g.cs + T(oy) * g.cs_lo);
                const T dz = (li.z - rt[u].l.z) - (T(oz) * g.cs + T(oz) * g.cs_lo);
                const T r2 = dx * dx + dy * dy + dz * dz;
                T rinv;
                if constexpr (sizeof(T) == 4) rinv = r2 > 0.f ? rsqrtf(r2) : 0.f;
                else rinv = r2 > 0.0 ? 1.0 / sqrt(r2) : 0.0;
                T F, GmF;
                if constexpr (CT) {
                    pair_fg_c(r2 * rinv, g, table, F, GmF);
                } else if constexpr (POLY) {
                    const V4<T> *tb = table + (int64_t)pair_index(spec_of(li), spec_of(rt[u].l), g.nspec) * PSE_TABLE_N;
                    pair_fg(r2 * rinv, g, tb, F, GmF);
                } else {
                    pair_fg(r2 * rinv, g, table, F, GmF);
                }
                const T hx = dx * rinv, hy = dy * rinv, hz = dz * rinv;
                const T dot = GmF * (hx * rt[u].q.x + hy * rt[u].q.y + hz * rt[u].q.z);
                ax += F * rt[u].q.x + dot * hx;
                ay += F * rt[u].q.y + dot * hy;
                az += F * rt[u].q.z + dot * hz;
            }
        }
    }
#pragma unroll
    for (int o = TPP / 2; o > 0; o >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, o);
        ay += __shfl_xor_sync(0xffffffffu, ay, o);
        az += __shfl_xor_sync(0xffffffffu, az, o);
    }
}

// Row s of M_r q without the self term and without a neighbour list (FP32):
// one thread walks the 27 stencil cells of its particle over the cell-sorted
// records, which carry q beside the cell-local offsets.  A candidate is kept
// by the neighbour search's own float32 test (below the top of the r_cut
// band), and one inside the band by the float64 decision from the wrapped
// positions, so the row sums exactly the pairs the neighbour list holds
// (summation in stencil order).
__device__ __forceinline__ void mr_row_nolist(int64_t s, bool active, const Geom<float> &g,
                                              const Rec<float> *__restrict__ rec,
                                              const int *__restrict__ cell_start,
                                              const V4<float> *__restrict__ pos, const V4<float> *tab,
                                              V4<float> &li, V4<float> &qi, float &ax, float &ay, float &az) {
    ax = ay = az = 0.f;
    if (!active) return;
    const Rec<float> ri = load_rec(rec + s);
    li = ri.l;
    qi = ri.q;
    const int c = (int)(w_bits_r(li.w) & PSE_CELL_MASK);
    const int nc = g.nc;
    int cx, cy, cz;
    cell_xyz(c, g.nb, cx, cy, cz);
    for (int ox = -1; ox <= 1; ++ox) {
        int axc = cx + ox;
        axc += axc < 0 ? nc : 0;
        axc -= axc >= nc ? nc : 0;
        const float sx = float(ox) * g.cs + float(ox) * g.cs_lo;
        for (int oy = -1; oy <= 1; ++oy) {
            int ayc = cy + oy;
            ayc += ayc < 0 ? nc : 0;
            ayc -= ayc >= nc ? nc : 0;
            const float sy = float(oy) * g.cs + float(oy) * g.cs_lo;
            for (int oz = -1; oz <= 1; ++oz) {
                int azc = cz + oz;
                azc += azc < 0 ? nc : 0;
                azc -= azc >= nc ? nc : 0;
                const float sz = float(oz) * g.cs + float(oz) * g.cs_lo;
                const int c2 = cell_id(axc, ayc, azc, g.nb);
                const int b = cell_start[c2], e = cell_start[c2 + 1];
                const int self = (ox | oy | oz) == 0 ? (int)s : -1;
                for (int t = b; t < e; ++t) {
                    if (t == self) continue;
                    const Rec<float> rt = load_rec(rec + t);
                    const float dx = (li.x - rt.l.x) - sx;
                    const float dy = (li.y - rt.l.y) - sy;
                    const float dz = (li.z - rt.l.z) - sz;
                    const float r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 >= g.rc2_hi) continue;
                    if (r2 >= g.rc2_lo && !pair_inside_f64(pos[s], pos[t], g)) continue;
                    const float rinv = r2 > 0.f ? rsqrtf(r2) : 0.f;
                    float F, GmF;
                    pair_fg_c(r2 * rinv, g, tab, F, GmF);
                    const float hx = dx * rinv, hy = dy * rinv, hz = dz * rinv;
                    const float dot = GmF * (hx * rt.q.x + hy * rt.q.y + hz * rt.q.z);
                    ax += F * rt.q.x + dot * hx;
                    ay += F * rt.q.y + dot * hy;
                    az += F * rt.q.z + dot * hz;
                }
            }
        }
    }
}

// Body of one Lanczos matvec over the nblk blocks of one system (bidx = this
// block's index among them).  NOLIST: rows by mr_row_nolist (FP32, TPP 1),
// which reads cell_start and the sorted positions instead of the list.
template <typename T, int TPP, int ILP, bool CT, bool POLY = false, bool NOLIST = false>
__device__ __forceinline__ void lz_matvec_body(int64_t N, int K, const Geom<T> &g, const Rec<T> *__restrict__ rec,
                                               const int *__restrict__ count, const int *__restrict__ nbr,
                                               const V4<T> *__restrict__ table, V4<T> *u, double *partials,
                                               LzState *lz, const float *__restrict__ pc,
                                               const V4<T> *__restrict__ basis, const V4<T> *__restrict__ add,
                                               int bidx, int nblk, double *sh,
                                               const int *__restrict__ cell_start = nullptr,
                                               const V4<T> *__restrict__ pos_sorted = nullptr) {
    const int j = lz->iter;
    if (j > PSE_MAXIT || !lz->active) return;  // uniform across the system's blocks
    __shared__ LzPrev prev;
    lz_prev(lz, j, &prev);
    typename Part<T>::type part = 0;
    const int lane_g = threadIdx.x % TPP;
    const int64_t per_block = blockDim.x / TPP;
    // contiguous chunk of particles per block (spatial locality across
    // iterations); whole groups stride together so group shuffles converge
    const int64_t chunk = ((N + nblk - 1) / nblk + per_block - 1) / per_block * per_block;
    const int64_t end = (bidx + 1) * chunk < N ? (bidx + 1) * chunk : N;
    for (int64_t base = bidx * chunk; base < end; base += per_block) {
        const int64_t s = base + threadIdx.x / TPP;
        const bool active = s < end;
        V4<T> li, qi;
        T ax, ay, az;
        if constexpr (NOLIST) {
            mr_row_nolist(s, active, g, rec, cell_start, pos_sorted, table, li, qi, ax, ay, az);
        } else {
            mr_row_part<T, TPP, ILP, CT, POLY>(N, s, lane_g, active, K, g, rec, count, nbr, table, li, qi, ax, ay,
                                               az);
        }
        if (active && lane_g == 0) {
            V4<T> o;
            const T self = POLY ? self_of(g, spec_of(li)) : g.self_m;
            o.x = ax + self * qi.x;
            o.y = ay + self * qi.y;
            o.z = az + self * qi.z;
            o.w = T(0);
            if (add) {  // full-mobility Lanczos: the wave product M_w q_j of the same vector
                const V4<T> aw = add[s];
                o.x += aw.x;
                o.y += aw.y;
                o.z += aw.z;
            }
            if constexpr (sizeof(T) == 4) {
                if (pc) {  // A = S M_r S: the record holds S q, apply S to the row, dot with q
                    T x, y, z;
                    sym3_apply(pc + s * 16, o.x, o.y, o.z, x, y, z);
                    o.x = x; o.y = y; o.z = z;
                    qi = basis[(int64_t)(j - 1) * N + s];
                }
            }
            u[s] = o;
            part += qi.x * o.x + qi.y * o.y + qi.z * o.z;
        }
    }
    const double bsum = block_total<T>(part, sh);
    double total;
    if (grid_sum_last(bsum, partials, &lz->counter_mv, sh, &total, bidx, nblk) && threadIdx.x == 0) {
        lz_alpha(lz, j, total, prev);
    }
}

// Float contexts stage the compact F, G table (16 KB) in shared memory:
// table lookups then cost shared-memory wavefronts instead of scattered L1
// lines.  The FP64 path uses the uniform table (r < 0.2a) and the closed form.
// BS threads per block: with large blocks fewer copies of the table share an
// SM, leaving more of its on-chip memory to the L1 that caches the records.
template <typename T, int TPP, int ILP, int BS = 128>
__global__ void __launch_bounds__(BS) k_lz_matvec(int64_t N, int K, Geom<T> g, const Rec<T> *__restrict__ rec,
                                                   const int *__restrict__ count, const int *__restrict__ nbr,
                                                   const V4<T> *__restrict__ table, const V4<T> *__restrict__ table_c,
                                                   V4<T> *u, double *partials, LzState *lz,
                                                   const float *__restrict__ pc, const V4<T> *__restrict__ basis,
                                                   const V4<T> *__restrict__ add) {
    __shared__ double sh[32];
    if constexpr (sizeof(T) == 4) {
        __shared__ V4<float> tab_s[PSE_TABLEC_N];
        for (int i = threadIdx.x; i < PSE_TABLEC_N; i += blockDim.x) tab_s[i] = table_c[i];
        __syncthreads();
        lz_matvec_body<T, TPP, ILP, true>(N, K, g, rec, count, nbr, tab_s, u, partials, lz, pc, basis, add,
                                          blockIdx.x, gridDim.x, sh);
    } else {
        lz_matvec_body<T, TPP, ILP, false>(N, K, g, rec, count, nbr, table, u, partials, lz, pc, basis, add,
                                           blockIdx.x, gridDim.x, sh);
    }
}

// ------------------------------------------------------------------ stored pair blocks (FP64)
// The block of a pair, F (I - rr) + G rr = F I + sign(g) w w^T with g = G - F
// and w = |g|^{1/2} r^, is the same in every product of one sample, and in
// FP64 its closed form (three exponentials, three complementary error
// functions, a dozen divisions) costs far more than streaming it: k_pairs
// evaluates it once per directed pair, one pair per thread at a time, and the
// products read a 4-byte entry (neighbour, the sign of g in bit 31) and a
// 32-byte record (w, F) in order and gather the neighbour's q.  N = 1000
// (phi = 0.1, J = 4): four products of 125 us each -> k_pairs 39 us and four
// of 9 us.  In FP32 the list form stays: a record costs 16 bytes more per pair
// and product than it saves in table lookups (N = 1e6: products 78 -> 69 us,
// but 143 us for k_pairs).
// Layout: slices of 32 consecutive particles, column k of a slice = 32
// entries (records) side by side, `cols` columns of room per slice.
// Columns past `cols` (lists about twice as long as the mean) are not stored:
// pair_far evaluates those pairs in each product.
__device__ __forceinline__ void pair_scalars(const V4<double> &li, const V4<double> &lt, int e, const Geom<double> &g,
                                             const V4<double> *table, double &F, double &GmF, double &hx, double &hy,
                                             double &hz) {
    const int ox = ((e >> 4) & 3) - 1, oy = ((e >> 2) & 3) - 1, oz = (e & 3) - 1;
    const double dx = (li.x - lt.x) - (double(ox) * g.cs + double(ox) * g.cs_lo);
    const double dy = (li.y - lt.y) - (double(oy) * g.cs + double(oy) * g.cs_lo);
    const double dz = (li.z - lt.z) - (double(oz) * g.cs + double(oz) * g.cs_lo);
    const double r2 = dx * dx + dy * dy + dz * dz;
    const double rinv = r2 > 0.0 ? 1.0 / sqrt(r2) : 0.0;
    pair_fg(r2 * rinv, g, table, F, GmF);
    hx = dx * rinv;
    hy = dy * rinv;
    hz = dz * rinv;
}

// Stored entry (record) k of particle s.
__device__ __forceinline__ uint32_t pair_at(uint32_t s, uint32_t k, uint32_t cols) {
    return ((s >> 5) * cols + k) * 32u + (s & 31u);
}

// TPP lanes share a particle: a warp works on SP = 32 / TPP consecutive
// particles, lanes of equal lane / SP on the same column; a block's share of
// these row groups is contiguous and its warps take consecutive groups.
template <int TPP> struct RowShare {
    static constexpr int SP = 32 / TPP;
    int p, c;  // this lane's particle of the group, column offset
    int64_t i, end;
    int step;
    __device__ RowShare(int64_t N) : p((threadIdx.x & 31) % SP), c((threadIdx.x & 31) / SP) {
        const int64_t groups = (N + SP - 1) / SP;
        i = blockIdx.x * groups / gridDim.x + (threadIdx.x >> 5);
        end = (blockIdx.x + 1) * groups / gridDim.x;
        step = blockDim.x >> 5;
    }
};

#define PSE_STORED_THREADS 256
template <int TPP>
__global__ void __launch_bounds__(PSE_STORED_THREADS) k_pairs(int64_t N, int cols, Geom<double> g,
                                                              const V4<double> *__restrict__ loc,
                                                              const int *__restrict__ count,
                                                              const int *__restrict__ nbr,
                                                              const V4<double> *__restrict__ table,
                                                              V4<double> *__restrict__ pair, int *__restrict__ pent) {
    for (RowShare<TPP> R(N); R.i < R.end; R.i += R.step) {
        const int64_t s = R.i * R.SP + R.p;
        if (s >= N) continue;
        const int n = min(count[s], cols);
        const V4<double> li = loc[s];
        for (int k = R.c; k < n; k += TPP) {
            const int e = nbr[(int64_t)k * N + s];
            V4<double> r;
            r.x = r.y = r.z = r.w = 0.0;
            int t = (int)s;  // a removed entry: a zero block
            if (e >= 0) {
                double F, g2, hx, hy, hz;
                pair_scalars(li, loc[e >> 6], e, g, table, F, g2, hx, hy, hz);
                const double c = sqrt(fabs(g2));
                r.x = c * hx; r.y = c * hy; r.z = c * hz; r.w = F;
                t = (e >> 6) | (g2 < 0.0 ? (int)0x80000000 : 0);
            }
            const uint32_t at = pair_at((uint32_t)s, (uint32_t)k, (uint32_t)cols);
            pair[at] = r;
            pent[at] = t;
        }
    }
}

// One pair past the stored columns.
__device__ __noinline__ V4<double> pair_far(int64_t s, int e, const Geom<double> *g,
                                            const V4<double> *__restrict__ loc, const V4<double> *__restrict__ table,
                                            V4<double> q) {
    double F, g2, hx, hy, hz;
    pair_scalars(loc[s], loc[e >> 6], e, *g, table, F, g2, hx, hy, hz);
    const double dot = g2 * (hx * q.x + hy * q.y + hz * q.z);
    V4<double> r;
    r.x = F * q.x + dot * hx;
    r.y = F * q.y + dot * hy;
    r.z = F * q.z + dot * hz;
    r.w = 0.0;
    return r;
}

// u = M_r q (+ add) over this block's particles; returns this thread's share
// of q.u.
template <int TPP>
__device__ __forceinline__ double stored_rows(int64_t N, int cols, const Geom<double> &g,
                                              const V4<double> *__restrict__ q, const V4<double> *__restrict__ loc,
                                              const int *__restrict__ count, const int *__restrict__ nbr,
                                              const V4<double> *__restrict__ pair, const int *__restrict__ pent,
                                              const V4<double> *__restrict__ table, V4<double> *__restrict__ u,
                                              const V4<double> *__restrict__ add) {
    double part = 0.0;
    for (RowShare<TPP> R(N); R.i < R.end; R.i += R.step) {
        const int64_t s = R.i * R.SP + R.p;
        const bool active = s < N;
        const int cnt = active ? count[s] : 0;
        const int n = cnt < cols ? cnt : cols;
        double ax = 0.0, ay = 0.0, az = 0.0;
        const uint32_t b = pair_at((uint32_t)s, 0, (uint32_t)cols);
#pragma unroll 2
        for (int k = R.c; k < n; k += TPP) {
            const int e = pent[b + 32u * k];
            const V4<double> r = pair[b + 32u * k], qt = q[e & 0x7fffffff];
            double dot = r.x * qt.x + r.y * qt.y + r.z * qt.z;
            dot = e < 0 ? -dot : dot;
            ax += r.w * qt.x + dot * r.x;
            ay += r.w * qt.y + dot * r.y;
            az += r.w * qt.z + dot * r.z;
        }
        for (int k = n + R.c; k < cnt; k += TPP) {
            const int e = nbr[(int64_t)k * N + s];
            if (e < 0) continue;
            const V4<double> f = pair_far(s, e, &g, loc, table, q[e >> 6]);
            ax += f.x;
            ay += f.y;
            az += f.z;
        }
#pragma unroll
        for (int o = R.SP; o < 32; o <<= 1) {
            ax += __shfl_xor_sync(0xffffffffu, ax, o);
            ay += __shfl_xor_sync(0xffffffffu, ay, o);
            az += __shfl_xor_sync(0xffffffffu, az, o);
        }
        if (active && R.c == 0) {
            const V4<double> qs = q[s];
            V4<double> o;
            o.x = ax + g.self_m * qs.x;
            o.y = ay + g.self_m * qs.y;
            o.z = az + g.self_m * qs.z;
            o.w = 0.0;
            if (add) {  // full-mobility Lanczos: the wave product M_w q_j of the same vector
                const V4<double> aw = add[s];
                o.x += aw.x;
                o.y += aw.y;
                o.z += aw.z;
            }
            u[s] = o;
            part += qs.x * o.x + qs.y * o.y + qs.z * o.z;
        }
    }
    return part;
}

template <int TPP>
__global__ void __launch_bounds__(PSE_STORED_THREADS) k_lz_matvec_stored(
    int64_t N, int cols, const __grid_constant__ Geom<double> g, const V4<double> *__restrict__ basis,
    const V4<double> *__restrict__ loc, const int *__restrict__ count, const int *__restrict__ nbr,
    const V4<double> *__restrict__ pair, const int *__restrict__ pent, const V4<double> *__restrict__ table,
    V4<double> *u, double *partials, LzState *lz, const V4<double> *__restrict__ add) {
    __shared__ double sh[32];
    const int j = lz->iter;
    if (j > PSE_MAXIT || !lz->active) return;  // uniform across the launch
    __shared__ LzPrev prev;
    lz_prev(lz, j, &prev);
    const double part = stored_rows<TPP>(N, cols, g, basis + (int64_t)(j - 1) * N, loc, count, nbr, pair, pent, table,
                                         u, add);
    const double bsum = block_sum(part, sh);
    double total;
    if (grid_sum_last(bsum, partials, &lz->counter_mv, sh, &total) && threadIdx.x == 0) lz_alpha(lz, j, total, prev);
}

// M_r v of a sorted vector (forces path).
template <int TPP>
__global__ void __launch_bounds__(PSE_STORED_THREADS) k_matvec_stored(
    int64_t N, int cols, const __grid_constant__ Geom<double> g, const V4<double> *__restrict__ v,
    const V4<double> *__restrict__ loc, const int *__restrict__ count, const int *__restrict__ nbr,
    const V4<double> *__restrict__ pair, const int *__restrict__ pent, const V4<double> *__restrict__ table,
    V4<double> *out) {
    stored_rows<TPP>(N, cols, g, v, loc, count, nbr, pair, pent, table, out, nullptr);
}

// ------------------------------------------------------------------ brick-tiled matvec
// FP32 monodisperse form that serves the neighbour records from shared
// memory.  A block takes one 4x4x4-cell brick at a time (a fixed, strided
// set of bricks: the per-block partial sums, and so alpha, do not depend on
// scheduling).  It stages the records of the brick's 6x6x6-cell
// neighbourhood -- runs of consecutive sorted particles, one per cell, read
// from L2 -- and a per-cell offset, so that the ELL entry (t, stencil code)
// of a particle in brick-local cell (lx, ly, lz) is found at
// t + hoff[((lx + 1 + ox) * 6 + (ly + 1 + oy)) * 6 + (lz + 1 + oz)].  The
// scattered 32-byte gathers then cost shared-memory wavefronts instead of
// L1/L2 lines.  A brick whose neighbourhood holds more than `cap` particles
// gathers from global memory instead.  The pair arithmetic is that of
// mr_row_part with the compact table.
#define PSE_TILE_THREADS 256
#define PSE_TILE_TPP 4
#define PSE_TILE_ILP 4
__global__ void __launch_bounds__(PSE_TILE_THREADS, 4) k_lz_matvec_tiled(
    int64_t N, int K, Geom<float> g, const Rec<float> *__restrict__ rec, const int *__restrict__ cell_start,
    const int *__restrict__ count, const int *__restrict__ nbr, const V4<float> *__restrict__ table_c,
    V4<float> *u, double *partials, LzState *lz, const V4<float> *__restrict__ add, int nbricks, int cap) {
    constexpr int TPP = PSE_TILE_TPP, ILP = PSE_TILE_ILP;
    __shared__ double sh[32];
    __shared__ V4<float> tab_s[PSE_TABLEC_N];
    __shared__ int hpre[217], hoff[216], hcell[216];
    extern __shared__ __align__(32) unsigned char tile_raw[];
    Rec<float> *halo = reinterpret_cast<Rec<float> *>(tile_raw);
    for (int i = threadIdx.x; i < PSE_TABLEC_N; i += blockDim.x) tab_s[i] = table_c[i];
    const int j = lz->iter;
    if (j > PSE_MAXIT || !lz->active) return;  // uniform across the launch
    __shared__ LzPrev prev;
    lz_prev(lz, j, &prev);
    float part = 0.f;
    const int nb = g.nb, nc = g.nc;
    const int lane_g = threadIdx.x % TPP;
    const int per_pass = blockDim.x / TPP;
    for (int b = blockIdx.x; b < nbricks; b += gridDim.x) {
        const int s0 = cell_start[b * 64], s1 = cell_start[b * 64 + 64];
        if (s0 == s1) continue;  // uniform: an empty brick (or cell slots past ncell)
        const int bz = b % nb, by = (b / nb) % nb, bx = b / (nb * nb);
        __syncthreads();  // the previous brick's readers are done with the tile
        for (int h = threadIdx.x; h < 216; h += blockDim.x) {
            const int hx = h / 36, hy = (h / 6) % 6, hz = h % 6;
            const int cx = ((bx * 4 - 1 + hx) % nc + nc) % nc;
            const int cy = ((by * 4 - 1 + hy) % nc + nc) % nc;
            const int cz = ((bz * 4 - 1 + hz) % nc + nc) % nc;
            const int c = cell_id(cx, cy, cz, nb);
            hcell[h] = c;
            hpre[h + 1] = cell_start[c + 1] - cell_start[c];
        }
        __syncthreads();
        if (threadIdx.x < 32) {  // exclusive prefix of the 216 counts, one warp
            int carry = 0;
            for (int base = 0; base < 216; base += 32) {
                const int h = base + threadIdx.x;
                int v = h < 216 ? hpre[h + 1] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, v, o);
                    if (threadIdx.x >= o) v += n;
                }
                if (h < 216) hpre[h + 1] = carry + v;
                carry += __shfl_sync(0xffffffffu, v, 31);
            }
            if (threadIdx.x == 0) hpre[0] = 0;
        }
        __syncthreads();
        const int total = hpre[216];
        const bool staged = total <= cap;
        if (staged) {
            for (int h = threadIdx.x; h < 216; h += blockDim.x) hoff[h] = hpre[h] - cell_start[hcell[h]];
            for (int i = threadIdx.x; i < total; i += blockDim.x) {
                int lo = 0, hi = 215;  // last halo cell with hpre <= i
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (hpre[mid] <= i) lo = mid;
                    else hi = mid - 1;
                }
                halo[i] = load_rec(rec + cell_start[hcell[lo]] + (i - hpre[lo]));
            }
        }
        __syncthreads();
        for (int base = s0; base < s1; base += per_pass) {
            const int s = base + threadIdx.x / TPP;
            const bool active = s < s1;
            float ax = 0.f, ay = 0.f, az = 0.f;
            Rec<float> ri;
            if (active) {
                ri = load_rec(rec + s);
                const int own = __float_as_int(ri.l.w) & 63;  // brick-local cell (lx, ly, lz)
                const int l0 = ((((own >> 4) & 3) + 1) * 6 + ((own >> 2) & 3) + 1) * 6 + (own & 3) + 1;
                const int cnt = count[s];
                for (int k0 = lane_g; k0 < cnt; k0 += ILP * TPP) {
                    int ent[ILP];
#pragma unroll
                    for (int q = 0; q < ILP; ++q) {
                        const int k = k0 + q * TPP;
                        ent[q] = k < cnt ? __ldg(nbr + (int64_t)k * N + s) : -1;
                    }
                    Rec<float> rt[ILP];
#pragma unroll
                    for (int q = 0; q < ILP; ++q) {
                        const int e = ent[q];
                        if (e < 0) continue;
                        const int t = e >> 6;
                        // stencil code (ox+1)<<4 | (oy+1)<<2 | (oz+1) shifts the halo index
                        const int hc = l0 - 43 + ((e >> 4) & 3) * 36 + ((e >> 2) & 3) * 6 + (e & 3);
                        rt[q] = staged ? halo[t + hoff[hc]] : load_rec(rec + t);
                    }
#pragma unroll
                    for (int q = 0; q < ILP; ++q) {
                        const int e = ent[q];
                        if (e < 0) continue;
                        const int ox = ((e >> 4) & 3) - 1, oy = ((e >> 2) & 3) - 1, oz = (e & 3) - 1;
                        const float dx = (ri.l.x - rt[q].l.x) - (float(ox) * g.cs + float(ox) * g.cs_lo);
                        const float dy = (ri.l.y - rt[q].l.y) - (float(oy) * g.cs + float(oy) * g.cs_lo);
                        const float dz = (ri.l.z - rt[q].l.z) - (float(oz) * g.cs + float(oz) * g.cs_lo);
                        const float r2 = dx * dx + dy * dy + dz * dz;
                        const float rinv = r2 > 0.f ? rsqrtf(r2) : 0.f;
                        float F, GmF;
                        pair_fg_c(r2 * rinv, g, tab_s, F, GmF);
                        const float hx = dx * rinv, hy = dy * rinv, hz = dz * rinv;
                        const float dot = GmF * (hx * rt[q].q.x + hy * rt[q].q.y + hz * rt[q].q.z);
                        ax += F * rt[q].q.x + dot * hx;
                        ay += F * rt[q].q.y + dot * hy;
                        az += F * rt[q].q.z + dot * hz;
                    }
                }
            }
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                ax += __shfl_xor_sync(0xffffffffu, ax, o);
                ay += __shfl_xor_sync(0xffffffffu, ay, o);
                az += __shfl_xor_sync(0xffffffffu, az, o);
            }
            if (active && lane_g == 0) {
                V4<float> o;
                o.x = ax + g.self_m * ri.q.x;
                o.y = ay + g.self_m * ri.q.y;
                o.z = az + g.self_m * ri.q.z;
                o.w = 0.f;
                if (add) {
                    const V4<float> aw = add[s];
                    o.x += aw.x;
                    o.y += aw.y;
                    o.z += aw.z;
                }
                u[s] = o;
                part += ri.q.x * o.x + ri.q.y * o.y + ri.q.z * o.z;
            }
        }
    }
    const double bsum = block_sum_fw(part, sh);
    double total;
    if (grid_sum_last(bsum, partials, &lz->counter_mv, sh, &total) && threadIdx.x == 0) {
        lz_alpha(lz, j, total, prev);
    }
}

// Polydisperse contexts (FP32): 4 threads x 4 gathers per particle in blocks
// of 1024, F and G from the uniform table block of each species pair.
__global__ void __launch_bounds__(1024) k_lz_matvec_poly(int64_t N, int K, Geom<float> g,
                                                         const Rec<float> *__restrict__ rec,
                                                         const int *__restrict__ count, const int *__restrict__ nbr,
                                                         const V4<float> *__restrict__ table, V4<float> *u,
                                                         double *partials, LzState *lz,
                                                         const V4<float> *__restrict__ basis) {
    __shared__ double sh[32];
    lz_matvec_body<float, 4, 4, false, true>(N, K, g, rec, count, nbr, table, u, partials, lz, nullptr, basis,
                                             nullptr, blockIdx.x, gridDim.x, sh);
}

// List-free Lanczos matvec (FP32 monodisperse, no preconditioner): one
// thread per particle in blocks of PSE_NOLIST_THREADS, compact table in
// shared memory.  The sample then builds no neighbour list.
__global__ void __launch_bounds__(PSE_NOLIST_THREADS) k_lz_matvec_nolist(
    int64_t N, Geom<float> g, const Rec<float> *__restrict__ rec, const int *__restrict__ cell_start,
    const V4<float> *__restrict__ pos_sorted, const V4<float> *__restrict__ table_c, V4<float> *u,
    double *partials, LzState *lz, const V4<float> *__restrict__ add) {
    __shared__ double sh[32];
    __shared__ V4<float> tab_s[PSE_TABLEC_N];
    for (int i = threadIdx.x; i < PSE_TABLEC_N; i += blockDim.x) tab_s[i] = table_c[i];
    __syncthreads();
    lz_matvec_body<float, 1, 1, true, false, true>(N, 0, g, rec, nullptr, nullptr, tab_s, u, partials, lz, nullptr,
                                                   nullptr, add, blockIdx.x, gridDim.x, sh, cell_start, pos_sorted);
}

// Fused over the systems of a batch: block b works for system blk2sys[b].
__global__ void __launch_bounds__(PSE_BATCH_MV_THREADS) k_lz_matvec_batch(const LzSys *__restrict__ sys,
                                                                          const int *__restrict__ blk2sys) {
    __shared__ double sh[32];
    __shared__ V4<float> tab_s[PSE_TABLEC_N];
    const LzSys &S = sys[blk2sys[blockIdx.x]];
    for (int i = threadIdx.x; i < PSE_TABLEC_N; i += blockDim.x) tab_s[i] = S.table_c[i];
    __syncthreads();
    lz_matvec_body<float, PSE_BATCH_MV_TPP, PSE_BATCH_MV_ILP, true>(S.N, S.K, S.g, S.rec, S.count, S.nbr, tab_s, S.u, S.part_mv,
                                                     S.lz, S.pc, S.basis, nullptr, blockIdx.x - S.blk_mv, S.nblk_mv,
                                                     sh);
}

// ------------------------------------------------------------------ Lanczos update
// Lanczos update of one system: block 0 is its T_j block (first, so that it is
// placed at once in a launch of several waves), blocks 1 .. nblk do the vectors.
template <typename T>
__device__ __forceinline__ void lz_update_body(int64_t N, V4<T> *basis, Rec<T> *rec, const V4<T> *u, double *partials,
                                               LzState *lz, double *qlws, const float *__restrict__ pc,
                                               const LzStop &st, int bidx, int nblk, double *sh, EigSmem *esm) {
    EigIn in;
    if (bidx == 0 && threadIdx.x < 32) in.fetch(lz, threadIdx.x);
    const int j = lz->iter;
    if (j > PSE_MAXIT || !lz->active) return;
    double bsum = 0.0;
    if (bidx == 0) {
        if (threadIdx.x < 32) lz_eig_body(lz, j, st, esm, qlws, in);
        __syncthreads();  // its writes are the ticket's to release
    } else {
        const T cu = (T)lz->c_u, cq = (T)lz->c_q, cp = (T)lz->c_p;
        const V4<T> *qj = basis + (int64_t)(j - 1) * N;
        const V4<T> *qp = basis + (int64_t)(j - 2) * N;
        V4<T> *qn = basis + (int64_t)j * N;
        typename Part<T>::type part = 0;
        for (int64_t s = (bidx - 1) * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)nblk * blockDim.x) {
            const V4<T> us = u[s];
            const V4<T> a = qj[s];
            V4<T> w;
            w.x = cu * us.x - cq * a.x;
            w.y = cu * us.y - cq * a.y;
            w.z = cu * us.z - cq * a.z;
            w.w = T(0);
            if (j >= 2) {
                const V4<T> b = qp[s];
                w.x -= cp * b.x;
                w.y -= cp * b.y;
                w.z -= cp * b.z;
            }
            qn[s] = w;
            if constexpr (sizeof(T) == 4) {
                if (pc) {
                    V4<T> p;
                    sym3_apply(pc + s * 16, w.x, w.y, w.z, p.x, p.y, p.z);
                    p.w = T(0);
                    rec[s].q = p;
                } else if (rec) {
                    rec[s].q = w;
                }
            } else if (rec) {
                rec[s].q = w;
            }
            part += w.x * w.x + w.y * w.y + w.z * w.z;
        }
        bsum = block_total<T>(part, sh);
    }
    double total;
    if (grid_sum_last(bsum, partials, &lz->counter_up, sh, &total, bidx, nblk + 1)) {
        // every block is done: join beta_j with the T_j block's decision
        __shared__ int s_stop;
        if (threadIdx.x == 0) {
            const double bi = total > 0.0 ? rsqrt_f64(total) : 0.0;
            lz->beta[j] = total * bi;
            lz->binv[j] = bi;
            lz->iter = j + 1;
            // beta_j = 0: the Krylov space is invariant and T_j^{1/2} e_1 is exact
            const bool breakdown = st.fixed_iter <= 0 && !(total > 0.0);
            const int stop = __ldcg(&lz->stop_y) || breakdown;
            if (breakdown) lz->converged = 1;
            if (stop) lz->J = j;
            lz->cont = stop ? 0 : 1;
            s_stop = stop;
            if (st.h) cudaGraphSetConditional(st.h, stop ? 0u : 1u);
        }
        __syncthreads();
        if (s_stop)  // coefficients of the final combination
            for (int i = threadIdx.x; i < j; i += blockDim.x)
                lz->coef[i] = (float)(__ldcg(&lz->beta[0]) * __ldcg(&lz->y[i]) * __ldcg(&lz->binv[i]));
    }
}

// (five FP32 blocks per SM)
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 1) k_lz_update(int64_t N, V4<T> *basis, Rec<T> *rec, const V4<T> *u,
                                                   double *partials, LzState *lz, double *qlws,
                                                   const float *__restrict__ pc, LzStop st) {
    __shared__ double sh[32];
    __shared__ EigSmem esm;
    lz_update_body<T>(N, basis, rec, u, partials, lz, qlws, pc, st, blockIdx.x, gridDim.x - 1, sh, &esm);
}

__global__ void __launch_bounds__(256, 5) k_lz_update_batch(const LzSys *__restrict__ sys, const int *__restrict__ blk2sys) {
    __shared__ double sh[32];
    __shared__ EigSmem esm;
    const LzSys &S = sys[blk2sys[blockIdx.x]];
    lz_update_body<float>(S.N, S.basis, S.rec, S.u, S.part_up, S.lz, S.qlws, S.pc, S.stop, blockIdx.x - S.blk_up,
                          S.nblk_up, sh, &esm);
}

// One thread per system: the systems whose stop test passed in this loop
// body become inactive for the next one; the shared WHILE node continues
// while any system is still active.
__global__ void k_batch_cond(LzState *const *lzs, int nsys, cudaGraphConditionalHandle h, int *any_out) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < nsys; k += blockDim.x) {
        LzState *lz = lzs[k];
        const int c = lz->active && lz->cont;
        lz->active = c;
        if (c) atomicOr(&any, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (h) cudaGraphSetConditional(h, any ? 1u : 0u);
        if (any_out) *any_out = any;
    }
}

// ------------------------------------------------------------------ final combination
// x_s = sum_{i=1..J} coef_i q_i[s]  (+ wave part), written in caller order.
// On the forces path (udet != null) out = c_noise x + c_det M_r F + wave, the
// wave part already carrying both weights.
// Three consecutive floats of a caller-order (N, 3) array in two stores:
// of two consecutive 4-byte aligned addresses one is 8-byte aligned, and the
// pair starting there goes out as one float2 (the scattered output writes
// are a third fewer).
__device__ __forceinline__ void store3(float *p, float x, float y, float z) {
    if ((reinterpret_cast<uintptr_t>(p) & 7) == 0) {
        *reinterpret_cast<float2 *>(p) = make_float2(x, y);
        p[2] = z;
    } else {
        p[0] = x;
        *reinterpret_cast<float2 *>(p + 1) = make_float2(y, z);
    }
}

template <typename T>
__device__ __forceinline__ void lz_final_body(int64_t N, const SampleArgs<T> *args, const V4<T> *pos_sorted,
                                              const V4<T> *basis, const V4<T> *uwave, const LzState *lz,
                                              bool with_wave, const float *__restrict__ pc, const V4<T> *udet,
                                              int64_t s) {
    __shared__ T cf[PSE_MAXIT + 2];
    __shared__ double cfd[PSE_MAXIT + 2];
    const int J = lz->J;
    for (int i = threadIdx.x; i < J; i += blockDim.x) {
        if constexpr (sizeof(T) == 4) cf[i] = lz->coef[i];
        else cfd[i] = lz->beta[0] * lz->y[i] / lz->beta[i];
    }
    __syncthreads();
    if (s >= N) return;
    T x = 0, y = 0, z = 0;
    for (int i = 0; i < J; ++i) {
        T c;
        if constexpr (sizeof(T) == 4) c = cf[i];
        else c = cfd[i];
        const V4<T> q = basis[(int64_t)i * N + s];
        x += c * q.x;
        y += c * q.y;
        z += c * q.z;
    }
    if constexpr (sizeof(T) == 4) {
        if (pc) {  // real part = S^{-1} (S M_r S)^{1/2} z1
            T a, b, c;
            sym3_apply(pc + s * 16 + 8, x, y, z, a, b, c);
            x = a; y = b; z = c;
        }
    }
    const int64_t o = 3 * w_bits_r(pos_sorted[s].w);
    T wx = 0, wy = 0, wz = 0;
    if (with_wave) {
        const V4<T> w = uwave[s];
        wx = w.x; wy = w.y; wz = w.z;
    }
    if (args->real) { args->real[o] = x; args->real[o + 1] = y; args->real[o + 2] = z; }
    if (args->wave && with_wave) { args->wave[o] = wx; args->wave[o + 1] = wy; args->wave[o + 2] = wz; }
    if (udet) {
        const T cn = (T)args->c_noise, cd = (T)args->c_det;
        const V4<T> m = udet[s];
        x = cn * x + cd * m.x;
        y = cn * y + cd * m.y;
        z = cn * z + cd * m.z;
    }
    if (args->out) {
        if constexpr (sizeof(T) == 4) {
            store3(args->out + o, x + wx, y + wy, z + wz);
        } else {
            args->out[o] = x + wx; args->out[o + 1] = y + wy; args->out[o + 2] = z + wz;
        }
    }
}

template <typename T>
__global__ void k_lz_final(int64_t N, const SampleArgs<T> *args, const V4<T> *pos_sorted, const V4<T> *basis,
                           const V4<T> *uwave, const LzState *lz, bool with_wave, const float *__restrict__ pc,
                           const V4<T> *udet) {
    lz_final_body<T>(N, args, pos_sorted, basis, uwave, lz, with_wave, pc, udet,
                     blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
}

// One block of 256 particles per launch block: each block's particles belong
// to one system (blocks never straddle systems).
__global__ void k_lz_final_batch(const BSys *__restrict__ sys, const int *__restrict__ tab) {
    const BSys &S = sys[tab[blockIdx.x]];
    const int lb = (int)blockIdx.x - S.b0[BK_FINAL];
    lz_final_body<float>(S.N, S.d.args, S.d.pos_sorted, S.d.basis, S.d.uwave, S.d.lz, true, S.d.pc_on, nullptr,
                         lb * (int64_t)blockDim.x + threadIdx.x);
}

// Forces path without noise: out = c_det M_r F + wave part (c_det M_w F), caller order.
template <typename T>
__global__ void k_det_final(int64_t N, const SampleArgs<T> *args, const V4<T> *pos_sorted, const V4<T> *udet,
                            const V4<T> *uwave) {
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N) return;
    const int64_t o = 3 * w_bits_r(pos_sorted[s].w);
    const T cd = (T)args->c_det;
    const V4<T> m = udet[s], w = uwave[s];
    args->out[o] = cd * m.x + w.x;
    args->out[o + 1] = cd * m.y + w.y;
    args->out[o + 2] = cd * m.z + w.z;
}

// ------------------------------------------------------------------ Brownian dynamics step
// Overlap repulsion F_s = k_rep sum_t (2a - r) rhat over the list entries of
// s closer than 2a (pair vectors from cell-local offsets, as in the matvec),
// plus the external force, written in caller order.
// TPP lanes per particle take every TPP-th entry, four of them in flight.
// Bound by the latency of entry -> offsets: one entry at a time took 25 us at
// 3e4 particles, on a step's critical path.  Steps in us (one lane and one
// entry; 1, 4 and 16 lanes with four): 3e4 particles 198; 184, 179, 183, FP64
// 1e3 -; 257, 235, 233, 1e5 -; 314, 312, 323, 3e5 -; 835, 836, 868, 1e6 -;
// 2233, 2259, 2396: four lanes up to PSE_REP_LANES, one above.
#define PSE_REP_LANES 200000
template <typename T, int TPP>
__global__ void k_repulsion(int64_t N, Geom<T> g, const SampleArgs<T> *args, const V4<T> *__restrict__ loc,
                            const int *__restrict__ count, const int *__restrict__ nbr,
                            const V4<T> *__restrict__ pos_sorted, T *F) {
    constexpr int U = 4;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int sub = (int)(t & (TPP - 1));
    const int64_t s = t / TPP < N ? t / TPP : N - 1;  // the last groups past the end repeat particle N - 1
    const V4<T> li = loc[s];
    const T two_a = T(2) * g.a, k = (T)args->k_rep;
    T fx = 0, fy = 0, fz = 0;
    const int cnt = count[s];
    for (int q0 = sub; q0 < cnt; q0 += U * TPP) {
        int e[U];
        V4<T> l[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = q0 + u * TPP;
            e[u] = q < cnt ? nbr[(int64_t)q * N + s] : -1;  // -1: removed by the float64 decision at r_cut
        }
#pragma unroll
        for (int u = 0; u < U; ++u) l[u] = loc[e[u] < 0 ? s : e[u] >> 6];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int ox = ((e[u] >> 4) & 3) - 1, oy = ((e[u] >> 2) & 3) - 1, oz = (e[u] & 3) - 1;
            const T dx = (li.x - l[u].x) - (T(ox) * g.cs + T(ox) * g.cs_lo);
            const T dy = (li.y - l[u].y) - (T(oy) * g.cs + T(oy) * g.cs_lo);
            const T dz = (li.z - l[u].z) - (T(oz) * g.cs + T(oz) * g.cs_lo);
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (e[u] >= 0 && r2 < two_a * two_a && r2 > T(0)) {
                const T r = sqrt_hd(r2);
                const T f = k * (two_a - r) / r;
                fx += f * dx;
                fy += f * dy;
                fz += f * dz;
            }
        }
    }
#pragma unroll
    for (int o = TPP / 2; o; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
    }
    if (sub || t / TPP >= N) return;
    const int64_t o = 3 * w_bits_r(pos_sorted[s].w);
    if (args->fext) {
        fx += args->fext[o];
        fy += args->fext[o + 1];
        fz += args->fext[o + 2];
    }
    F[o] = fx;
    F[o + 1] = fy;
    F[o + 2] = fz;
}

// x <- x + dx, wrapped into [0, L) (caller order).
template <typename T> __global__ void k_advance(int64_t N, Geom<T> g, const SampleArgs<T> *args) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= 3 * N || !args->advance) return;
    T x = args->advance[i] + args->out[i];
    x -= g.L * floor_hd(x / g.L);
    if (x >= g.L || x < T(0)) x = T(0);
    args->advance[i] = x;
}

// ------------------------------------------------------------------ caller-vector matvec
template <typename T>
__global__ void k_gather_vec(int64_t N, const SampleArgs<T> *args, const V4<T> *pos_sorted, Rec<T> *rec, V4<T> *vec) {
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= N) return;
    const int64_t o = 3 * w_bits_r(pos_sorted[s].w);
    V4<T> v;
    v.x = args->vin[o]; v.y = args->vin[o + 1]; v.z = args->vin[o + 2]; v.w = T(0);
    if (vec) vec[s] = v;
    else rec[s].q = v;
}

template <typename T, int TPP, bool POLY = false>
__global__ void __launch_bounds__(128) k_matvec_scatter(int64_t N, int K, const SampleArgs<T> *args, Geom<T> g,
                                                        const Rec<T> *rec, const int *count, const int *nbr,
                                                        const V4<T> *table, const V4<T> *pos_sorted) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t s = tid / TPP;
    const int lane_g = (int)(tid % TPP);
    const bool active = s < N;
    V4<T> li, qi;
    T ax, ay, az;
    mr_row_part<T, TPP, 4, false, POLY>(N, s, lane_g, active, K, g, rec, count, nbr, table, li, qi, ax, ay, az);
    if (!active || lane_g != 0) return;
    const int64_t i = 3 * w_bits_r(pos_sorted[s].w);
    const T self = POLY ? self_of(g, spec_of(li)) : g.self_m;
    args->out[i] = ax + self * qi.x;
    args->out[i + 1] = ay + self * qi.y;
    args->out[i + 2] = az + self * qi.z;
}

// M_r v for v already gathered into the records; output in sorted order.
template <typename T, int TPP>
__global__ void __launch_bounds__(128) k_matvec_sorted(int64_t N, int K, Geom<T> g, const Rec<T> *rec,
                                                       const int *count, const int *nbr, const V4<T> *table,
                                                       V4<T> *out) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t s = tid / TPP;
    const int lane_g = (int)(tid % TPP);
    const bool active = s < N;
    V4<T> li, qi;
    T ax, ay, az;
    mr_row_part<T, TPP, 4>(N, s, lane_g, active, K, g, rec, count, nbr, table, li, qi, ax, ay, az);
    if (!active || lane_g != 0) return;
    V4<T> o;
    o.x = ax + g.self_m * qi.x;
    o.y = ay + g.self_m * qi.y;
    o.z = az + g.self_m * qi.z;
    o.w = T(0);
    out[s] = o;
}

// ------------------------------------------------------------------ launchers
static inline unsigned nb(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }
// persistent grid: at most `per_sm` resident blocks per SM
static inline unsigned pgrid(int64_t work_items, int items_per_block, int per_sm) {
    const int64_t need = (work_items + items_per_block - 1) / items_per_block;
    const int64_t cap = (int64_t)num_sms() * per_sm;
    return (unsigned)(need < cap ? (need > 0 ? need : 1) : cap);
}

static constexpr int kMvTpp = 4;

template <typename T>
void launch_lz_init(int64_t N, const SampleArgs<T> *args, int system, const Dev<T> &d, cudaStream_t s) {
    k_lz_init<T><<<pgrid(N, 256, 8), 256, 0, s>>>(N, args, system, d.pos_sorted, d.basis, rec_q(d), d.partials, d.lz,
                                                  sizeof(T) == 4 ? d.pc_on : nullptr);
}
// Matvec launch shapes (threads per particle, independent gathers per thread),
// selected by Geom::mv; the sampler may time them all and keep the fastest.
// Persistent grid: one wave of resident blocks (at most 16 per SM), so that
// no second, partly filled wave of equal-work blocks trails the first.
template <typename T, int TPP, int ILP, int BS = 128> int mv_blocks_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_matvec<T, TPP, ILP, BS>, BS, 0) != cudaSuccess ||
            nb < 1) {
            cudaGetLastError();
            nb = BS >= 1024 ? 1 : 2048 / BS;
        }
        per_sm = nb < 16 ? nb : 16;
    }
    return per_sm;
}
// resident blocks per SM of the fused batch matvec (at most 16)
int matvec_blocks_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_matvec_batch, PSE_BATCH_MV_THREADS, 0) !=
                cudaSuccess ||
            nb < 1) {
            cudaGetLastError();
            nb = 1;
        }
        per_sm = nb < 16 ? nb : 16;
    }
    return per_sm;
}
// the same for the Lanczos update (FP32 and FP64), at most 8 per SM
template <typename T> int up_blocks_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_update<T>, 256, 0) != cudaSuccess || nb < 1) {
            cudaGetLastError();
            nb = 8;
        }
        per_sm = nb < 8 ? nb : 8;
    }
    return per_sm;
}
int update_blocks_per_sm() { return up_blocks_per_sm<float>(); }
// occupancy of every matvec shape, queried once outside any stream capture
static int mv_poly_blocks_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_matvec_poly, 1024, 0) != cudaSuccess || nb < 1) {
            cudaGetLastError();
            nb = 1;
        }
        per_sm = nb;
    }
    return per_sm;
}
static int mv_nolist_blocks_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_matvec_nolist, PSE_NOLIST_THREADS, 0) !=
                cudaSuccess ||
            nb < 1) {
            cudaGetLastError();
            nb = 1;
        }
        per_sm = nb;
    }
    return per_sm;
}
// Launch geometry of the brick-tiled matvec: the staging capacity follows the
// mean neighbourhood occupancy 216 N / ncell^3 with six standard deviations
// of Poisson slack; blocks per SM from the shared memory that leaves.
static size_t g_tile_static_smem = 0, g_sm_smem = 0;
static int g_tile_regs = 0;
static int tile_cap(int64_t N, int nc) {
    const double mean = 216.0 * (double)N / ((double)nc * nc * nc);
    int cap = (int)(mean + 6.0 * sqrt(mean) + 32.0);
    cap = (cap + 31) & ~31;
    return cap < 256 ? 256 : (cap > 4096 ? 4096 : cap);
}
static void tile_prepare() {
    if (g_sm_smem) return;
    int dev = 0, v = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
        cudaFuncGetAttributes(&fa, k_lz_matvec_tiled) == cudaSuccess &&
        cudaFuncSetAttribute(k_lz_matvec_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             4096 * (int)sizeof(Rec<float>)) == cudaSuccess) {
        g_tile_static_smem = fa.sharedSizeBytes;
        g_tile_regs = fa.numRegs;
        g_sm_smem = (size_t)v;
    } else {
        cudaGetLastError();
    }
}
static int tile_blocks_per_sm(size_t dyn) {
    if (!g_sm_smem) return 1;
    const size_t per_block = g_tile_static_smem + dyn + 1024;  // 1 KB per block reserved by the runtime
    int nb = (int)(g_sm_smem / per_block);
    const int by_regs = 65536 / ((g_tile_regs > 0 ? g_tile_regs : 64) * PSE_TILE_THREADS);
    nb = nb < by_regs ? nb : by_regs;
    nb = nb < 2048 / PSE_TILE_THREADS ? nb : 2048 / PSE_TILE_THREADS;
    return nb > 0 ? nb : 1;
}

template <typename T> void mv_prepare_all() {
    mv_blocks_per_sm<T, 4, 4>(); mv_blocks_per_sm<T, 8, 2>();
    mv_blocks_per_sm<T, 16, 1>(); mv_blocks_per_sm<T, 4, 2>();
    mv_blocks_per_sm<T, 4, 4, 1024>(); mv_blocks_per_sm<T, 4, 4, 512>();
    mv_blocks_per_sm<T, 8, 2, 1024>(); mv_blocks_per_sm<T, 4, 2, 1024>();
    mv_blocks_per_sm<T, 1, 4, 1024>(); mv_blocks_per_sm<T, 2, 4, 1024>();
    if constexpr (sizeof(T) == 4) {
        mv_poly_blocks_per_sm();
        mv_nolist_blocks_per_sm();
    }
}
static void stored_prepare();
void matvec_prepare() {
    tile_prepare();
    mv_prepare_all<float>();
    mv_prepare_all<double>();
    up_blocks_per_sm<float>(); up_blocks_per_sm<double>();
    matvec_blocks_per_sm();
    stored_prepare();
}

template <typename T, int TPP, int ILP, int BS = 128>
void mv_launch(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    k_lz_matvec<T, TPP, ILP, BS><<<pgrid(N, BS / TPP, mv_blocks_per_sm<T, TPP, ILP, BS>()), BS, 0, s>>>(
        N, nbr_k(N, d.nbr_cap), g, d.rec, d.nbr_count, d.nbr, d.table, d.table_c, d.u, d.partials, d.lz,
        sizeof(T) == 4 ? d.pc_on : nullptr, d.basis, d.mv_add);
}
// Stored pair blocks: threads per particle by N (few particles need more
// threads each to fill the GPU and to shorten the chain of columns).
template <typename F> static void with_stored_tpp(int64_t N, F &&f) {
    using std::integral_constant;
    if (N >= 60000) f(integral_constant<int, 2>{});
    else if (N >= 15000) f(integral_constant<int, 4>{});
    else f(integral_constant<int, 16>{});
}
// one wave of resident blocks (at most 8 per SM)
template <int TPP> static int stored_per_sm() {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_lz_matvec_stored<TPP>, PSE_STORED_THREADS, 0) !=
                cudaSuccess ||
            nb < 1) {
            cudaGetLastError();
            nb = 1;
        }
        per_sm = nb < 8 ? nb : 8;
    }
    return per_sm;
}
static void stored_prepare() {
    stored_per_sm<2>();
    stored_per_sm<4>();
    stored_per_sm<16>();
}
template <typename T> void launch_pairs(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    if constexpr (sizeof(T) == 8) {
        if (!stored(d)) return;
        with_stored_tpp(N, [&](auto tpp) {
            k_pairs<tpp()><<<nb(N * tpp(), PSE_STORED_THREADS), PSE_STORED_THREADS, 0, s>>>(
                N, d.pair_cols, g, d.loc_sorted, d.nbr_count, d.nbr, d.table, d.pair, d.pent);
        });
    }
}
template <typename T> void launch_lz_matvec(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    if constexpr (sizeof(T) == 8) {
        if (stored(d)) {
            with_stored_tpp(N, [&](auto tpp) {
                k_lz_matvec_stored<tpp()>
                    <<<pgrid(N, PSE_STORED_THREADS / tpp(), stored_per_sm<tpp()>()), PSE_STORED_THREADS, 0, s>>>(
                        N, d.pair_cols, g, d.basis, d.loc_sorted, d.nbr_count, d.nbr, d.pair, d.pent, d.table, d.u,
                        d.partials, d.lz, d.mv_add);
            });
            return;
        }
    }
    if constexpr (sizeof(T) == 4) {
        if (g.mv == PSE_MV_TILED && g.nspec <= 1 && !d.pc_on && g_sm_smem) {
            const int cap = tile_cap(N, g.nc);
            const size_t dyn = (size_t)cap * sizeof(Rec<float>);
            const int nbricks = g.nb * g.nb * g.nb;
            k_lz_matvec_tiled<<<pgrid(nbricks, 1, tile_blocks_per_sm(dyn)), PSE_TILE_THREADS, dyn, s>>>(
                N, nbr_k(N, d.nbr_cap), g, d.rec, d.cell_start, d.nbr_count, d.nbr, d.table_c, d.u, d.partials, d.lz,
                d.mv_add, nbricks, cap);
            return;
        }
        if (g.mv == PSE_MV_NOLIST && g.nspec <= 1 && !d.pc_on) {
            k_lz_matvec_nolist<<<pgrid(N, PSE_NOLIST_THREADS, mv_nolist_blocks_per_sm()), PSE_NOLIST_THREADS, 0, s>>>(
                N, g, d.rec, d.cell_start, d.pos_sorted, d.table_c, d.u, d.partials, d.lz, d.mv_add);
            return;
        }
        if (g.nspec > 1) {
            k_lz_matvec_poly<<<pgrid(N, 1024 / 4, mv_poly_blocks_per_sm()), 1024, 0, s>>>(
                N, nbr_k(N, d.nbr_cap), g, d.rec, d.nbr_count, d.nbr, d.table, d.u, d.partials, d.lz, d.basis);
            return;
        }
    }
    switch (g.mv) {
        case 1: mv_launch<T, 8, 2>(N, g, d, s); break;
        case 2: mv_launch<T, 16, 1>(N, g, d, s); break;
        case 3: mv_launch<T, 4, 2>(N, g, d, s); break;
        case 4:
        case PSE_MV_TILED: mv_launch<T, 4, 4, 1024>(N, g, d, s); break;
        case 5: mv_launch<T, 4, 4, 512>(N, g, d, s); break;
        case 6: mv_launch<T, 8, 2, 1024>(N, g, d, s); break;
        case 7: mv_launch<T, 4, 2, 1024>(N, g, d, s); break;
        case 8: mv_launch<T, 1, 4, 1024>(N, g, d, s); break;
        case 9: mv_launch<T, 2, 4, 1024>(N, g, d, s); break;
        default: mv_launch<T, 4, 4>(N, g, d, s); break;
    }
}
// the T_j^{1/2} e_1 block and the vector blocks, together one wave of resident
// blocks at most (one block more than that trailed it by a block's time: 19.5
// -> 22 us at N = 1e6)
template <typename T>
void launch_lz_update(int64_t N, const LzStop &stop, const Dev<T> &d, cudaStream_t s) {
    const unsigned most = (unsigned)num_sms() * up_blocks_per_sm<T>(), vec = (unsigned)((N + 255) / 256);
    k_lz_update<T><<<vec < most ? vec + 1 : most, 256, 0, s>>>(
        N, d.basis, rec_q(d), d.u, d.partials + num_sms() * 16 + 32, d.lz, d.qlws, sizeof(T) == 4 ? d.pc_on : nullptr,
        stop);
}
void launch_batch_cond(LzState *const *lzs, int nsys, cudaGraphConditionalHandle h, cudaStream_t s, int *any_out) {
    k_batch_cond<<<1, 256, 0, s>>>(lzs, nsys, h, any_out);
}
void launch_lz_matvec_batch(const LzSys *sys, const int *blk2sys, int nblocks, cudaStream_t s) {
    k_lz_matvec_batch<<<nblocks, PSE_BATCH_MV_THREADS, 0, s>>>(sys, blk2sys);
}
void launch_lz_update_batch(const LzSys *sys, const int *blk2sys, int nblocks, cudaStream_t s) {
    k_lz_update_batch<<<nblocks, 256, 0, s>>>(sys, blk2sys);
}
void launch_batch_init(const BSys *sys, int *const *tab, const int *nblk, cudaStream_t s) {
    k_lz_init_batch<<<nblk[BK_INIT], 256, 0, s>>>(sys, tab[BK_INIT]);
}
void launch_batch_final(const BSys *sys, int *const *tab, const int *nblk, cudaStream_t s) {
    k_lz_final_batch<<<nblk[BK_FINAL], 256, 0, s>>>(sys, tab[BK_FINAL]);
}
template <typename T>
void launch_lz_final(int64_t N, const SampleArgs<T> *args, const Dev<T> &d, bool with_wave, cudaStream_t s) {
    k_lz_final<T><<<nb(N, 256), 256, 0, s>>>(N, args, d.pos_sorted, d.basis, d.uwave, d.lz, with_wave,
                                             sizeof(T) == 4 ? d.pc_on : nullptr, nullptr);
}
template <typename T>
void launch_lz_final_forces(int64_t N, const SampleArgs<T> *args, const Dev<T> &d, cudaStream_t s) {
    k_lz_final<T><<<nb(N, 256), 256, 0, s>>>(N, args, d.pos_sorted, d.basis, d.uwave, d.lz, true,
                                             sizeof(T) == 4 ? d.pc_on : nullptr, d.udet);
}
template <typename T> void launch_repulsion(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    auto go = [&](auto kernel, int tpp) {
        kernel<<<nb(N * tpp, 128), 128, 0, s>>>(N, g, d.args, d.loc_sorted, d.nbr_count, d.nbr, d.pos_sorted, d.bd_force);
    };
    if (N < PSE_REP_LANES) go(k_repulsion<T, 4>, 4);
    else go(k_repulsion<T, 1>, 1);
}
template <typename T> void launch_advance(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    k_advance<T><<<nb(3 * N, 256), 256, 0, s>>>(N, g, d.args);
}
template <typename T> void launch_det_final(int64_t N, const SampleArgs<T> *args, const Dev<T> &d, cudaStream_t s) {
    k_det_final<T><<<nb(N, 256), 256, 0, s>>>(N, args, d.pos_sorted, d.udet, d.uwave);
}
// the vector goes to the records, or to d.u for the stored pair blocks
template <typename T> void launch_gather_vec(int64_t N, const SampleArgs<T> *args, const Dev<T> &d, cudaStream_t s) {
    k_gather_vec<T><<<nb(N, 256), 256, 0, s>>>(N, args, d.pos_sorted, d.rec, stored(d) ? d.u : nullptr);
}
template <typename T> void launch_matvec_sorted(int64_t N, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    if constexpr (sizeof(T) == 8) {
        if (stored(d)) {
            with_stored_tpp(N, [&](auto tpp) {
                k_matvec_stored<tpp()>
                    <<<pgrid(N, PSE_STORED_THREADS / tpp(), stored_per_sm<tpp()>()), PSE_STORED_THREADS, 0, s>>>(
                        N, d.pair_cols, g, d.u, d.loc_sorted, d.nbr_count, d.nbr, d.pair, d.pent, d.table, d.udet);
            });
            return;
        }
    }
    k_matvec_sorted<T, kMvTpp><<<nb(N * kMvTpp, 128), 128, 0, s>>>(N, nbr_k(N, d.nbr_cap), g, d.rec, d.nbr_count,
                                                                    d.nbr, d.table, d.udet);
}
template <typename T>
void launch_matvec_caller(int64_t N, const SampleArgs<T> *args, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    k_gather_vec<T><<<nb(N, 256), 256, 0, s>>>(N, args, d.pos_sorted, d.rec, nullptr);
    if (g.nspec > 1)
        k_matvec_scatter<T, kMvTpp, true><<<nb(N * kMvTpp, 128), 128, 0, s>>>(N, nbr_k(N, d.nbr_cap), args, g, d.rec,
                                                                              d.nbr_count, d.nbr, d.table,
                                                                              d.pos_sorted);
    else
        k_matvec_scatter<T, kMvTpp><<<nb(N * kMvTpp, 128), 128, 0, s>>>(N, nbr_k(N, d.nbr_cap), args, g, d.rec,
                                                                         d.nbr_count, d.nbr, d.table,
                                                                         d.pos_sorted);
}

#define PSE_INST(T)                                                                                          \
    template void launch_lz_init<T>(int64_t, const SampleArgs<T> *, int, const Dev<T> &, cudaStream_t);        \
    template void launch_lz_matvec<T>(int64_t, Geom<T>, const Dev<T> &, cudaStream_t);                       \
    template void launch_pairs<T>(int64_t, Geom<T>, const Dev<T> &, cudaStream_t);                           \
    template void launch_lz_update<T>(int64_t, const LzStop &, const Dev<T> &, cudaStream_t);                \
    template void launch_lz_final<T>(int64_t, const SampleArgs<T> *, const Dev<T> &, bool, cudaStream_t);    \
    template void launch_lz_final_forces<T>(int64_t, const SampleArgs<T> *, const Dev<T> &, cudaStream_t);   \
    template void launch_det_final<T>(int64_t, const SampleArgs<T> *, const Dev<T> &, cudaStream_t);         \
    template void launch_repulsion<T>(int64_t, Geom<T>, const Dev<T> &, cudaStream_t);                       \
    template void launch_advance<T>(int64_t, Geom<T>, const Dev<T> &, cudaStream_t);                         \
    template void launch_gather_vec<T>(int64_t, const SampleArgs<T> *, const Dev<T> &, cudaStream_t);        \
    template void launch_matvec_sorted<T>(int64_t, Geom<T>, const Dev<T> &, cudaStream_t);                   \
    template void launch_matvec_caller<T>(int64_t, const SampleArgs<T> *, Geom<T>, const Dev<T> &, cudaStream_t);
PSE_INST(float)
PSE_INST(double)
#undef PSE_INST

}  // namespace pse
