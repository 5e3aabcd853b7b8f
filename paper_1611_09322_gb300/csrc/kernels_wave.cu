// Wave-space sample M_w^{1/2} dW2 (Sec. II B 2): complex Hermitian noise,
// B^{1/2} scaling with the Gaussian deconvolution, inverse FFT (three passes
// of our own where fft_wins_* says so, else cuFFT C2R launched by the host), and
// Gaussian interpolation S^dagger = h^3 S^T at the particles; the forces
// path's spreading and forward transform.  sm_103a.
//
// Per mode k = 2 pi n / L of the half spectrum (nz >= 0):
//   vhat(k) = V^{-1/2} sinc(ka)/k sqrt(1 + k^2/4xi^2) exp(-(1 - eta) k^2 / 8xi^2)
//             (I - kk) dW2(k)
// which, interpolated with g(r) = (2xi^2/(pi eta))^{3/2} exp(-2 xi^2 r^2 / eta)
// (Fourier transform exp(-eta k^2 / 8 xi^2)), reproduces the eq. Mwave
// factor sinc^2(ka) H(k, xi) / (V k^2) in the covariance.
#include "pse_internal.cuh"

namespace pse {

template <typename T> struct Cplx;
template <> struct Cplx<float> { using type = cufftComplex; };
template <> struct Cplx<double> { using type = cufftDoubleComplex; };

template <typename T> __device__ __forceinline__ T exp_t(T x) {
    if constexpr (sizeof(T) == 4) return expf(x);
    else return exp(x);
}

// Mode (ix, iy, iz) of the half spectrum, iz in [0, M/2]: signed indices,
// and whether it carries noise (k != 0, no Nyquist index).
struct ModeIdx {
    int ix, iy, iz, nx, ny, nz;
    bool live;
};
// n / d for 32-bit n with the multiplier m and shift l of d >= 2
// (Granlund and Montgomery, PLDI 1994, the round-up method).
__device__ __forceinline__ uint32_t udiv_magic(uint32_t n, uint32_t m, int l) {
    const uint32_t t1 = __umulhi(m, n);
    return (t1 + ((n - t1) >> 1)) >> (l - 1);
}
template <typename T> __device__ __forceinline__ ModeIdx mode_of(int64_t t, const WaveGeom<T> &w) {
    ModeIdx m;
    const int M = w.M, Mh1 = w.Mh1;
    if (!w.big) {
        const uint32_t u = (uint32_t)t;
        const uint32_t r = udiv_magic(u, w.dv_h1_m, w.dv_h1_l);
        const uint32_t x = udiv_magic(r, w.dv_M_m, w.dv_M_l);
        m.iz = (int)(u - r * (uint32_t)Mh1);
        m.iy = (int)(r - x * (uint32_t)M);
        m.ix = (int)x;
    } else {
        m.iz = (int)(t % Mh1);
        m.iy = (int)((t / Mh1) % M);
        m.ix = (int)(t / ((int64_t)Mh1 * M));
    }
    const int half = M / 2;
    m.nx = m.ix <= half ? m.ix : m.ix - M;
    m.ny = m.iy <= half ? m.iy : m.iy - M;
    m.nz = m.iz;
    const bool nyq = (M % 2) == 0 && (m.ix == half || m.iy == half || m.iz == half);
    m.live = !nyq && (m.nx | m.ny | m.nz) != 0;
    return m;
}

// dW2 of a live mode: the noise of a {k, -k} pair is keyed by its
// representative (nz > 0, or nz = 0 and (ny > 0 or (ny = 0 and nx > 0))),
// id q = (ix*M + iy)*Mh1 + iz, Philox blocks 2q and 2q+1; a mode holding the
// partner draws the same numbers and conjugates them, so the kz = 0 plane is
// exactly Hermitian.
template <typename T>
__device__ __forceinline__ void mode_noise(const ModeIdx &m, int M, int Mh1, uint32_t strm, uint64_t seed,
                                           uint64_t sample, T wr[3], T wi[3]) {
    int rx = m.ix, ry = m.iy;
    bool conj = false;
    if (m.nz == 0 && !(m.ny > 0 || (m.ny == 0 && m.nx > 0))) {
        rx = (M - m.ix) % M;
        ry = (M - m.iy) % M;
        conj = true;
    }
    const uint32_t q = (uint32_t)(((int64_t)rx * M + ry) * Mh1 + m.iz);
    const Normals4<T> a = normals4<T>(2u * q, strm, seed, sample);
    const Normals4<T> b = normals4<T>(2u * q + 1u, strm, seed, sample);
    const T s2 = T(0.70710678118654752440);
    wr[0] = a.v[0] * s2; wr[1] = a.v[2] * s2; wr[2] = b.v[0] * s2;
    wi[0] = a.v[1] * s2; wi[1] = a.v[3] * s2; wi[2] = b.v[1] * s2;
    if (conj) { wi[0] = -wi[0]; wi[1] = -wi[1]; wi[2] = -wi[2]; }
}

// Unit wave vector and the noise scale
//   sc(k) = V^{-1/2} sinc(ka)/k sqrt(1 + k^2/4xi^2) exp(-(1 - eta) k^2 / 8xi^2)
// of a live mode.  sc and 1/|n| depend on the integer n^2 = nx^2 + ny^2 + nz^2
// only; both come from a table evaluated in FP64 on the host.
template <typename T>
__device__ __forceinline__ T mode_scale(const ModeIdx &m, const WaveGeom<T> &w, T &hx, T &hy, T &hz) {
    const int n2 = m.nx * m.nx + m.ny * m.ny + m.nz * m.nz;
    T sc, inv;
    if constexpr (sizeof(T) == 4) {
        const float2 e = __ldg(reinterpret_cast<const float2 *>(w.sc_tab) + n2);
        sc = e.x;
        inv = e.y;
    } else {
        const double2 e = __ldg(reinterpret_cast<const double2 *>(w.sc_tab) + n2);
        sc = e.x;
        inv = e.y;
    }
    hx = T(m.nx) * inv;
    hy = T(m.ny) * inv;
    hz = T(m.nz) * inv;
    return sc;
}

// One thread per half-spectrum mode: vhat = sc(k) (I - kk) dW2(k); k = 0 and
// Nyquist modes are zero.
template <typename T>
__device__ __forceinline__ void wave_noise_elem(int64_t t, const WaveGeom<T> &w, const SampleArgs<T> *args,
                                                int system, typename Cplx<T>::type *spec, int64_t plane) {
    using C = typename Cplx<T>::type;
    const ModeIdx m = mode_of(t, w);
    C o0, o1, o2;
    o0.x = o0.y = o1.x = o1.y = o2.x = o2.y = T(0);
    T pr[3] = {T(0), T(0), T(0)}, pi[3] = {T(0), T(0), T(0)};  // (I - kk) dW2
    int n2 = 0;
    T sc = T(0);
    if (m.live) {
        T wr[3], wi[3];
        mode_noise<T>(m, w.M, w.Mh1, 2u * system + 1u, args->seed, args->sample, wr, wi);
        T hx, hy, hz;
        sc = mode_scale<T>(m, w, hx, hy, hz);
        n2 = m.nx * m.nx + m.ny * m.ny + m.nz * m.nz;
        const T dr = hx * wr[0] + hy * wr[1] + hz * wr[2];
        const T di = hx * wi[0] + hy * wi[1] + hz * wi[2];
        pr[0] = wr[0] - hx * dr; pi[0] = wi[0] - hx * di;
        pr[1] = wr[1] - hy * dr; pi[1] = wi[1] - hy * di;
        pr[2] = wr[2] - hz * dr; pi[2] = wi[2] - hz * di;
    }
    o0.x = sc * pr[0]; o0.y = sc * pi[0];
    o1.x = sc * pr[1]; o1.y = sc * pi[1];
    o2.x = sc * pr[2]; o2.y = sc * pi[2];
    spec[t] = o0;
    spec[plane + t] = o1;
    spec[2 * plane + t] = o2;
    // polydisperse: species s scales the same noise with its own shape factor
    for (int sp = 1; sp < w.nspec; ++sp) {
        const T scs = m.live ? w.sc_tab[sp * w.sc_stride + 2 * n2] : T(0);
        C *o = spec + (int64_t)sp * 3 * plane;
        C q;
        q.x = scs * pr[0]; q.y = scs * pi[0]; o[t] = q;
        q.x = scs * pr[1]; q.y = scs * pi[1]; o[plane + t] = q;
        q.x = scs * pr[2]; q.y = scs * pi[2]; o[2 * plane + t] = q;
    }
}

template <typename T>
__global__ void k_wave_noise(WaveGeom<T> w, const SampleArgs<T> *args, int system, typename Cplx<T>::type *spec,
                             int64_t plane) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < (int64_t)w.M * w.M * w.Mh1) wave_noise_elem<T>(t, w, args, system, spec, plane);
}

// Mode factor applied in place to a forward (R2C) spectrum, one thread per
// half-spectrum mode, k = 0 and Nyquist set to zero:
//   WAVE_MODE_DET:       vhat = c_det norm sc^2 (I - kk) Fhat  [+ c_noise sc (I - kk) dW2]
//     Fhat = DFT of the unnormalised spread grid sum_i w_x w_y w_z F_i; with the
//     Gaussian's constant norm = (2xi^2/(pi eta))^{3/2} h^3 this is
//     h^3 B(k)/V (I - kk) DFT(S F), the deterministic wave product, and the
//     optional k-space noise term fuses the Brownian wave part into the same
//     inverse FFT (Sec. III);
//   WAVE_MODE_GRIDNOISE: vhat = c_noise sc M^{-3/2} (I - kk) What, What the DFT of white
//     grid noise, which on every live mode pair has the law of dW2.
template <typename T>
__global__ void k_wave_apply(WaveGeom<T> w, const SampleArgs<T> *args, int system, typename Cplx<T>::type *spec,
                             int64_t plane, int mode, int with_noise) {
    using C = typename Cplx<T>::type;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t nmodes = (int64_t)w.M * w.M * w.Mh1;
    if (t >= nmodes) return;
    const ModeIdx m = mode_of(t, w);
    C o[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c].x = o[c].y = T(0);
    if (m.live) {
        T hx, hy, hz;
        const T sc = mode_scale<T>(m, w, hx, hy, hz);
        const C i0 = spec[t], i1 = spec[plane + t], i2 = spec[2 * plane + t];
        T f;
        if (mode == WAVE_MODE_DET) f = (T)args->c_det * w.norm * sc * sc;
        else f = (T)args->c_noise * sc * w.inv_M15;
        T vr[3] = {i0.x, i1.x, i2.x}, vi[3] = {i0.y, i1.y, i2.y};
        const T dr = hx * vr[0] + hy * vr[1] + hz * vr[2];
        const T di = hx * vi[0] + hy * vi[1] + hz * vi[2];
        const T hh[3] = {hx, hy, hz};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[c].x = f * (vr[c] - hh[c] * dr);
            o[c].y = f * (vi[c] - hh[c] * di);
        }
        if (mode == WAVE_MODE_DET && with_noise) {
            T wr[3], wi[3];
            mode_noise<T>(m, w.M, w.Mh1, 2u * system + 1u, args->seed, args->sample, wr, wi);
            const T g = (T)args->c_noise * sc;
            const T er = hx * wr[0] + hy * wr[1] + hz * wr[2];
            const T ei = hx * wi[0] + hy * wi[1] + hz * wi[2];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                o[c].x += g * (wr[c] - hh[c] * er);
                o[c].y += g * (wi[c] - hh[c] * ei);
            }
        }
    }
    spec[t] = o[0];
    spec[plane + t] = o[1];
    spec[2 * plane + t] = o[2];
}

// White noise on the grid: node g = (ix*M + iy)*M + iz keys one Philox block
// on the wave stream; its first three normals are the x, y, z components.
template <typename T>
__global__ void k_grid_noise(int64_t M3, const SampleArgs<T> *args, int system, T *grid) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= M3) return;
    const Normals4<T> n = normals4<T>((uint32_t)g, 2u * system + 1u, args->seed, args->sample);
    grid[g] = n.v[0];
    grid[M3 + g] = n.v[1];
    grid[2 * M3 + g] = n.v[2];
}

// Support start and fractional offset of one coordinate: s = x M / L as a
// float-float product, i0 = floor(s - P/2) + 1 decided exactly, and
// u = s - i0 in [P/2 - 1, P/2) (grid units).
__device__ __forceinline__ void support(float x, const WaveGeom<float> &w, int &i0, float &u) {
    const float hi = x * w.gl_hi;
    const float lo = fmaf(x, w.gl_lo, fmaf(x, w.gl_hi, -hi));
    const float th = hi - 0.5f * (float)w.P;  // exact: P/2 lies on the ulp grid of hi
    float fl = floorf(th);
    float rem = (th - fl) + lo;
    // rem = s - P/2 - fl to float rounding; its sign decides the floor.  A
    // tiny negative rem moves the support down one node, and rem + 1 may
    // round to 1: keep it just below 1 so that it does not move back.
    if (rem < 0.f) {
        fl -= 1.f;
        rem = fminf(rem + 1.f, 0.99999994f);
    } else if (rem >= 1.f) {
        fl += 1.f;
        rem -= 1.f;
    }
    i0 = (int)fl + 1;
    u = rem + 0.5f * (float)w.P - 1.f;
}
__device__ __forceinline__ void support(double x, const WaveGeom<double> &w, int &i0, double &u) {
    const double hi = x * w.gl_hi;
    const double lo = fma(x, w.gl_hi, -hi);
    const double th = hi - 0.5 * w.P;
    double fl = floor(th);
    double rem = (th - fl) + lo;
    if (rem < 0.0) {  // as in the float form: a tiny negative rem must not round back to 1
        fl -= 1.0;
        rem = fmin(rem + 1.0, 0.99999999999999989);
    } else if (rem >= 1.0) {
        fl += 1.0;
        rem -= 1.0;
    }
    i0 = (int)fl + 1;
    u = rem + 0.5 * w.P - 1.0;
}

#define PSE_PMAX 16

__device__ __forceinline__ int wrap_grid(int i, int M) {  // valid for i in [-M, 2M)
    i = i < 0 ? i + M : i;
    return i >= M ? i - M : i;
}

// ------------------------------------------------------------------ spreading
// Grid force density (unnormalised): grid_c(x_g) += sum_i w_x w_y w_z F_i,c over
// each particle's P^3 support, w = exp(-ch2 (u - p)^2) per axis as in the
// interpolation (the Gaussian's constant is applied in the mode factor).
//
// FP64, the planar interpolation and a tile asked for: one CTA per tile of
// G^3 cells (FP32 with the node-major grid: k_spread4).  The tile's particles
// (cell-sorted, so each cell is a contiguous run) are spread into a padded E^3 node block in shared
// memory with shared-memory atomics, CP components per pass.  The block
// starts at the node orig[t] of each axis (host-computed: the support start of
// the tile's lower corner less one node) and E bounds the support of every
// particle of the tile with one node of margin on each side.  Two ways out:
//   scratch != null: the block is stored to scratch[tile][component] (plain
//     coalesced stores); k_spread_gather then sums, for every grid node, the
//     blocks that cover it (no global atomics);
//   scratch == null: the block is added to the grid with one coalesced float
//     atomic per nonzero node.
// A particle whose support still falls outside the block (not expected, kept
// for safety) adds straight into the global grid, which is cleared first.
#define PSE_SPREAD_THREADS 1024  // threads per CTA (occupancy while the shared atomics wait)
#define PSE_SPREAD_CHUNK 256     // particles staged per pass

__device__ __forceinline__ int pmod(int i, int M) {
    const int r = i % M;
    return r < 0 ? r + M : r;
}

template <typename T> __device__ __forceinline__ int64_t caller_of(T w) {
    if constexpr (sizeof(T) == 4) return (int64_t)__float_as_int(w);
    else return (int64_t)__double_as_longlong(w);
}

template <typename T>
__global__ void __launch_bounds__(PSE_SPREAD_THREADS)
    k_spread(WaveGeom<T> w, Geom<T> g, SpreadTile st, const int *__restrict__ orig, const V4<T> *__restrict__ pos_sorted,
             const int *__restrict__ cell_start, const SampleArgs<T> *args, T *grid, T *scratch,
             const Rec<T> *__restrict__ src) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int E = st.E, E2 = E * E, E3 = E2 * E, P = w.P, CP = st.CP, G = st.G, M = w.M;
    const int64_t M3 = (int64_t)M * M * M;
    T *tile = (T *)smem_raw;                                // CP * E^3
    T *wts = tile + CP * E3;                                // CHUNK * 3P
    T *fv = wts + PSE_SPREAD_CHUNK * 3 * P;                 // CHUNK * 3
    int *base = (int *)(fv + PSE_SPREAD_CHUNK * 3);         // CHUNK
    int *cst = base + PSE_SPREAD_CHUNK;                     // 64: first sorted index of each cell
    int *coff = cst + 64;                                   // 65: prefix of the cells' counts
    __shared__ int s_ncell;

    const int t = blockIdx.x;
    const int tz = t % st.ntx, ty = (t / st.ntx) % st.ntx, tx = t / (st.ntx * st.ntx);
    const int c0x = tx * G, c0y = ty * G, c0z = tz * G;
    const int ox = orig[tx], oy = orig[ty], oz = orig[tz];
    // cells of the tile and their particle runs
    const int G3 = G * G * G;
    if (threadIdx.x < G3) {
        const int a = threadIdx.x / (G * G), b = (threadIdx.x / G) % G, c = threadIdx.x % G;
        const int cx = c0x + a, cy = c0y + b, cz = c0z + c;
        int s0 = 0, n = 0;
        if (cx < g.nc && cy < g.nc && cz < g.nc) {
            const int id = cell_id(cx, cy, cz, g.nb);
            s0 = cell_start[id];
            n = cell_start[id + 1] - s0;
        }
        cst[threadIdx.x] = s0;
        coff[threadIdx.x + 1] = n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        coff[0] = 0;
        for (int j = 1; j <= G3; ++j) coff[j] += coff[j - 1];
        s_ncell = G3;
    }
    __syncthreads();
    const int ntile = coff[s_ncell];
    T *out = scratch ? scratch + (int64_t)t * 3 * E3 : nullptr;
    if (ntile == 0) {
        if (out)
            for (int i = threadIdx.x; i < 3 * E3; i += blockDim.x) out[i] = T(0);
        return;
    }
    const int PP = P * P;

    for (int cp0 = 0; cp0 < 3; cp0 += CP) {
        for (int i = threadIdx.x; i < CP * E3; i += blockDim.x) tile[i] = T(0);
        __syncthreads();
        for (int p0 = 0; p0 < ntile; p0 += PSE_SPREAD_CHUNK) {
            const int np = min(PSE_SPREAD_CHUNK, ntile - p0);
            if (threadIdx.x < np) {
                const int k = p0 + threadIdx.x;
                int lo = 0, hi = s_ncell - 1;  // last cell j with coff[j] <= k
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (coff[mid] <= k) lo = mid;
                    else hi = mid - 1;
                }
                const int64_t si = cst[lo] + (k - coff[lo]);
                const V4<T> p = pos_sorted[si];
                int i0x, i0y, i0z;
                T ux, uy, uz;
                support(p.x, w, i0x, ux);
                support(p.y, w, i0y, uy);
                support(p.z, w, i0z, uz);
                T *wv = wts + threadIdx.x * 3 * P;
                for (int q = 0; q < P; ++q) {
                    const T dx = ux - T(q), dy = uy - T(q), dz = uz - T(q);
                    wv[q] = exp_t(-w.ch2 * dx * dx);
                    wv[P + q] = exp_t(-w.ch2 * dy * dy);
                    wv[2 * P + q] = exp_t(-w.ch2 * dz * dz);
                }
                T *f = fv + threadIdx.x * 3;
                if (src) {  // a sorted-order vector (the Lanczos vector of the full-mobility iteration)
                    const V4<T> q = src[si].q;
                    f[0] = q.x; f[1] = q.y; f[2] = q.z;
                } else {
                    const T *F = args->vin + 3 * caller_of(p.w);
                    f[0] = F[0]; f[1] = F[1]; f[2] = F[2];
                }
                const int lx = i0x - ox, ly = i0y - oy, lz = i0z - oz;
                const bool inside = lx >= 0 && ly >= 0 && lz >= 0 && lx + P <= E && ly + P <= E && lz + P <= E;
                base[threadIdx.x] = inside ? (lx * E + ly) * E + lz : -1;
                if (!inside) {
                    for (int a = 0; a < P; ++a)
                        for (int b = 0; b < P; ++b)
                            for (int c = 0; c < P; ++c) {
                                const T wt = wv[a] * wv[P + b] * wv[2 * P + c];
                                const int64_t gi =
                                    ((int64_t)pmod(i0x + a, M) * M + pmod(i0y + b, M)) * M + pmod(i0z + c, M);
                                for (int cc = 0; cc < CP; ++cc) atomicAdd(grid + (cp0 + cc) * M3 + gi, wt * f[cp0 + cc]);
                            }
                }
            }
            __syncthreads();
            // thread t owns the (y, z) node pair q = t mod P^2 of particles
            // t / P^2, t / P^2 + stride, ...: no divisions in the loop
            const int stride = blockDim.x / PP;
            if (threadIdx.x < stride * PP) {
                const int q = threadIdx.x % PP, b = q / P, c = q - b * P;
                for (int pp = threadIdx.x / PP; pp < np; pp += stride) {
                    const int b0 = base[pp];
                    if (b0 < 0) continue;
                    const T *wv = wts + pp * 3 * P;
                    const T *f = fv + pp * 3 + cp0;
                    const T wyz = wv[P + b] * wv[2 * P + c];
                    const int row = b0 + b * E + c;
                    for (int a = 0; a < P; ++a) {
                        const T wt = wv[a] * wyz;
                        for (int cc = 0; cc < CP; ++cc) atomicAdd(tile + cc * E3 + row + a * E2, wt * f[cc]);
                    }
                }
            }
            __syncthreads();
        }
        if (out) {
            for (int i = threadIdx.x; i < CP * E3; i += blockDim.x) out[cp0 * E3 + i] = tile[i];
        } else {
            for (int i = threadIdx.x; i < E3; i += blockDim.x) {
                const int lz = i % E, ly = (i / E) % E, lx = i / E2;
                const int64_t gi = ((int64_t)pmod(ox + lx, M) * M + pmod(oy + ly, M)) * M + pmod(oz + lz, M);
                for (int cc = 0; cc < CP; ++cc) {
                    const T v = tile[cc * E3 + i];
                    if (v != T(0)) atomicAdd(grid + (cp0 + cc) * M3 + gi, v);
                }
            }
        }
        __syncthreads();
    }
}

// Second phase of the two-phase spreading: one thread per grid node (z
// fastest, so the reads of one block row are coalesced) adds the values the
// covering tile blocks hold for it.  cover[x * PSE_COVER + k] = (tile index
// along the axis, node offset in that tile's block) for the cnt[x] blocks
// covering node x along one axis (the same on the three axes of a cube).
template <typename T>
__global__ void __launch_bounds__(256) k_spread_gather(int M, int E, int ntx, const int2 *__restrict__ cover,
                                                       const int *__restrict__ cnt, const T *__restrict__ scratch,
                                                       T *grid) {
    const int64_t M3 = (int64_t)M * M * M;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= M3) return;
    const int z = (int)(g % M), y = (int)((g / M) % M), x = (int)(g / ((int64_t)M * M));
    const int E3 = E * E * E;
    const int nx = cnt[x], ny = cnt[y], nz = cnt[z];
    T a0 = 0, a1 = 0, a2 = 0;
    for (int i = 0; i < nx; ++i) {
        const int2 cx = cover[x * PSE_COVER + i];
        for (int j = 0; j < ny; ++j) {
            const int2 cy = cover[y * PSE_COVER + j];
            for (int k = 0; k < nz; ++k) {
                const int2 cz = cover[z * PSE_COVER + k];
                const int64_t tb = ((int64_t)(cx.x * ntx + cy.x) * ntx + cz.x) * 3 * E3;
                const int off = (cx.y * E + cy.y) * E + cz.y;
                a0 += scratch[tb + off];
                a1 += scratch[tb + E3 + off];
                a2 += scratch[tb + 2 * E3 + off];
            }
        }
    }
    grid[g] += a0;
    grid[M3 + g] += a1;
    grid[2 * M3 + g] += a2;
}

size_t spread_smem_bytes(SpreadTile st, int P, size_t elem) {
    return elem * ((size_t)st.CP * st.E * st.E * st.E + (size_t)PSE_SPREAD_CHUNK * (3 * P + 3)) +
           sizeof(int) * (PSE_SPREAD_CHUNK + 64 + 65);
}

// G lanes per sorted particle (G = 8, 16 or 32 divides the warp):
// u_w = norm * sum_{P^3} g_x g_y g_z v(node), separable weights
// exp(-ch2 (u - p)^2) per axis, periodic node indices.  Lane g of the group
// owns the (y, z) node pairs g, g + G, ...; for each x node the group's loads
// are runs of consecutive floats along z (the grid's contiguous axis).  The
// first P lanes of the group evaluate the 3P one-dimensional weights, shared
// by shuffles inside the group.
template <typename T, int G>
__device__ __forceinline__ void interp_particle(int64_t s, bool active, int lg, int gbase, const WaveGeom<T> &w,
                                                const V4<T> *__restrict__ pos_sorted, const T *__restrict__ grid,
                                                V4<T> *uwave) {
    const V4<T> p = pos_sorted[active ? s : 0];
    const int M = w.M, P = w.P;
    const int64_t M3 = (int64_t)M * M * M;
    int i0x, i0y, i0z;
    T ux, uy, uz;
    support(p.x, w, i0x, ux);
    support(p.y, w, i0y, uy);
    support(p.z, w, i0z, uz);
    T wxl = 0, wyl = 0, wzl = 0;
    if (lg < P) {
        const T dx = ux - T(lg), dy = uy - T(lg), dz = uz - T(lg);
        wxl = exp_t(-w.ch2 * dx * dx);
        wyl = exp_t(-w.ch2 * dy * dy);
        wzl = exp_t(-w.ch2 * dz * dz);
    }
    T ax = 0, ay = 0, az = 0;
    const int PP = P * P;
    for (int q0 = 0; q0 < PP; q0 += G) {
        const int q = q0 + lg;
        const bool on = active && q < PP;
        const int b = q < PP ? q / P : 0;
        const int c = q < PP ? q - b * P : 0;
        const T wy = __shfl_sync(0xffffffffu, wyl, gbase + (b < G ? b : 0));
        const T wz = __shfl_sync(0xffffffffu, wzl, gbase + (c < G ? c : 0));
        const int iy = wrap_grid(i0y + b, M), iz = wrap_grid(i0z + c, M);
        const T wyz = wy * wz;
        const int64_t rowyz = (int64_t)iy * M + iz;
        for (int a = 0; a < P; ++a) {
            const T wx = __shfl_sync(0xffffffffu, wxl, gbase + (a < G ? a : 0));
            if (on) {
                const int64_t idx = (int64_t)wrap_grid(i0x + a, M) * M * M + rowyz;
                const T wt = wx * wyz;
                ax += wt * __ldg(grid + idx);
                ay += wt * __ldg(grid + M3 + idx);
                az += wt * __ldg(grid + 2 * M3 + idx);
            }
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, o);
        ay += __shfl_xor_sync(0xffffffffu, ay, o);
        az += __shfl_xor_sync(0xffffffffu, az, o);
    }
    if (active && lg == 0) {
        V4<T> o;
        o.x = ax * w.norm; o.y = ay * w.norm; o.z = az * w.norm; o.w = T(0);
        uwave[s] = o;
    }
}

// Fused over the systems of a batch (wave noise of every system's half
// spectrum; interpolation with 16 lanes per particle, P <= 16).
__global__ void k_wave_noise_batch(const BSys *__restrict__ sys, const int *__restrict__ tab) {
    const BSys &S = sys[tab[blockIdx.x]];
    const int lb = (int)blockIdx.x - S.b0[BK_NOISE];
    const int64_t plane = (int64_t)S.w.M * S.w.M * S.w.Mh1;
    const int64_t stride = (int64_t)S.nb[BK_NOISE] * blockDim.x;
    for (int64_t t = lb * (int64_t)blockDim.x + threadIdx.x; t < plane; t += stride)
        wave_noise_elem<float>(t, S.w, S.d.args, S.system, (cufftComplex *)S.d.spec, plane);
}

// One lane group per particle, one launch-wide pass.
template <typename T, int G>
__global__ void __launch_bounds__(128) k_interp(int64_t N, WaveGeom<T> w, const V4<T> *__restrict__ pos_sorted,
                                                const T *__restrict__ grid, V4<T> *uwave) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lg = threadIdx.x % G;
    interp_particle<T, G>(tid / G, tid / G < N, lg, (threadIdx.x & 31) - lg, w, pos_sorted, grid, uwave);
}

__global__ void __launch_bounds__(128) k_interp_batch(const BSys *__restrict__ sys, const int *__restrict__ tab) {
    constexpr int G = PSE_BATCH_INTERP_G;
    const BSys &S = sys[tab[blockIdx.x]];
    const int lb = (int)blockIdx.x - S.b0[BK_INTERP];
    const int lg = threadIdx.x % G;
    const int64_t per_block = blockDim.x / G;
    for (int64_t base = lb * per_block; base < S.N; base += (int64_t)S.nb[BK_INTERP] * per_block) {  // uniform
        const int64_t s = base + threadIdx.x / G;
        interp_particle<float, G>(s, s < S.N, lg, (threadIdx.x & 31) - lg, S.w, S.d.pos_sorted, S.d.grid, S.d.uwave);
    }
}

// Node-major copy of the three planar velocity grids: one 16-byte record
// (x, y, z, 0) per node, so that the interpolation reads a node with one load.
__global__ void k_grid_aos(int64_t M3, const float *__restrict__ g, V4<float> *__restrict__ g4) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= M3) return;
    V4<float> v;
    v.x = __ldg(g + i);
    v.y = __ldg(g + M3 + i);
    v.z = __ldg(g + 2 * M3 + i);
    v.w = 0.f;
    g4[i] = v;
}

// Interpolation from the node-major grid: a group of P lanes per particle,
// floor(32 / P) particles per warp (consecutive in cell order, so their
// supports overlap in L1).  Lane c of a group owns the z-node c of the
// support and walks the P x P (x, y) columns, one 16-byte load per node; it
// evaluates the 1-D weights of index c on all three axes, which the group's
// lanes exchange by shuffles.  The group's partial sums meet in its first lane.
template <int P>
__device__ __forceinline__ void interp4_warp(int64_t warp0, int64_t N, const WaveGeom<float> &w,
                                             const V4<float> *__restrict__ pos_sorted,
                                             const V4<float> *__restrict__ grid4, V4<float> *uwave,
                                             const V4<float> *__restrict__ loc = nullptr) {
    constexpr int R = 32 / P;  // particles per warp; lanes R P .. 31 idle
    const int lane = threadIdx.x & 31;
    const int g = lane / P, c = lane - (lane / P) * P;
    const int64_t s = warp0 + g;
    const bool act = g < R && s < N;
    const int base = (g < R ? g : 0) * P;  // first lane of the group
    const V4<float> p = pos_sorted[act ? s : 0];
    const int M = w.M;
    if (loc) {  // polydisperse: the grid of this particle's species
        const int sp = (__float_as_int(loc[act ? s : 0].w) >> PSE_SPECIES_SHIFT) & 3;
        grid4 += (int64_t)sp * M * M * M;
    }
    int i0x, i0y, i0z;
    float ux, uy, uz;
    support(p.x, w, i0x, ux);
    support(p.y, w, i0y, uy);
    support(p.z, w, i0z, uz);
    const float fc = float(c);
    const float ex = ux - fc, ey = uy - fc, ez = uz - fc;
    const float wxc = expf(-w.ch2 * ex * ex);
    const float wyc = expf(-w.ch2 * ey * ey);
    const float wzc = expf(-w.ch2 * ez * ez);
    const int izc = wrap_grid(i0z + c, M);
    float wyz[P];
    int row[P];
#pragma unroll
    for (int b = 0; b < P; ++b) {
        wyz[b] = __shfl_sync(0xffffffffu, wyc, base + b) * wzc;
        row[b] = wrap_grid(i0y + b, M) * M + izc;
    }
    const float4 *g4 = reinterpret_cast<const float4 *>(grid4);
    const int64_t MM = (int64_t)M * M;
    float ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll 1
    for (int a = 0; a < P; ++a) {
        const float wxa = __shfl_sync(0xffffffffu, wxc, base + a);
        const float4 *plane = g4 + wrap_grid(i0x + a, M) * MM;
        if (act) {
#pragma unroll
            for (int b = 0; b < P; ++b) {
                const float4 v = __ldg(plane + row[b]);
                const float wt = wxa * wyz[b];
                ax = fmaf(wt, v.x, ax);
                ay = fmaf(wt, v.y, ay);
                az = fmaf(wt, v.z, az);
            }
        }
    }
    float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
    for (int k = 0; k < P; ++k) {
        sx += __shfl_sync(0xffffffffu, ax, base + k);
        sy += __shfl_sync(0xffffffffu, ay, base + k);
        sz += __shfl_sync(0xffffffffu, az, base + k);
    }
    if (act && c == 0) {
        V4<float> o;
        o.x = sx * w.norm; o.y = sy * w.norm; o.z = sz * w.norm; o.w = 0.f;
        uwave[s] = o;
    }
}

template <int P>
__global__ void __launch_bounds__(128) k_interp4(int64_t N, WaveGeom<float> w,
                                                 const V4<float> *__restrict__ pos_sorted,
                                                 const V4<float> *__restrict__ grid4, V4<float> *uwave,
                                                 const V4<float> *__restrict__ loc) {
    const int64_t warp0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * (32 / P);
    if (warp0 >= N) return;  // whole warps leave together
    interp4_warp<P>(warp0, N, w, pos_sorted, grid4, uwave, loc);
}

// Fused over the systems of a batch: the node-major copy of every system's
// grid, then the interpolation of every system (all with the same P).
__global__ void k_grid_aos_batch(const BSys *__restrict__ sys, const int *__restrict__ tab) {
    const BSys &S = sys[tab[blockIdx.x]];
    const int lb = (int)blockIdx.x - S.b0[BK_COPY];
    const int64_t M3 = (int64_t)S.w.M * S.w.M * S.w.M;
    const int64_t stride = (int64_t)S.nb[BK_COPY] * blockDim.x;
    for (int64_t i = lb * (int64_t)blockDim.x + threadIdx.x; i < M3; i += stride) {
        V4<float> v;
        v.x = __ldg(S.d.grid + i);
        v.y = __ldg(S.d.grid + M3 + i);
        v.z = __ldg(S.d.grid + 2 * M3 + i);
        v.w = 0.f;
        S.d.grid4[i] = v;
    }
}
template <int P> __global__ void __launch_bounds__(128) k_interp4_batch(const BSys *__restrict__ sys,
                                                                         const int *__restrict__ tab) {
    constexpr int R = 32 / P;
    const BSys &S = sys[tab[blockIdx.x]];
    const int lb = (int)blockIdx.x - S.b0[BK_INTERP];
    const int64_t per_block = (blockDim.x / 32) * R;
    const int64_t wofs = (threadIdx.x >> 5) * R;
    for (int64_t base = lb * per_block; base < S.N; base += (int64_t)S.nb[BK_INTERP] * per_block)  // uniform
        if (base + wofs < S.N) interp4_warp<P>(base + wofs, S.N, S.w, S.d.pos_sorted, S.d.grid4, S.d.uwave);
}

// Spreading into the node-major grid, the interpolation's mirror image: a
// group of P lanes per particle, lane c on the z-node c, one 16-byte vector
// reduction (all three components) per node.  Bound by the reductions on
// their way through L1TEX and into L2 (2e5 particles, P = 5: 2.5e7 of them in
// 73 us, 5.5 TB/s of values; L1TEX 84% and L2 70% busy, issue 22%); the tiles
// of k_spread serialise on shared-memory atomics and their blocks pass through
// memory twice more (146 us and 78 us for the gather).  Forces calls, tiles ->
// reductions, us: 1e3 particles 117 -> 114, 1e5 369 -> 305, 2e5 664 -> 493,
// 1e6 2657 -> 1999; P = 9, 1e5 dense 1393 -> 1115, 3e4 dilute 1912 -> 736; no
// density, support or N was found where tiles win.
template <int P>
__global__ void __launch_bounds__(128) k_spread4(int64_t N, WaveGeom<float> w, const V4<float> *__restrict__ pos_sorted,
                                                 const SampleArgs<float> *args, const Rec<float> *__restrict__ src,
                                                 V4<float> *grid4) {
    constexpr int R = 32 / P;
    const int lane = threadIdx.x & 31, g = lane / P, c = lane - g * P;
    const int64_t s = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * R + g;
    const bool act = g < R && s < N;
    const int base = (g < R ? g : 0) * P;
    const V4<float> p = pos_sorted[act ? s : 0];
    const int M = w.M;
    int i0x, i0y, i0z;
    float ux, uy, uz;
    support(p.x, w, i0x, ux);
    support(p.y, w, i0y, uy);
    support(p.z, w, i0z, uz);
    const float fc = float(c), ex = ux - fc, ey = uy - fc, ez = uz - fc;
    const float wxc = expf(-w.ch2 * ex * ex), wyc = expf(-w.ch2 * ey * ey), wzc = expf(-w.ch2 * ez * ez);
    const int izc = wrap_grid(i0z + c, M);
    float fx = 0.f, fy = 0.f, fz = 0.f;
    if (act) {
        if (src) {  // a sorted-order vector (the Lanczos vector of the full-mobility iteration)
            const V4<float> q = src[s].q;
            fx = q.x; fy = q.y; fz = q.z;
        } else {
            const float *F = args->vin + 3 * caller_of(p.w);
            fx = F[0]; fy = F[1]; fz = F[2];
        }
    }
    float wyz[P];
    int row[P];
#pragma unroll
    for (int b = 0; b < P; ++b) {
        wyz[b] = __shfl_sync(0xffffffffu, wyc, base + b) * wzc;
        row[b] = wrap_grid(i0y + b, M) * M + izc;
    }
    const int64_t MM = (int64_t)M * M;
#pragma unroll 1
    for (int a = 0; a < P; ++a) {
        const float wxa = __shfl_sync(0xffffffffu, wxc, base + a);
        V4<float> *plane = grid4 + wrap_grid(i0x + a, M) * MM;
        if (act) {
#pragma unroll
            for (int b = 0; b < P; ++b) {
                const float wt = wxa * wyz[b];
                asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(plane + row[b]),
                             "f"(wt * fx), "f"(wt * fy), "f"(wt * fz), "f"(0.f)
                             : "memory");
            }
        }
    }
}
// Node-major force grid to the planar grids that cuFFT reads.
__global__ void k_grid_planar(int64_t M3, const V4<float> *__restrict__ g4, float *__restrict__ g) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= M3) return;
    const V4<float> v = g4[i];
    g[i] = v.x;
    g[M3 + i] = v.y;
    g[2 * M3 + i] = v.z;
}

static inline unsigned nbw(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <int P>
static void interp4(int64_t N, const WaveGeom<float> &w, const Dev<float> &d, cudaStream_t s) {
    const int64_t warps = (N + 32 / P - 1) / (32 / P);
    k_interp4<P><<<nbw(warps * 32, 128), 128, 0, s>>>(N, w, d.pos_sorted, d.grid4, d.uwave,
                                                      w.nspec > 1 ? d.loc_sorted : nullptr);
}

void launch_batch_noise(const BSys *sys, int *const *tab, const int *nblk, cudaStream_t s) {
    if (nblk[BK_NOISE]) k_wave_noise_batch<<<nblk[BK_NOISE], 256, 0, s>>>(sys, tab[BK_NOISE]);
}
void launch_batch_interp(const BSys *sys, int *const *tab, const int *nblk, int P4, cudaStream_t s) {
    if (P4 == 0) {
        k_interp_batch<<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]);
        return;
    }
    if (nblk[BK_COPY]) k_grid_aos_batch<<<nblk[BK_COPY], 256, 0, s>>>(sys, tab[BK_COPY]);
    switch (P4) {
        case 3: k_interp4_batch<3><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 4: k_interp4_batch<4><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 5: k_interp4_batch<5><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 6: k_interp4_batch<6><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 7: k_interp4_batch<7><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 8: k_interp4_batch<8><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        case 9: k_interp4_batch<9><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
        default: k_interp4_batch<10><<<nblk[BK_INTERP], 128, 0, s>>>(sys, tab[BK_INTERP]); break;
    }
}

// Spread into d.grid4 (cleared here); P in 3..10.
cudaError_t launch_spread4(int64_t N, const WaveGeom<float> &w, const Dev<float> &d, const Rec<float> *src,
                           cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(d.grid4, 0, sizeof(V4<float>) * w.M * w.M * (size_t)w.M, s);
    if (e != cudaSuccess) return e;
    auto go = [&](auto kernel) {
        const int64_t per = 32 / w.P, warps = (N + per - 1) / per;
        kernel<<<nbw(warps * 32, 128), 128, 0, s>>>(N, w, d.pos_sorted, d.args, src, d.grid4);
    };
    switch (w.P) {
        case 3: go(k_spread4<3>); break;
        case 4: go(k_spread4<4>); break;
        case 5: go(k_spread4<5>); break;
        case 6: go(k_spread4<6>); break;
        case 7: go(k_spread4<7>); break;
        case 8: go(k_spread4<8>); break;
        case 9: go(k_spread4<9>); break;
        default: go(k_spread4<10>); break;
    }
    return cudaGetLastError();
}
void launch_grid_planar(const WaveGeom<float> &w, const Dev<float> &d, cudaStream_t s) {
    const int64_t M3 = (int64_t)w.M * w.M * w.M;
    k_grid_planar<<<nbw(M3, 256), 256, 0, s>>>(M3, d.grid4, d.grid);
}
template <typename T>
void launch_wave_noise(WaveGeom<T> w, const SampleArgs<T> *args, int system, void *spec, cudaStream_t s) {
    const int64_t plane = (int64_t)w.M * w.M * w.Mh1;
    k_wave_noise<T><<<nbw(plane, 256), 256, 0, s>>>(w, args, system, (typename Cplx<T>::type *)spec, plane);
}
template <typename T> void launch_grid_copy(WaveGeom<T> w, const Dev<T> &d, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (w.interp_lanes == 0 && w.P >= 3 && w.P <= 10) {
            const int64_t M3 = (int64_t)w.M * w.M * w.M;
            for (int sp = 0; sp < (w.nspec > 1 ? w.nspec : 1); ++sp)  // one grid per species
                k_grid_aos<<<nbw(M3, 256), 256, 0, s>>>(M3, d.grid + (int64_t)sp * 3 * M3, d.grid4 + sp * M3);
        }
    }
}
template <typename T> void launch_interp(int64_t N, WaveGeom<T> w, Geom<T> g, const Dev<T> &d, cudaStream_t s) {
    if constexpr (sizeof(T) == 4) {
        if (w.interp_lanes == 0 && w.P >= 3 && w.P <= 10) {
            switch (w.P) {
                case 3: interp4<3>(N, w, d, s); break;
                case 4: interp4<4>(N, w, d, s); break;
                case 5: interp4<5>(N, w, d, s); break;
                case 6: interp4<6>(N, w, d, s); break;
                case 7: interp4<7>(N, w, d, s); break;
                case 8: interp4<8>(N, w, d, s); break;
                case 9: interp4<9>(N, w, d, s); break;
                default: interp4<10>(N, w, d, s); break;
            }
            return;
        }
    }
    // the group must hold the P lanes that evaluate the 1-D weights
    const int G = w.interp_lanes >= w.P ? w.interp_lanes : (w.P <= 8 ? 8 : (w.P <= 16 ? 16 : 32));
    if (G <= 8) k_interp<T, 8><<<nbw(N * 8, 128), 128, 0, s>>>(N, w, d.pos_sorted, d.grid, d.uwave);
    else if (G <= 16) k_interp<T, 16><<<nbw(N * 16, 128), 128, 0, s>>>(N, w, d.pos_sorted, d.grid, d.uwave);
    else k_interp<T, 32><<<nbw(N * 32, 128), 128, 0, s>>>(N, w, d.pos_sorted, d.grid, d.uwave);
}

template <typename T>
void launch_wave_apply(WaveGeom<T> w, const SampleArgs<T> *args, int system, void *spec, int mode, int with_noise,
                       cudaStream_t s) {
    const int64_t plane = (int64_t)w.M * w.M * w.Mh1;
    k_wave_apply<T><<<nbw(plane, 256), 256, 0, s>>>(w, args, system, (typename Cplx<T>::type *)spec, plane, mode,
                                                    with_noise);
}
template <typename T> void launch_grid_noise(WaveGeom<T> w, const SampleArgs<T> *args, int system, T *grid,
                                             cudaStream_t s) {
    const int64_t M3 = (int64_t)w.M * w.M * w.M;
    k_grid_noise<T><<<nbw(M3, 256), 256, 0, s>>>(M3, args, system, grid);
}
// Opt the spreading kernel in to all the dynamic shared memory a block may
// have on this device (the opt-in limit less the kernel's static shared
// memory); returns that size.  Called once, outside any stream capture.
template <typename T> cudaError_t spread_prepare(size_t *max_dynamic) {
    *max_dynamic = 0;
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_spread<T>);
    if (e != cudaSuccess) return e;
    const size_t avail = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
    e = cudaFuncSetAttribute(k_spread<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)avail);
    if (e == cudaSuccess) *max_dynamic = avail;
    return e;
}
// Spread into d.grid (cleared by the caller).  With a cover table the tile
// blocks go through scratch and the gather kernel; otherwise they are added
// with atomics.
template <typename T>
cudaError_t launch_spread(WaveGeom<T> w, Geom<T> g, SpreadTile st, const int *orig, const int2 *cover,
                          const int *cover_cnt, T *scratch, const Dev<T> &d, cudaStream_t s,
                          const Rec<T> *src) {
    const size_t smem = spread_smem_bytes(st, w.P, sizeof(T));
    const unsigned tiles = (unsigned)st.ntx * st.ntx * st.ntx;
    const bool two_phase = scratch && cover && cover_cnt;
    k_spread<T><<<tiles, PSE_SPREAD_THREADS, smem, s>>>(w, g, st, orig, d.pos_sorted, d.cell_start, d.args, d.grid,
                                                         two_phase ? scratch : nullptr, src);
    if (two_phase) {
        const int64_t M3 = (int64_t)w.M * w.M * w.M;
        k_spread_gather<T><<<nbw(M3, 256), 256, 0, s>>>(w.M, st.E, st.ntx, cover, cover_cnt, scratch, d.grid);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ the sampler's own 3-D transforms
// FP32 grids of 16 <= M <= 512 without prime factors above 7, with the
// node-major interpolation (P = 3..10): the inverse transform of a sample in
// three passes of our own, the noise drawn inside the first and the last one
// writing the node-major records that the interpolation reads, and the forward
// transform of the forces path with the mode factor between the two passes
// over x.  The transforms are bound by memory traffic; against noise kernel +
// cuFFT C2R + node-major copy they save the noise's write and read and the
// planar grids' (noise, x, y / z: M = 200 157 -> 139 / 138 -> 77 us, 189 158
// -> 115 / 135 -> 66, 378 973 -> 1000 / 795 -> 511; fft_wins_* have the rule).
//   x pass: tile of (y, kz) modes, three components: noise (or forward
//           transform over x, mode factor, noise), inverse over x;
//   y pass: per x, tile of kz, one component, in place;
//   z pass: per x, tile of y rows: real transform over kz, two real rows per
//           complex line (z = IDFT(Ya + i Yb): x_a = Re z, x_b = Im z).
// Spectrum layout: ((c M + x) M + y) KP + kz, kz < nkz: rows padded to whole
// sectors, the Nyquist plane of even M (zero: it carries no noise) left out.
// Lines lie in shared memory as [point][line], so that consecutive threads
// touch consecutive words in every pass whatever its stride; each pass is one
// radix of a Stockham transform (natural order in and out), from one buffer
// to the other.  A thread transforms two neighbouring lines at a time (one
// 16-byte access, one set of indices and twiddles for both): with one line per
// thread a point cost 39 instructions a pass (y pass at M = 200 67 us; 48 now,
// of 30 at the memory's rate).  Bound by issue and the latency between the
// barriers of a few blocks: at M = 200 x, y and z issue on 60, 48 and 46% of
// the cycles with a third of the warps resident, z with L1TEX at 71%, DRAM at
// 6, 35 and 31%.
constexpr int PSE_FFT_MAXM = 512;
constexpr int PSE_FFT_TQ = 8;    // (y, kz) modes per block of the x pass
constexpr int PSE_FFT_TX = 256;  // its threads
constexpr int PSE_FFT_TZ = 16;   // kz per block of the y pass
constexpr int PSE_FFT_TY = 256;  // its threads
constexpr int PSE_FFT_TR = 8;    // y rows per block of the z passes
constexpr int PSE_FFT_NL = 3 * PSE_FFT_TR / 2;  // their complex lines
constexpr int PSE_FFT_LS = PSE_FFT_NL + 2;      // room per point: the fill along kz meets 2-way bank conflicts
// Threads of the z passes: a radix-8 pass has M / 8 butterflies on 6 pairs of
// lines, so 384 threads are half idle on small grids while three or more
// blocks of 192 fit an SM (us, 384 -> 192: M = 147 42 -> 33, 200 84 -> 77, 245
// 145 -> 125, 294 260 -> 252); where two blocks fit, 192 are too few (375 554
// -> 648).
constexpr int PSE_FFT_TT_MANY = 384, PSE_FFT_TT_FEW = 192, PSE_FFT_FEW_MAXM = 300;

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 caddf(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csubf(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// i^S a (S = +1 inverse, -1 forward)
template <int S> __device__ __forceinline__ float2 rotf(float2 a) {
    return S > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}
// times e^{S i phi} given (cos phi, sin phi)
template <int S> __device__ __forceinline__ float2 twf(float2 a, float c, float s) {
    return cmulf(a, make_float2(c, S > 0 ? s : -s));
}

// DFT of R points in registers, natural order in and out.
template <int R, int S> struct Dft;
template <int S> struct Dft<2, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float2 a = v[0], b = v[1];
        v[0] = caddf(a, b);
        v[1] = csubf(a, b);
    }
};
template <int S> struct Dft<3, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float2 a = caddf(v[1], v[2]), b = rotf<S>(csubf(v[1], v[2]));
        const float2 m = make_float2(v[0].x - 0.5f * a.x, v[0].y - 0.5f * a.y);
        constexpr float h = 0.86602540378443864676f;
        v[0] = caddf(v[0], a);
        v[1] = make_float2(m.x + h * b.x, m.y + h * b.y);
        v[2] = make_float2(m.x - h * b.x, m.y - h * b.y);
    }
};
template <int S> struct Dft<4, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float2 a = caddf(v[0], v[2]), b = csubf(v[0], v[2]), c = caddf(v[1], v[3]),
                     d = rotf<S>(csubf(v[1], v[3]));
        v[0] = caddf(a, c);
        v[1] = caddf(b, d);
        v[2] = csubf(a, c);
        v[3] = csubf(b, d);
    }
};
// prime R: pairs v[k] +- v[R - k] against the cosines and sines of 2 pi / R
template <int R, int S> __device__ __forceinline__ void dft_prime(float2 *v, const float (&c)[R / 2], const float (&s)[R / 2]) {
    constexpr int H = R / 2;
    float2 a[H], b[H], out[R];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        a[k] = caddf(v[k + 1], v[R - 1 - k]);
        b[k] = rotf<S>(csubf(v[k + 1], v[R - 1 - k]));
    }
    out[0] = v[0];
#pragma unroll
    for (int k = 0; k < H; ++k) out[0] = caddf(out[0], a[k]);
#pragma unroll
    for (int j = 1; j <= H; ++j) {
        float2 e = v[0], o = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            const int r = (j * k) % R;
            const float cc = c[(r <= H ? r : R - r) - 1], ss = r <= H ? s[r - 1] : -s[R - r - 1];
            e.x = fmaf(cc, a[k - 1].x, e.x);
            e.y = fmaf(cc, a[k - 1].y, e.y);
            o.x = fmaf(ss, b[k - 1].x, o.x);
            o.y = fmaf(ss, b[k - 1].y, o.y);
        }
        out[j] = caddf(e, o);
        out[R - j] = csubf(e, o);
    }
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = out[k];
}
template <int S> struct Dft<5, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float c[2] = {0.30901699437494742410f, -0.80901699437494742410f};
        const float s[2] = {0.95105651629515357212f, 0.58778525229247312917f};
        dft_prime<5, S>(v, c, s);
    }
};
template <int S> struct Dft<7, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        const float c[3] = {0.62348980185873353053f, -0.22252093395631440429f, -0.90096886790241912624f};
        const float s[3] = {0.78183148246802980871f, 0.97492791218182360702f, 0.43388373911755812048f};
        dft_prime<7, S>(v, c, s);
    }
};
// R = A B: A-point DFTs over the stride-B subsequences, twiddles w_R^{b j},
// B-point DFTs; TW(b, j, value) applies a twiddle.
template <int A, int B, int S, class TW> __device__ __forceinline__ void dft_split(float2 *v, TW tw) {
    float2 t[A * B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        float2 u[A];
#pragma unroll
        for (int a = 0; a < A; ++a) u[a] = v[a * B + b];
        Dft<A, S>::run(u);
#pragma unroll
        for (int j = 0; j < A; ++j) t[j * B + b] = b * j ? tw(b * j, u[j]) : u[j];
    }
#pragma unroll
    for (int j = 0; j < A; ++j) {
        Dft<B, S>::run(t + j * B);
#pragma unroll
        for (int b = 0; b < B; ++b) v[j + A * b] = t[j * B + b];
    }
}
template <int S> struct Dft<6, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        dft_split<3, 2, S>(v, [](int e, float2 a) {
            return e == 1 ? twf<S>(a, 0.5f, 0.86602540378443864676f) : twf<S>(a, -0.5f, 0.86602540378443864676f);
        });
    }
};
template <int S> struct Dft<8, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        dft_split<4, 2, S>(v, [](int e, float2 a) {
            constexpr float h = 0.70710678118654752440f;
            return e == 1 ? twf<S>(a, h, h) : (e == 2 ? rotf<S>(a) : twf<S>(a, -h, h));
        });
    }
};
template <int S> struct Dft<9, S> {
    static __device__ __forceinline__ void run(float2 *v) {
        dft_split<3, 3, S>(v, [](int e, float2 a) {
            return e == 1   ? twf<S>(a, 0.76604444311897803520f, 0.64278760968653932632f)
                   : e == 2 ? twf<S>(a, 0.17364817766693034885f, 0.98480775301220805937f)
                            : twf<S>(a, -0.93969262078590838405f, 0.34202014332566873304f);
        });
    }
};
// One Stockham pass of radix R over this thread's butterflies j = j0, j0 + dj, ...
// of its two lines.  ld(n): point n of both (x, y the first line's, z, w the
// second's); st(n, value).
template <int R, int S, class Ld, class St>
__device__ __forceinline__ void fft_pass(int M, int ns, uint32_t mg, int j0, int dj, const float2 *tw, Ld ld, St st) {
    const int MR = M / R, step = MR / ns;
    for (int j = j0; j < MR; j += dj) {
        float2 a[R], b[R];
#pragma unroll
        for (int m = 0; m < R; ++m) {
            const float4 v = ld(j + m * MR);
            a[m] = make_float2(v.x, v.y);
            b[m] = make_float2(v.z, v.w);
        }
        int q = j, k = 0;
        if (ns > 1) {
            q = __umulhi((uint32_t)j, mg);
            k = j - q * ns;
            const float2 *t = tw + k * step;
            const float2 *e = t;
#pragma unroll
            for (int m = 1; m < R; ++m, e += k * step) {
                float2 w = *e;
                if (S < 0) w.y = -w.y;
                a[m] = cmulf(a[m], w);
                b[m] = cmulf(b[m], w);
            }
        }
        Dft<R, S>::run(a);
        Dft<R, S>::run(b);
        const int o = q * ns * R + k;
#pragma unroll
        for (int m = 0; m < R; ++m) st(o + m * ns, make_float4(a[m].x, a[m].y, b[m].x, b[m].y));
    }
}
template <int S, class Ld, class St>
__device__ __forceinline__ void fft_pass_any(const FftPlan &p, int i, int j0, int dj, const float2 *tw, Ld ld, St st) {
    switch (p.rad[i]) {  // uniform
        case 2: fft_pass<2, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 3: fft_pass<3, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 4: fft_pass<4, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 5: fft_pass<5, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 6: fft_pass<6, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 7: fft_pass<7, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        case 8: fft_pass<8, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
        default: fft_pass<9, S>(p.M, p.ns[i], p.mg[i], j0, dj, tw, ld, st); break;
    }
}

// Passes [i0, i1) from one shared buffer to the other (L lines of room per
// point, this thread on lines `line` and line + 1, line even; `on`: it has
// lines); returns the buffer that holds the result.  The caller has
// synchronised; so has this on return.
template <int S, int L>
__device__ __forceinline__ float2 *fft_smem(const FftPlan &p, int i0, int i1, int line, bool on, int j0, int dj,
                                            const float2 *tw, float2 *cur, float2 *oth) {
    for (int i = i0; i < i1; ++i) {
        const float2 *in = cur + line;
        float2 *out = oth + line;
        if (on)
            fft_pass_any<S>(p, i, j0, dj, tw, [&](int n) { return *reinterpret_cast<const float4 *>(in + n * L); },
                            [&](int n, float4 v) { *reinterpret_cast<float4 *>(out + n * L) = v; });
        __syncthreads();
        float2 *t = cur;
        cur = oth;
        oth = t;
    }
    return cur;
}

// x pass, blockIdx = (tile of the M KP modes (y, kz), species).
// FORCES false: modes filled with the scaled projected noise; true: the
// forward transform over x of the spread forces' spectrum, the mode factor of
// WAVE_MODE_DET (see k_wave_apply), with noise when with_noise.
// The three components share one second buffer (they are transformed one
// after the other): two blocks fit an SM up to M = 430.
template <bool FORCES>
__global__ void __launch_bounds__(PSE_FFT_TX, 3) k_fft_x(const __grid_constant__ FftPlan p,
                                                         const __grid_constant__ FftJob job, int with_noise) {
    constexpr int TQ = PSE_FFT_TQ, TF = PSE_FFT_TX / TQ, TJ = 2 * TF;
    extern __shared__ __align__(16) float2 fsm[];
    const WaveGeom<float> &w = job.w;
    const int M = p.M, sp = blockIdx.y;
    float2 *A = fsm, *B = A + 3 * M * TQ, *tw = B + M * TQ;
    for (int k = threadIdx.x; k < M; k += PSE_FFT_TX) tw[k] = p.tw[k];
    const int plane = M * p.KP, q0 = blockIdx.x * TQ;
    // transforms: lines (modes) q0 + line, + 1 (plane is a multiple of 4)
    const int line = 2 * (threadIdx.x % (TQ / 2)), jj = threadIdx.x / (TQ / 2);
    const bool on = q0 + line < plane;
    float2 *g = job.spec + (int64_t)sp * 3 * M * plane + q0 + line;  // point n of component c: g[(c M + n) plane]
    __syncthreads();
    if constexpr (FORCES) {
        for (int c = 0; c < 3; ++c) {
            // an even number of shared passes after the first one ends in A
            float2 *Ac = A + c * M * TQ, *cur = (p.nf & 1) ? Ac : B, *oth = (p.nf & 1) ? B : Ac;
            const float2 *gc = g + (int64_t)c * M * plane;
            float2 *a = cur + line;
            if (on)
                fft_pass_any<-1>(p, 0, jj, TJ, tw,
                                 [&](int n) { return *reinterpret_cast<const float4 *>(gc + (int64_t)n * plane); },
                                 [&](int n, float4 v) { *reinterpret_cast<float4 *>(a + n * TQ) = v; });
            __syncthreads();
            fft_smem<-1, TQ>(p, 1, p.nf, line, on, jj, TJ, tw, cur, oth);
        }
    }
    {
        // one mode (of each kx) per thread
        const int fl = threadIdx.x % TQ, q = q0 + fl;
        ModeIdx m;
        m.iy = q / p.KP;
        m.iz = q - m.iy * p.KP;
        m.nz = m.iz;
        m.ny = m.iy <= M / 2 ? m.iy : m.iy - M;
        const bool col = q < plane && m.iz < p.nkz && !((M & 1) == 0 && m.iy == M / 2);
        const uint32_t strm = 2u * job.system + 1u;
        const uint64_t seed = job.args->seed, sample = job.args->sample;
        const float cd = FORCES ? (float)job.args->c_det * w.norm : 0.f, cn = FORCES ? (float)job.args->c_noise : 1.f;
        for (int kx = threadIdx.x / TQ; kx < M; kx += TF) {
            m.ix = kx;
            m.nx = kx <= M / 2 ? kx : kx - M;
            m.live = col && !((M & 1) == 0 && kx == M / 2) && (m.nx | m.ny | m.nz) != 0;
            float2 o[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            float2 *at = A + kx * TQ + fl;
            if (m.live) {
                float hx, hy, hz;
                float sc = mode_scale<float>(m, w, hx, hy, hz);
                if (!FORCES && sp) sc = w.sc_tab[sp * w.sc_stride + 2 * (m.nx * m.nx + m.ny * m.ny + m.nz * m.nz)];
                const float hh[3] = {hx, hy, hz};
                if constexpr (FORCES) {
                    const float f = cd * sc * sc;
                    const float2 v[3] = {at[0], at[M * TQ], at[2 * M * TQ]};
                    const float dr = hx * v[0].x + hy * v[1].x + hz * v[2].x;
                    const float di = hx * v[0].y + hy * v[1].y + hz * v[2].y;
#pragma unroll
                    for (int d = 0; d < 3; ++d) o[d] = make_float2(f * (v[d].x - hh[d] * dr), f * (v[d].y - hh[d] * di));
                }
                if (!FORCES || with_noise) {
                    float wr[3], wi[3];
                    mode_noise<float>(m, M, w.Mh1, strm, seed, sample, wr, wi);
                    const float f = cn * sc;
                    const float dr = hx * wr[0] + hy * wr[1] + hz * wr[2];
                    const float di = hx * wi[0] + hy * wi[1] + hz * wi[2];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        o[d].x += f * (wr[d] - hh[d] * dr);
                        o[d].y += f * (wi[d] - hh[d] * di);
                    }
                }
            }
            at[0] = o[0];
            at[M * TQ] = o[1];
            at[2 * M * TQ] = o[2];
        }
    }
    __syncthreads();
    for (int c = 0; c < 3; ++c) {
        const float2 *in = fft_smem<1, TQ>(p, 0, p.nf - 1, line, on, jj, TJ, tw, A + c * M * TQ, B) + line;
        float2 *gc = g + (int64_t)c * M * plane;
        if (on)
            fft_pass_any<1>(p, p.nf - 1, jj, TJ, tw,
                            [&](int n) { return *reinterpret_cast<const float4 *>(in + n * TQ); },
                            [&](int n, float4 v) { *reinterpret_cast<float4 *>(gc + (int64_t)n * plane) = v; });
        __syncthreads();  // B is the next component's
    }
}

// y pass in place, blockIdx = (tile of kz, x, component + 3 species).
template <int S>
__global__ void __launch_bounds__(PSE_FFT_TY, 3) k_fft_y(const __grid_constant__ FftPlan p,
                                                         float2 *__restrict__ spec) {
    constexpr int TZ = PSE_FFT_TZ, TJ = 2 * PSE_FFT_TY / TZ;
    extern __shared__ __align__(16) float2 fsm[];
    const int M = p.M;
    float2 *A = fsm, *B = A + M * TZ, *tw = B + M * TZ;
    for (int k = threadIdx.x; k < M; k += PSE_FFT_TY) tw[k] = p.tw[k];
    const int line = 2 * (threadIdx.x % (TZ / 2)), jj = threadIdx.x / (TZ / 2), kz = blockIdx.x * TZ + line;
    const bool on = kz < p.KP;  // even KP: both lines have room
    float2 *g = spec + ((int64_t)blockIdx.z * M + blockIdx.y) * M * p.KP + kz;
    __syncthreads();
    float2 *a = A + line;
    if (on)
        fft_pass_any<S>(p, 0, jj, TJ, tw, [&](int n) { return *reinterpret_cast<const float4 *>(g + n * p.KP); },
                        [&](int n, float4 v) { *reinterpret_cast<float4 *>(a + n * TZ) = v; });
    __syncthreads();
    const float2 *in = fft_smem<S, TZ>(p, 1, p.nf - 1, line, on, jj, TJ, tw, A, B) + line;
    if (on)
        fft_pass_any<S>(p, p.nf - 1, jj, TJ, tw, [&](int n) { return *reinterpret_cast<const float4 *>(in + n * TZ); },
                        [&](int n, float4 v) { *reinterpret_cast<float4 *>(g + n * p.KP) = v; });
}

// Inverse z pass, blockIdx = (tile of y rows, x, species): spectrum rows -> node-major records.
template <int T>
__global__ void __launch_bounds__(T, 768 / T) k_fft_z_inv(const __grid_constant__ FftPlan p,
                                                          const float2 *__restrict__ spec,
                                                          V4<float> *__restrict__ grid4) {
    constexpr int TR = PSE_FFT_TR, NL = PSE_FFT_NL, LS = PSE_FFT_LS;
    extern __shared__ __align__(16) float2 fsm[];
    const int M = p.M, sp = blockIdx.z, H = M / 2, nkz = p.nkz;
    float2 *A = fsm, *B = A + M * LS, *tw = B + M * LS;
    for (int k = threadIdx.x; k < M; k += T) tw[k] = p.tw[k];
    const int y0 = blockIdx.x * TR, x = blockIdx.y;
    const float2 *src = spec + ((int64_t)sp * 3 * M + x) * M * p.KP;
    // line l = 3 pair + component holds rows y0 + 2 pair, + 1
    for (int l = threadIdx.x / 32; l < NL; l += T / 32) {
        const int pr = l / 3, c = l - 3 * pr, ya = y0 + 2 * pr;
        const float2 *ra = src + ((int64_t)c * M * M + ya) * p.KP;
        const bool oa = ya < M, ob = ya + 1 < M;
        float2 *d = A + l;
        for (int k0 = threadIdx.x & 31; k0 < nkz; k0 += 128) {  // four loads of each row in flight
            float2 a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 32 * u;
                a[u] = oa && k < nkz ? ra[k] : make_float2(0.f, 0.f);
                b[u] = ob && k < nkz ? ra[p.KP + k] : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 32 * u;
                if (k >= nkz) break;
                if (k == 0) {
                    d[0] = make_float2(a[u].x, b[u].x);  // the mean of a real row is real
                } else {
                    d[k * LS] = make_float2(a[u].x - b[u].y, a[u].y + b[u].x);
                    d[(M - k) * LS] = make_float2(a[u].x + b[u].y, b[u].x - a[u].y);
                }
            }
        }
        if ((M & 1) == 0 && (threadIdx.x & 31) == 0) d[H * LS] = make_float2(0.f, 0.f);  // Nyquist
    }
    __syncthreads();
    const int line = 2 * (threadIdx.x % (NL / 2)), jj = threadIdx.x / (NL / 2);
    const float2 *z = fft_smem<1, LS>(p, 0, p.nf, line, true, jj, 2 * T / NL, tw, A, B);
    V4<float> *out = grid4 + (((int64_t)sp * M + x) * M + y0) * M;
    // a warp writes 32 consecutive records of a pair's two rows
    const int chunks = (M + 31) >> 5;
    for (int t = threadIdx.x >> 5; t < TR / 2 * chunks; t += T / 32) {
        const int pr = t & (TR / 2 - 1), n = (t / (TR / 2)) * 32 + (threadIdx.x & 31), ya = y0 + 2 * pr;
        if (n >= M) continue;
        const float2 *e = z + n * LS + 3 * pr;
        const float2 v0 = e[0], v1 = e[1], v2 = e[2];
        V4<float> r;
        r.w = 0.f;
        if (ya < M) {
            r.x = v0.x; r.y = v1.x; r.z = v2.x;
            out[2 * pr * M + n] = r;
        }
        if (ya + 1 < M) {
            r.x = v0.y; r.y = v1.y; r.z = v2.y;
            out[(2 * pr + 1) * M + n] = r;
        }
    }
}

// Forward z pass: real grids, planar or (grid4) node-major, -> spectrum rows
// (kz < nkz).
template <int T>
__global__ void __launch_bounds__(T, 768 / T) k_fft_z_fwd(const __grid_constant__ FftPlan p, const float *__restrict__ grid,
                                                          const V4<float> *__restrict__ grid4, float2 *__restrict__ spec) {
    constexpr int TR = PSE_FFT_TR, NL = PSE_FFT_NL, LS = PSE_FFT_LS;
    extern __shared__ __align__(16) float2 fsm[];
    const int M = p.M;
    float2 *A = fsm, *B = A + M * LS, *tw = B + M * LS;
    for (int k = threadIdx.x; k < M; k += T) tw[k] = p.tw[k];
    const int y0 = blockIdx.x * TR, x = blockIdx.y;
    if (grid4) {
        // a warp reads 32 consecutive records of a pair's two rows
        const V4<float> *in = grid4 + ((int64_t)x * M + y0) * M;
        const int chunks = (M + 31) >> 5;
        for (int t = threadIdx.x >> 5; t < TR / 2 * chunks; t += T / 32) {
            const int pr = t & (TR / 2 - 1), n = (t / (TR / 2)) * 32 + (threadIdx.x & 31), ya = y0 + 2 * pr;
            if (n >= M) continue;
            V4<float> a{}, b{};
            if (ya < M) a = in[2 * pr * M + n];
            if (ya + 1 < M) b = in[(2 * pr + 1) * M + n];
            float2 *e = A + n * LS + 3 * pr;
            e[0] = make_float2(a.x, b.x);
            e[1] = make_float2(a.y, b.y);
            e[2] = make_float2(a.z, b.z);
        }
    }
    for (int l = grid4 ? NL : threadIdx.x / 32; l < NL; l += T / 32) {
        const int pr = l / 3, c = l - 3 * pr, ya = y0 + 2 * pr;
        const float *ra = grid + (((int64_t)c * M + x) * M + ya) * M;
        const bool oa = ya < M, ob = ya + 1 < M;
        for (int n = threadIdx.x & 31; n < M; n += 32)
            A[n * LS + l] = make_float2(oa ? ra[n] : 0.f, ob ? ra[M + n] : 0.f);
    }
    __syncthreads();
    const int line = 2 * (threadIdx.x % (NL / 2)), jj = threadIdx.x / (NL / 2);
    const float2 *z = fft_smem<-1, LS>(p, 0, p.nf, line, true, jj, 2 * T / NL, tw, A, B);
    for (int l = threadIdx.x / 32; l < NL; l += T / 32) {
        const int pr = l / 3, c = l - 3 * pr, ya = y0 + 2 * pr;
        float2 *ra = spec + (((int64_t)c * M + x) * M + ya) * p.KP;
        for (int k = threadIdx.x & 31; k < p.nkz; k += 32) {
            const float2 a = z[k * LS + l], b = z[(k ? M - k : 0) * LS + l];
            // Ya = (Z_k + conj Z_{M-k}) / 2, Yb = (Z_k - conj Z_{M-k}) / 2i
            if (ya < M) ra[k] = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
            if (ya + 1 < M) ra[p.KP + k] = make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
        }
    }
}

static size_t fft_smem_x(int M) { return sizeof(float2) * M * (1 + 4 * PSE_FFT_TQ); }
static size_t fft_smem_y(int M) { return sizeof(float2) * M * (1 + 2 * PSE_FFT_TZ); }
static size_t fft_smem_z(int M) { return sizeof(float2) * M * (1 + 2 * PSE_FFT_LS); }

// ------------------------------------------------------------------ samples on 256^3 by radix-16 register passes
// Grids of M = R^2 points (R = 16: M = 256, with wave_fft = 1): the same three
// passes over x, y and z, each line transformed by R threads in two register
// passes (the four-step split n = t + R m, k = k1 + R k2):
//   A_t[k1] = w_M^{t k1} sum_m x[t + R m] w_R^{m k1},
//   X[k1 + R k2] = sum_t A_t[k1] w_R^{t k2},  w_L = e^{2 pi i / L},
// with one padded shared-memory transpose between them.  Noise, x, y and z 385
// us alone, the general passes (8, 8, 4 through shared memory) 404; sample of
// 1e6 1228 against 1256 us.  Spectrum rows of M / 2 + 1 modes.
constexpr int PSE_FFTR_TZ = 8;   // kz values per block in the x and y passes
constexpr int PSE_FFTR_TY = 8;   // iy rows per block in the z pass

template <int R> __device__ __forceinline__ constexpr int bitrev_c(int v) {
    int r = 0;
    for (int b = 1; b < R; b <<= 1) {
        r = (r << 1) | (v & 1);
        v >>= 1;
    }
    return r;
}
// In-register radix-2 DIT of R points: v in bit-reversed order, output in
// natural order, w[k] = w_R^k for k < R/2.
template <int R> __device__ __forceinline__ void fft_reg(float2 (&v)[R], const float2 (&w)[R / 2]) {
#pragma unroll
    for (int half = 1; half < R; half <<= 1) {
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            const int pos = j & (half - 1);
            const int i0 = ((j - pos) << 1) + pos, i1 = i0 + half;
            const float2 t = cmulf(w[pos * (R / (2 * half))], v[i1]);
            const float2 a = v[i0];
            v[i0] = make_float2(a.x + t.x, a.y + t.y);
            v[i1] = make_float2(a.x - t.x, a.y - t.y);
        }
    }
}

// w_M^j for any j >= 0 from the half-circle table tw[k] = w_M^k, k < M/2.
template <int M> __device__ __forceinline__ float2 tw_full(const float2 *tw, int j) {
    j &= M - 1;
    const float2 e = tw[j & (M / 2 - 1)];
    return j < M / 2 ? e : make_float2(-e.x, -e.y);
}

// One line of M = R^2 points, natural order in `line` (stride 1, R (R + 1)
// entries of room), transformed by the R threads t = 0..R-1 of a group;
// returns X[t + R k2] in out[k2].  The group's threads must lie in one warp.
template <int R>
__device__ __forceinline__ void fft_line_sq(float2 *line, int t, const float2 *tw, const float2 (&wR)[R / 2],
                                            float2 (&out)[R]) {
    constexpr int M = R * R;
    float2 v[R];
#pragma unroll
    for (int m = 0; m < R; ++m) v[m] = line[t + R * bitrev_c<R>(m)];
    fft_reg<R>(v, wR);
#pragma unroll
    for (int k1 = 1; k1 < R; ++k1) v[k1] = cmulf(v[k1], tw_full<M>(tw, t * k1));
    __syncwarp();
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) line[k1 * (R + 1) + t] = v[k1];
    __syncwarp();
#pragma unroll
    for (int m = 0; m < R; ++m) out[m] = line[t * (R + 1) + bitrev_c<R>(m)];
    fft_reg<R>(out, wR);
    __syncwarp();
}

// Shared-memory line stride: room for the R (R + 1) transpose, padded to
// 4 mod 16 float2 so that the TZ lines touched by one row of a tile load or
// store start on different banks.
template <int R> constexpr int fft_lsz() { return R * (R + 1) + ((4 - R * (R + 1)) % 16 + 16) % 16; }

template <int R> __device__ __forceinline__ void load_wR(const float2 *tw, float2 (&wR)[R / 2]) {
#pragma unroll
    for (int k = 0; k < R / 2; ++k) wR[k] = tw[k * R];  // w_R^k = w_M^{k R}
}

// pass x: block = (tile of TZ kz values, ky); threads: 3 TZ lines x R.
template <int R>
__global__ void __launch_bounds__(3 * PSE_FFTR_TZ * R, 3) k_fftx_noise(WaveGeom<float> w, const SampleArgs<float> *args,
                                                                   int system, const float2 *__restrict__ tw_g,
                                                                   float2 *spec) {
    constexpr int M = R * R, TZ = PSE_FFTR_TZ, LSZ = fft_lsz<R>(), Mh1 = M / 2 + 1;
    extern __shared__ float2 sm[];
    float2 *tw = sm;           // M/2
    float2 *buf = sm + M / 2;  // [3 TZ lines][LSZ], line = c * TZ + kzl
    for (int k = threadIdx.x; k < M / 2; k += blockDim.x) tw[k] = tw_g[k];
    const int kz0 = blockIdx.x * TZ, ky = blockIdx.y;
    const uint32_t strm = 2u * system + 1u;
    const uint64_t seed = args->seed, sample = args->sample;
    for (int i = threadIdx.x; i < M * TZ; i += blockDim.x) {
        const int kzl = i % TZ, kx = i / TZ;
        ModeIdx m;
        m.ix = kx; m.iy = ky; m.iz = kz0 + kzl;
        m.nx = kx <= M / 2 ? kx : kx - M;
        m.ny = ky <= M / 2 ? ky : ky - M;
        m.nz = m.iz;
        m.live = kx != M / 2 && ky != M / 2 && (m.nx | m.ny | m.nz) != 0;
        float2 o0 = make_float2(0.f, 0.f), o1 = o0, o2 = o0;
        if (m.live) {
            float wr[3], wi[3];
            mode_noise<float>(m, M, Mh1, strm, seed, sample, wr, wi);
            float hx, hy, hz;
            const float sc = mode_scale<float>(m, w, hx, hy, hz);
            const float dr = hx * wr[0] + hy * wr[1] + hz * wr[2];
            const float di = hx * wi[0] + hy * wi[1] + hz * wi[2];
            o0 = make_float2(sc * (wr[0] - hx * dr), sc * (wi[0] - hx * di));
            o1 = make_float2(sc * (wr[1] - hy * dr), sc * (wi[1] - hy * di));
            o2 = make_float2(sc * (wr[2] - hz * dr), sc * (wi[2] - hz * di));
        }
        buf[(0 * TZ + kzl) * LSZ + kx] = o0;
        buf[(1 * TZ + kzl) * LSZ + kx] = o1;
        buf[(2 * TZ + kzl) * LSZ + kx] = o2;
    }
    __syncthreads();
    float2 wR[R / 2];
    load_wR<R>(tw, wR);
    const int line = threadIdx.x / R, t = threadIdx.x % R;
    float2 out[R];
    fft_line_sq<R>(buf + line * LSZ, t, tw, wR, out);
#pragma unroll
    for (int k2 = 0; k2 < R; ++k2) buf[line * LSZ + t + R * k2] = out[k2];
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * M * TZ; i += blockDim.x) {
        const int kzl = i % TZ, rest = i / TZ, ix = rest % M, c = rest / M;
        spec[(((int64_t)c * M + ix) * M + ky) * Mh1 + kz0 + kzl] = buf[(c * TZ + kzl) * LSZ + ix];
    }
}

// pass y: block = (tile of TZ kz values, ix); in place.
template <int R>
__global__ void __launch_bounds__(3 * PSE_FFTR_TZ * R, 3) k_ffty(const float2 *__restrict__ tw_g, float2 *spec) {
    constexpr int M = R * R, TZ = PSE_FFTR_TZ, LSZ = fft_lsz<R>(), Mh1 = M / 2 + 1;
    extern __shared__ float2 sm[];
    float2 *tw = sm;
    float2 *buf = sm + M / 2;
    for (int k = threadIdx.x; k < M / 2; k += blockDim.x) tw[k] = tw_g[k];
    const int kz0 = blockIdx.x * TZ, ix = blockIdx.y;
    for (int i = threadIdx.x; i < 3 * M * TZ; i += blockDim.x) {
        const int kzl = i % TZ, rest = i / TZ, ky = rest % M, c = rest / M;
        buf[(c * TZ + kzl) * LSZ + ky] = spec[(((int64_t)c * M + ix) * M + ky) * Mh1 + kz0 + kzl];
    }
    __syncthreads();
    float2 wR[R / 2];
    load_wR<R>(tw, wR);
    const int line = threadIdx.x / R, t = threadIdx.x % R;
    float2 out[R];
    fft_line_sq<R>(buf + line * LSZ, t, tw, wR, out);
#pragma unroll
    for (int k2 = 0; k2 < R; ++k2) buf[line * LSZ + t + R * k2] = out[k2];
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * M * TZ; i += blockDim.x) {
        const int kzl = i % TZ, rest = i / TZ, ky = rest % M, c = rest / M;
        spec[(((int64_t)c * M + ix) * M + ky) * Mh1 + kz0 + kzl] = buf[(c * TZ + kzl) * LSZ + ky];
    }
}

// pass z: block = (tile of TY iy rows, ix); the 3 TY real rows (c, iyl) are
// transformed in pairs (c, iyl) + i (c, iyl + TY/2).
template <int R>
__global__ void __launch_bounds__(3 * PSE_FFTR_TY / 2 * R) k_fftz_c2r(const float2 *__restrict__ tw_g,
                                                                   const float2 *__restrict__ spec, V4<float> *grid4) {
    constexpr int M = R * R, H = M / 2, TY = PSE_FFTR_TY, LSZ = fft_lsz<R>(), Mh1 = M / 2 + 1, NP = 3 * TY / 2;
    extern __shared__ float2 sm[];
    float2 *tw = sm;                      // M/2
    float2 *raw = tw + M / 2;             // [3][TY][H]
    float2 *buf = raw + 3 * TY * H;       // [NP][LSZ]
    float *xo = reinterpret_cast<float *>(raw);  // [3][TY][M], over raw once Z is built
    for (int k = threadIdx.x; k < M / 2; k += blockDim.x) tw[k] = tw_g[k];
    const int iy0 = blockIdx.x * TY, ix = blockIdx.y;
    for (int i = threadIdx.x; i < 3 * TY * H; i += blockDim.x) {
        const int k = i % H, rest = i / H, iyl = rest % TY, c = rest / TY;
        raw[i] = spec[(((int64_t)c * M + ix) * M + iy0 + iyl) * Mh1 + k];
    }
    __syncthreads();
    // pair p = c * (TY/2) + j holds rows (c, j) and (c, j + TY/2)
    for (int i = threadIdx.x; i < NP * M; i += blockDim.x) {
        const int k = i % M, p = i / M, c = p / (TY / 2), j = p % (TY / 2);
        const float2 *ra = raw + (c * TY + j) * H, *rb = raw + (c * TY + j + TY / 2) * H;
        float2 ya, yb;
        if (k < H) {
            ya = ra[k];
            yb = rb[k];
        } else if (k == H) {
            ya = yb = make_float2(0.f, 0.f);
        } else {
            const float2 a = ra[M - k], b = rb[M - k];
            ya = make_float2(a.x, -a.y);
            yb = make_float2(b.x, -b.y);
        }
        buf[p * LSZ + k] = make_float2(ya.x - yb.y, ya.y + yb.x);  // Ya + i Yb
    }
    __syncthreads();
    float2 wR[R / 2];
    load_wR<R>(tw, wR);
    const int p = threadIdx.x / R, t = threadIdx.x % R;
    float2 out[R];
    fft_line_sq<R>(buf + p * LSZ, t, tw, wR, out);
    {
        const int c = p / (TY / 2), j = p % (TY / 2);
        float *xa = xo + (c * TY + j) * M, *xb = xo + (c * TY + j + TY / 2) * M;
#pragma unroll
        for (int k2 = 0; k2 < R; ++k2) {
            xa[t + R * k2] = out[k2].x;
            xb[t + R * k2] = out[k2].y;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TY * M; i += blockDim.x) {
        const int iz = i % M, iyl = i / M;
        V4<float> v;
        v.x = xo[(0 * TY + iyl) * M + iz];
        v.y = xo[(1 * TY + iyl) * M + iz];
        v.z = xo[(2 * TY + iyl) * M + iz];
        v.w = 0.f;
        grid4[((int64_t)ix * M + iy0 + iyl) * M + iz] = v;
    }
}

template <int R> static size_t fftr_smem_xy() {
    return sizeof(float2) * (R * R / 2 + 3 * PSE_FFTR_TZ * fft_lsz<R>());
}
template <int R> static size_t fftr_smem_z() {
    constexpr int M = R * R;  // raw (3 TY rows of M/2 float2) is reused for the 3 TY rows of M real outputs
    return sizeof(float2) * (M / 2 + 3 * PSE_FFTR_TY * (M / 2) + 3 * PSE_FFTR_TY / 2 * fft_lsz<R>());
}
template <int R> static void fftr_sample(const FftPlan &p, const FftJob &job, int parts, cudaStream_t s) {
    constexpr int M = R * R;
    const dim3 gxy(M / 2 / PSE_FFTR_TZ, M), gz(M / PSE_FFTR_TY, M);
    if (parts & 1)
        k_fftx_noise<R><<<gxy, 3 * PSE_FFTR_TZ * R, fftr_smem_xy<R>(), s>>>(job.w, job.args, job.system, p.tw, job.spec);
    if (parts & 2) k_ffty<R><<<gxy, 3 * PSE_FFTR_TZ * R, fftr_smem_xy<R>(), s>>>(p.tw, job.spec);
    if (parts & 4) k_fftz_c2r<R><<<gz, 3 * PSE_FFTR_TY / 2 * R, fftr_smem_z<R>(), s>>>(p.tw, job.spec, job.grid4);
}
template <int R> static cudaError_t fftr_attrs() {
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_fftx_noise<R>, attr, (int)fftr_smem_xy<R>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ffty<R>, attr, (int)fftr_smem_xy<R>());
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fftz_c2r<R>, attr, (int)fftr_smem_z<R>());
    return e;
}

// Factors of M (2..4 of them, as few as possible, then the smallest largest
// one) among the radices above; false where there are none.
bool fft_plan(int M, FftPlan *p) {
    static const int R[] = {9, 8, 7, 6, 5, 4, 3, 2};
    if (M < 16 || M > PSE_FFT_MAXM) return false;
    int best[4] = {}, nbest = 5, bmax = 99, cur[4] = {};
    auto rec = [&](auto &&self, int m, int n, int i0) -> void {
        if (m == 1) {
            if (n < 2) return;
            if (n < nbest || (n == nbest && cur[0] < bmax)) {
                nbest = n;
                bmax = cur[0];
                for (int i = 0; i < n; ++i) best[i] = cur[i];
            }
            return;
        }
        if (n == 4) return;
        for (int i = i0; i < (int)(sizeof(R) / sizeof(R[0])); ++i)
            if (m % R[i] == 0) {
                cur[n] = R[i];
                self(self, m / R[i], n + 1, i);
            }
    };
    rec(rec, M, 0, 0);
    if (nbest > 4) return false;
    p->M = M;
    p->nkz = (M + 1) / 2;
    p->KP = (p->nkz + 3) & ~3;
    p->nf = nbest;
    int ns = 1;
    for (int i = 0; i < nbest; ++i) {
        p->rad[i] = best[i];
        p->ns[i] = ns;
        p->mg[i] = ns > 1 ? (uint32_t)((0x100000000ull + ns - 1) / ns) : 0u;  // j / ns for j < 2^16
        ns *= best[i];
    }
    return true;
}

// Shared memory of the passes for every grid size; once per device, outside
// any capture.
cudaError_t fft_prepare() {
    const int zx = (int)fft_smem_x(PSE_FFT_MAXM), zy = (int)fft_smem_y(PSE_FFT_MAXM), zz = (int)fft_smem_z(PSE_FFT_MAXM);
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_fft_x<false>, attr, zx);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_x<true>, attr, zx);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_y<1>, attr, zy);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_y<-1>, attr, zy);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_z_inv<PSE_FFT_TT_MANY>, attr, zz);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_z_inv<PSE_FFT_TT_FEW>, attr, zz);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_z_fwd<PSE_FFT_TT_MANY>, attr, zz);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_z_fwd<PSE_FFT_TT_FEW>, attr, zz);
    return e == cudaSuccess ? fftr_attrs<16>() : e;
}

// Where these transforms are faster than cuFFT's: a whole call both ways, in
// turn, on every grid size without prime factors above 7 from 96 to 500 and at
// M^3 / N = 57, 17, 8.5 and 4.2 (lattices of spheres, xi a = 0.52), cuFFT over
// ours, so above 1 where ours win.
// Sizes: from M = 126 on for sizes with a factor 5 or 7 (samples at 17, forces
// at 17: M = 120 1.00, 1.01; 125 1.00, 0.95; 126 0.97, 1.14; 135 1.00, 1.16;
// 147 1.15, 1.30; 200 1.14, 1.15; 245 1.27, 1.35); from 162 on without, since
// cuFFT is at its best on small products of 2 and 3 (96 0.98, 1.01; 108 0.92,
// 0.99; 128 1.00, 0.97; 144 0.96, 0.95; 162 1.12, 1.19; 192 1.04, 1.05); not
// powers of two (256 0.96, 1.00); up to 486 (480 1.02, 1.04; 486 1.20, 1.26;
// 490 0.97, 0.97; 500 0.93, 0.92: an empirical line).
static bool fft_sizes(int M) {
    int m = M;
    while (m % 2 == 0) m /= 2;
    const bool pow2 = m == 1;
    while (m % 3 == 0) m /= 3;
    return M >= (m == 1 ? 162 : 126) && M < 490 && !pow2;
}
// Forces: at every density (at 4.2: M = 147 1.04, 189 1.04, 243 1.01, 245 1.07,
// 288 1.03, 294 1.08, 343 1.01; their transforms are the longer branch).
bool fft_wins_forces(int M) { return fft_sizes(M); }
// Samples: in dense systems the near field is the longer branch, and while
// blocks of our passes are resident its one-wave kernels wait for them longer
// than for cuFFT's shorter blocks.  Below M = 200 that is within the spread of
// sizes at any density (at 4.2: 162 1.02, 168 0.98, 189 1.03, 196 1.00); above,
// ours lose at 4.2 (216 0.98, 225 0.96, 240 0.98, 243 0.96, 250 0.96, 288
// 0.92) and, on products of 2 and 3, at 8.5 (216 0.96, 243 0.96, 288 0.93, 324
// 0.99; other sizes 210 1.06, 225 1.00, 245 1.09, 250 0.98, 270 0.96, 294
// 1.14, 336 1.04); at 17 they win up to 375 (243 1.01, 252 1.09, 294 1.34, 324
// 1.05, 375 1.21) and are even above (378 0.99, 384 1.02, 405 1.16, 420 0.99),
// at 34 everywhere (378 1.09, 420 1.11, 480 1.04).
bool fft_wins_sample(int M, int nspec, int64_t N) {
    if (!fft_sizes(M)) return false;
    int m = M;
    while (m % 2 == 0) m /= 2;
    while (m % 3 == 0) m /= 3;
    const double per = (double)M * M * M * nspec / N, most = m == 1 ? 12.0 : 6.0;
    return M <= 200 || per >= (M > 375 ? 30.0 : (M > 245 && most < 10.0 ? 10.0 : most));
}

template <int S> static void fft_y(const FftPlan &p, const FftJob &job, int nspec, cudaStream_t s) {
    const dim3 grid((p.nkz + PSE_FFT_TZ - 1) / PSE_FFT_TZ, p.M, 3 * nspec);
    k_fft_y<S><<<grid, PSE_FFT_TY, fft_smem_y(p.M), s>>>(p, job.spec);
}
static void fft_z_inv(const FftPlan &p, const FftJob &job, int nspec, cudaStream_t s) {
    const dim3 grid((p.M + PSE_FFT_TR - 1) / PSE_FFT_TR, p.M, nspec);
    if (p.M <= PSE_FFT_FEW_MAXM)
        k_fft_z_inv<PSE_FFT_TT_FEW><<<grid, PSE_FFT_TT_FEW, fft_smem_z(p.M), s>>>(p, job.spec, job.grid4);
    else
        k_fft_z_inv<PSE_FFT_TT_MANY><<<grid, PSE_FFT_TT_MANY, fft_smem_z(p.M), s>>>(p, job.spec, job.grid4);
}
// parts: bit 0 the x pass (with the noise), bit 1 the y pass, bit 2 the z pass
void launch_fft_sample(const FftPlan &p, const FftJob &job, int parts, cudaStream_t s) {
    if (p.M == 16 * 16) {  // (one species: wave_fft = 1)
        fftr_sample<16>(p, job, parts, s);
        return;
    }
    const int nspec = job.w.nspec > 1 ? job.w.nspec : 1;
    const dim3 gx((p.M * p.KP + PSE_FFT_TQ - 1) / PSE_FFT_TQ, nspec);
    if (parts & 1) k_fft_x<false><<<gx, PSE_FFT_TX, fft_smem_x(p.M), s>>>(p, job, 0);
    if (parts & 2) fft_y<1>(p, job, nspec, s);
    if (parts & 4) fft_z_inv(p, job, nspec, s);
}
// The wave product of the spread grid (planar, or with grid null the node-major
// one): forward transform, mode factor (and noise), inverse transform into the
// node-major grid.
void launch_fft_forces(const FftPlan &p, const FftJob &job, const float *grid, int with_noise, cudaStream_t s) {
    const dim3 gz((p.M + PSE_FFT_TR - 1) / PSE_FFT_TR, p.M);
    const V4<float> *grid4 = grid ? nullptr : job.grid4;
    if (p.M <= PSE_FFT_FEW_MAXM)
        k_fft_z_fwd<PSE_FFT_TT_FEW><<<gz, PSE_FFT_TT_FEW, fft_smem_z(p.M), s>>>(p, grid, grid4, job.spec);
    else
        k_fft_z_fwd<PSE_FFT_TT_MANY><<<gz, PSE_FFT_TT_MANY, fft_smem_z(p.M), s>>>(p, grid, grid4, job.spec);
    fft_y<-1>(p, job, 1, s);
    const dim3 gx((p.M * p.KP + PSE_FFT_TQ - 1) / PSE_FFT_TQ);
    k_fft_x<true><<<gx, PSE_FFT_TX, fft_smem_x(p.M), s>>>(p, job, with_noise);
    fft_y<1>(p, job, 1, s);
    fft_z_inv(p, job, 1, s);
}

#define PSE_INST(T)                                                                                      \
    template void launch_wave_noise<T>(WaveGeom<T>, const SampleArgs<T> *, int, void *, cudaStream_t); \
    template void launch_interp<T>(int64_t, WaveGeom<T>, Geom<T>, const Dev<T> &, cudaStream_t);       \
    template void launch_grid_copy<T>(WaveGeom<T>, const Dev<T> &, cudaStream_t);                        \
    template void launch_wave_apply<T>(WaveGeom<T>, const SampleArgs<T> *, int, void *, int, int, cudaStream_t); \
    template void launch_grid_noise<T>(WaveGeom<T>, const SampleArgs<T> *, int, T *, cudaStream_t);   \
    template cudaError_t launch_spread<T>(WaveGeom<T>, Geom<T>, SpreadTile, const int *, const int2 *, const int *, \
                                          T *, const Dev<T> &, cudaStream_t, const Rec<T> *);                                      \
    template cudaError_t spread_prepare<T>(size_t *);
PSE_INST(float)
PSE_INST(double)
#undef PSE_INST

}  // namespace pse
