// bd_state.cu -- set-up, refresh and read-out kernels of libbdecon.
//
//   a1  set-up (double): normalised PSF (Eq. 1-2), per-pixel photon-unit
//       constants of Eq. 4-6, Dirichlet hyperparameters |OTF| / sum |OTF| of
//       Eq. 8 per patch shape, twiddle tables, initial object.
//   a8  refresh (double): mu = K (x) rho by direct summation, patch spectra
//       by direct DFT, and the full log posterior of Eq. 9; it replaces the
//       incrementally updated mu and spectra (drift correction) and rebases
//       the trace.
// Every reduction uses a fixed block size and a fixed tree, so results do
// not depend on the launch plan of the sweep kernel.
#include <cmath>


#include "bd_device.cuh"

namespace bd {

// deterministic block sum (kRedThreads threads)
__device__ __forceinline__ double block_sum(double v, double* sh)
{
    const int tid = threadIdx.x;
    sh[tid] = v;
    __syncthreads();
    for (int o = kRedThreads / 2; o > 0; o >>= 1) {
        if (tid < o) sh[tid] += sh[tid + o];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// ------------------------------------------------------------------ a1 ---
__global__ void __launch_bounds__(kRedThreads) k_setup_psf(int L, const double* psf, double* K64, float* K32)
{
    __shared__ double sh[kRedThreads];
    double s = 0.0;
    for (int k = threadIdx.x; k < L * L; k += kRedThreads) s += psf[k];
    const double tot = block_sum(s, sh);
    for (int k = threadIdx.x; k < L * L; k += kRedThreads) {
        const double v = psf[k] / tot;
        K64[k] = v;
        K32[k] = (float)v;
    }
}

// Effective kernel of a lattice f times finer than the camera: a camera
// pixel sums the f x f cells of its area (the pixel integral of Eq. 1), so
// Ke[p][q] = sum_{u,v < f} K[p-u][q-v], side Le = L + f - 1.
__global__ void k_setup_eff(int L, int f, const double* K64, double* Ke64, float* Ke32)
{
    const int Le = L + f - 1;
    for (int idx = threadIdx.x; idx < Le * Le; idx += blockDim.x) {
        const int p = idx / Le, q = idx % Le;
        double s = 0.0;
        for (int u = 0; u < f; ++u)
            for (int v = 0; v < f; ++v) {
                const int pp = p - u, qq = q - v;
                if (pp >= 0 && pp < L && qq >= 0 && qq < L) s += K64[pp * L + qq];
            }
        Ke64[idx] = s;
        Ke32[idx] = (float)s;
    }
}

// c = (w - o)/G, s^2 = var/G^2 (photon units), 1/s^2, exp(-1/s^2), -log(2 pi var)/2
__global__ void __launch_bounds__(kRedThreads) k_setup_data(int n, const float* w, const float* g, const float* o,
                                                           const float* v, double gs, double os, double vs,
                                                           double* dat64, float* dat32, double* part_c)
{
    __shared__ double sh[kRedThreads];
    const int idx = blockIdx.x * kRedThreads + threadIdx.x;
    double c = 0.0;
    if (idx < n) {
        const double G = g ? (double)g[idx] : gs;
        const double off = o ? (double)o[idx] : os;
        const double var = v ? (double)v[idx] : vs;
        c = ((double)w[idx] - off) / G;
        const double is2 = G * G / var;
        const double beta = exp(-is2);
        const double lnorm = -0.5 * log(2.0 * CUDART_PI * var);
        dat64[4 * (size_t)idx + 0] = c;
        dat64[4 * (size_t)idx + 1] = is2;
        dat64[4 * (size_t)idx + 2] = beta;
        dat64[4 * (size_t)idx + 3] = lnorm;
        dat32[4 * (size_t)idx + 0] = (float)c;
        dat32[4 * (size_t)idx + 1] = (float)is2;
        dat32[4 * (size_t)idx + 2] = (float)beta;
        dat32[4 * (size_t)idx + 3] = (float)lnorm;
    }
    const double s = block_sum(c, sh);
    if (threadIdx.x == 0) part_c[blockIdx.x] = s;
}

// b0 = max(0.1, mean_n c_n)
__global__ void __launch_bounds__(kRedThreads) k_setup_b0(const double* part_c, int nblk, int npix, int f, double* b0)
{
    __shared__ double sh[kRedThreads];
    double s = 0.0;
    for (int k = threadIdx.x; k < nblk; k += kRedThreads) s += part_c[k];
    const double tot = block_sum(s, sh);
    if (threadIdx.x == 0) {
        const double m = tot / (double)npix;
        b0[0] = (m > 0.1 ? m : 0.1) / (double)(f * f);   // a camera pixel collects f^2 cells
    }
}

// exp(-2 pi i j / n) for j < n
__global__ void k_setup_tw(int n, double* tw64, float* tw32)
{
    for (int j = threadIdx.x + blockIdx.x * blockDim.x; j < n; j += blockDim.x * gridDim.x) {
        double s, c;
        sincospi(2.0 * (double)j / (double)n, &s, &c);
        tw64[2 * j] = c;
        tw64[2 * j + 1] = -s;
        tw32[2 * j] = (float)c;
        tw32[2 * j + 1] = (float)-s;
    }
}

// Eq. 8 hyperparameter for one patch shape: alpha = |DFT(PSF wrapped onto the
// ph x pw torus, centre at the origin)| / sum, then the weights of the
// canonical half-spectrum entries: mult * (alpha - 1) / 2 and mult.
//
// One block: the wrapped kernel gathered per torus pixel, its transform taken
// by rows and then columns in shared memory (ph pw (ph + pw) products; the
// direct sum and a one-thread wrap took 646 us at 25 x 25, four shapes a problem).
__global__ void __launch_bounds__(kRedThreads) k_setup_alpha(int L, const double* K64, int ph, int pw,
                                                            const int* ent_kl, int nhalf, double* mag, double* wa64,
                                                            double* m64, float* wa32, float* m32, const double2* twh,
                                                            const double2* tww)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ double sh[kRedThreads];
    const int R = L / 2, n = ph * pw;
    double2* Y = reinterpret_cast<double2*>(dyn);           // [ph][pw]
    double* x = reinterpret_cast<double*>(Y + n);           // [ph][pw]
    for (int e = threadIdx.x; e < n; e += kRedThreads) {
        // kernel rows p with (p - R) mod ph = u, columns alike
        const int u = e / pw, v = e - u * pw;
        double k = 0.0;
        for (int p = (u + R) % ph; p < L; p += ph)
            for (int q = (v + R) % pw; q < L; q += pw) k += K64[p * L + q];
        x[e] = k;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += kRedThreads) {
        const int u = e / pw, l = e - u * pw;
        double re = 0.0, im = 0.0;
        for (int v = 0, j = 0; v < pw; ++v) {
            const double2 w = tww[j];
            re += x[u * pw + v] * w.x;
            im += x[u * pw + v] * w.y;
            j += l;
            j -= j >= pw ? pw : 0;
        }
        Y[e] = make_double2(re, im);
    }
    __syncthreads();
    double part = 0.0;
    for (int e = threadIdx.x; e < n; e += kRedThreads) {
        const int k = e / pw, l = e - k * pw;
        double re = 0.0, im = 0.0;
        for (int u = 0, j = 0; u < ph; ++u) {
            const double2 w = twh[j], y = Y[u * pw + l];
            re += y.x * w.x - y.y * w.y;
            im += y.x * w.y + y.y * w.x;
            j += k;
            j -= j >= ph ? ph : 0;
        }
        mag[e] = hypot(re, im);
        part += mag[e];
    }
    // the sum over all frequencies, in a fixed order
    __syncthreads();
    const double tot = block_sum(part, sh);
    for (int e = threadIdx.x; e < nhalf; e += kRedThreads) {
        const int kl = ent_kl[e];
        const int k = kl >> 16, l = kl & 0xffff;
        const bool self = ((ph - k) % ph == k) && ((pw - l) % pw == l);
        const double mult = self ? 1.0 : 2.0;
        const double a = mag[k * pw + l] / tot;
        wa64[e] = 0.5 * mult * (a - 1.0);
        m64[e] = mult;
        wa32[e] = (float)wa64[e];
        m32[e] = (float)mult;
    }
}

// Initial object rho0_m = b0 exp(z_m / 10), z_m the Box-Muller normal of the
// Philox counter (m, 0, chain, 0): sweep index 0 is never a sampling sweep.
template <typename T>
__global__ void k_init_rho(int n, uint32_t seed_lo, uint32_t seed_hi, int chain, const double* b0, T* rho)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n) return;
    const uint4 x = philox4x32_10(make_uint4((uint32_t)m, 0u, (uint32_t)chain, 0u), seed_lo, seed_hi);
    const double z = sqrt(-2.0 * log(uniform23<double>(x.x))) * cos(2.0 * CUDART_PI * uniform23<double>(x.y));
    rho[m] = (T)(b0[0] * exp(0.1 * z));
}

cudaError_t launch_setup(const Image& im, const Image* d_im, const float* w, const float* g, const float* o,
                  const float* v, double gs, double os, double vs, const double* psf_raw, double* b0_out,
                  double* scratch, cudaStream_t st, int64_t* launches)
{
    (void)d_im;
    k_setup_psf<<<1, kRedThreads, 0, st>>>(im.L, psf_raw, const_cast<double*>(im.K64), const_cast<float*>(im.K32));
    if (im.f > 1) {
        k_setup_eff<<<1, 256, 0, st>>>(im.L, im.f, im.K64, const_cast<double*>(im.Ke64), const_cast<float*>(im.Ke32));
        ++*launches;
    }
    const int npix = im.H * im.W;
    const int nblk = (npix + kRedThreads - 1) / kRedThreads;
    double* part_c = scratch;                       // nblk
    k_setup_data<<<nblk, kRedThreads, 0, st>>>(npix, w, g, o, v, gs, os, vs, const_cast<double*>(im.dat64),
                                               const_cast<float*>(im.dat32), part_c);
    k_setup_b0<<<1, kRedThreads, 0, st>>>(part_c, nblk, npix, im.f, b0_out);
    *launches += 3;
    // twiddles: the distinct patch sides appear at the shapes' offsets
    for (int s = 0; s < kMaxShapes; ++s) {
        const Shape& sh = im.shape[s];
        if (sh.nhalf == 0) continue;
        k_setup_tw<<<1, 128, 0, st>>>(sh.ph, const_cast<double*>(im.tw64) + 2 * sh.twh_off,
                                      const_cast<float*>(im.tw32) + 2 * sh.twh_off);
        k_setup_tw<<<1, 128, 0, st>>>(sh.pw, const_cast<double*>(im.tw64) + 2 * sh.tww_off,
                                      const_cast<float*>(im.tw32) + 2 * sh.tww_off);
        double* mag = scratch + nblk + 8;
        const size_t sm = 24 * (size_t)sh.ph * sh.pw;
        const cudaError_t e = raise_smem_limit((const void*)k_setup_alpha, sm);
        if (e != cudaSuccess) return e;
        k_setup_alpha<<<1, kRedThreads, sm, st>>>(im.L, im.K64, sh.ph, sh.pw, im.ent_kl + sh.ent_off, sh.nhalf, mag,
                                                 const_cast<double*>(im.ent_wa64) + sh.ent_off,
                                                 const_cast<double*>(im.ent_m64) + sh.ent_off,
                                                 const_cast<float*>(im.ent_wa32) + sh.ent_off,
                                                 const_cast<float*>(im.ent_m32) + sh.ent_off,
                                                 reinterpret_cast<const double2*>(im.tw64) + sh.twh_off,
                                                 reinterpret_cast<const double2*>(im.tw64) + sh.tww_off);
        *launches += 3;
    }
    return cudaGetLastError();
}

template <typename T>
void launch_init_rho(const Image& im, const Chain& ch, const double* b0, cudaStream_t st, int64_t* launches)
{
    const int n = im.Ho * im.Wo;
    k_init_rho<T><<<(n + 255) / 256, 256, 0, st>>>(n, im.seed_lo, im.seed_hi, ch.chain, b0, reinterpret_cast<T*>(ch.rho));
    ++*launches;
}
template void launch_init_rho<float>(const Image&, const Chain&, const double*, cudaStream_t, int64_t*);
template void launch_init_rho<double>(const Image&, const Chain&, const double*, cudaStream_t, int64_t*);

// ------------------------------------------------------------------ a8 ---
// mu = K (x) rho (Eq. 1-2) and the per-pixel log likelihood (Eq. 6), double.
// A block takes a tile of TW x (TY RJ) camera pixels, its object values
// converted to double once into shared memory (read straight from the float
// object, each product paid a conversion, on the FP64 unit as well).  A thread
// sums RJ pixels TY rows apart, so a kernel entry is loaded once for RJ
// products.  Bound by the FP64 unit (half a lane a cycle per sub-partition):
// L^2 products and about 170..290 operations of the photon sum a pixel; 1024 x
// 1024, L = 25: with the cumulants 4.2 -> 1.9 ms, without 3.1 -> 1.6.  Small frames take 128-pixel
// tiles, one pixel a thread, to reach more SMs.
__device__ __forceinline__ double block_sum_n(double v, double* sh, int n)
{
    const int tid = threadIdx.x;
    sh[tid] = v;
    __syncthreads();
    for (int o = n / 2; o > 0; o >>= 1) {
        if (tid < o) sh[tid] += sh[tid + o];
        __syncthreads();
    }
    return sh[0];
}

// log likelihood of camera pixel (a, b) at mu; with write, the state derived from mu
template <typename T>
__device__ __forceinline__ double refresh_pixel(const Image& im, const Chain& ch, int a, int b, double mu, int write, int* err)
{
    const size_t x = (size_t)a * im.mu_pitch + b;
    double ll = 0.0;
    if (!(mu > 0.0) || !isfinite(mu)) {
        atomicOr(err, kErrNumeric);
    } else {
        const double* d = im.dat64 + 4 * ((size_t)a * im.W + b);
        Cum6 q;
        if (write && ch.phi) {   // augmented chain: the completed likelihood at its counts
            const int phi = (int)reinterpret_cast<const T*>(ch.phi)[x];
            ll = d[3] + phi_logterm_tab(phi, ::log((double)(T)mu), d[0], d[1], im.lgam) - (double)(T)mu;
        } else if (write && ch.cum) {
            // the cache describes the stored (rounded) expected image
            ll = loglik_sum64<true>(mu, (double)(T)mu, d[0], d[1], d[2], d[3], im.lgam, q);
            ch.cum[x] = q.a;
            ch.cum2[x] = q.b;
        } else if (write && ch.cum64) {
            const double S = photon_record64(mu, d[0], d[1], d[2], ch.cum64 + kCum64 * x);
            ll = loglik_from_sum64(mu, d[0], d[1], d[3], S, photon_mode((float)mu, (float)d[0], (float)d[1]), im.lgam);
        } else {
            ll = loglik_sum64<false>(mu, mu, d[0], d[1], d[2], d[3], im.lgam, q);
        }
    }
    if (write) reinterpret_cast<T*>(ch.mu)[x] = (T)mu;
    return ll;
}

template <typename T, int TW, int TY, int RJ>
__global__ void __launch_bounds__(TW * TY) k_refresh_mu(Image im, Chain ch, double* part_ll, int write, int* err)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ double sh[TW * TY];
    const int L = im.L, tid = threadIdx.x, TC = TW + L - 1, TR = TY * RJ + L - 1;
    double* K = reinterpret_cast<double*>(dyn);                 // [L][L]
    double* r = K + ((L * L + 1) & ~1);                         // [TR][TC]
    const int ntw = (im.W + TW - 1) / TW;
    const int a0 = blockIdx.x / ntw * (TY * RJ), b0 = blockIdx.x % ntw * TW;
    const T* rho = reinterpret_cast<const T*>(ch.rho);
    for (int k = tid; k < L * L; k += TW * TY) K[k] = im.Ke64[k];
    for (int k = tid; k < TR * TC; k += TW * TY) {
        const int i = a0 + k / TC, j = b0 + k % TC;
        r[k] = i < im.Ho && j < im.Wo ? (double)rho[(size_t)i * im.Wo + j] : 0.0;
    }
    __syncthreads();
    // mu[a][b] = sum K[p][q] rho[a + L-1-p][b + L-1-q]
    const int tx = tid % TW, ty = tid / TW;
    double mu[RJ];
#pragma unroll
    for (int j = 0; j < RJ; ++j) mu[j] = 0.0;
    for (int p = 0; p < L; ++p) {
        const double* row = r + (ty + L - 1 - p) * TC + tx + L - 1;
        for (int q = 0; q < L; ++q) {
            const double k = K[p * L + q];
#pragma unroll
            for (int j = 0; j < RJ; ++j) mu[j] += k * row[j * TY * TC - q];
        }
    }
    double ll = 0.0;
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
        const int a = a0 + ty + j * TY, b = b0 + tx;
        if (a < im.H && b < im.W) ll += refresh_pixel<T>(im, ch, a, b, mu[j], write, err);
    }
    const double s = block_sum_n(ll, sh, TW * TY);
    if (tid == 0) part_ll[blockIdx.x] = s;
}

// Object lattice finer than the camera: straight from the object.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_refresh_mu_fine(Image im, Chain ch, double* part_ll, int write, int* err)
{
    __shared__ double sh[kRedThreads];
    const int idx = blockIdx.x * kRedThreads + threadIdx.x;
    double ll = 0.0;
    if (idx < im.H * im.W) {
        const int a = idx / im.W, b = idx % im.W;
        const T* rho = reinterpret_cast<const T*>(ch.rho);
        // Eq. 1 on the object lattice: mu[a][b] = sum Ke[p][q] rho[f a + Le-1-p][f b + Le-1-q]
        const int Le = im.Le, f = im.f;
        double mu = 0.0;
        for (int p = 0; p < Le; ++p) {
            const T* row = rho + (size_t)(f * a + Le - 1 - p) * im.Wo + (f * b + Le - 1);
            for (int q = 0; q < Le; ++q) mu += im.Ke64[p * Le + q] * (double)row[-q];
        }
        ll = refresh_pixel<T>(im, ch, a, b, mu, write, err);
    }
    const double s = block_sum(ll, sh);
    if (threadIdx.x == 0) part_ll[blockIdx.x] = s;
}

// Patch spectra by direct DFT (canonical half) and the patch log prior of Eq. 8:
//   sum_e mult_e (alpha_e - 1) log|X_e| + (K - 1) log sum_e mult_e |X_e|.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_refresh_spec(Image im, Chain ch, double* part_lp, int write)
{
    // one block per patch: its half spectrum by the 2-D DFT taken as two
    // 1-D transforms (rows, then columns), O(ph pw (ph + pw)) instead of
    // O((ph pw)^2) for the direct sum, in double in shared memory:
    //   Y[u][l] = sum_v x[u][v] exp(-2 pi i l v / pw),
    //   X[k][l] = sum_u Y[u][l] exp(-2 pi i k u / ph)
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ double sh[kRedThreads];
    const int p = blockIdx.x;
    const int pi = p / im.npj, pj = p % im.npj;
    const Shape& sp = im.shape[shape_index(im, pi, pj)];
    const int ph = sp.ph, pw = sp.pw, n = ph * pw;
    double* x = reinterpret_cast<double*>(dyn);                    // [ph][pw]
    double2* Y = reinterpret_cast<double2*>(dyn) + (n + 1) / 2;     // [ph][pw]
    const T* rho = reinterpret_cast<const T*>(ch.rho) + (size_t)pi * im.S * im.Wo + pj * im.S;
    const double2* twh = reinterpret_cast<const double2*>(im.tw64) + sp.twh_off;
    const double2* tww = reinterpret_cast<const double2*>(im.tw64) + sp.tww_off;
    for (int e = threadIdx.x; e < n; e += kRedThreads) {
        const int u = e / pw, v = e - (e / pw) * pw;
        x[e] = (double)rho[(size_t)u * im.Wo + v];
    }
    __syncthreads();
    // (every l, although the rows are real: the table's conjugate twiddles differ
    // in their last place, which would turn float roundings of small coefficients)
    for (int e = threadIdx.x; e < n; e += kRedThreads) {
        const int u = e / pw, l = e - u * pw;
        double re = 0.0, imv = 0.0;
        for (int v = 0, j = 0; v < pw; ++v) {
            const double2 w = tww[j];
            re += x[u * pw + v] * w.x;
            imv += x[u * pw + v] * w.y;
            j += l;
            j -= j >= pw ? pw : 0;
        }
        Y[e] = make_double2(re, imv);
    }
    __syncthreads();
    using T2 = typename Vec2<T>::type;
    T2* spec = reinterpret_cast<T2*>(ch.spec) + im.patch_off[p];
    double sl = 0.0, sm = 0.0;
    for (int e = threadIdx.x; e < sp.nhalf; e += kRedThreads) {
        const int kl = im.ent_kl[sp.ent_off + e];
        const int k = kl >> 16, l = kl & 0xffff;
        double re = 0.0, imv = 0.0;
        for (int u = 0, j = 0; u < ph; ++u) {
            const double2 w = twh[j];
            const double2 y = Y[u * pw + l];
            re += y.x * w.x - y.y * w.y;
            imv += y.x * w.y + y.y * w.x;
            j += k;
            j -= j >= ph ? ph : 0;
        }
        if (write) {
            T2 X;
            X.x = (T)re;
            X.y = (T)imv;
            spec[e] = X;
        }
        const double n2 = re * re + imv * imv;
        sl += im.ent_wa64[sp.ent_off + e] * log(n2);
        sm += im.ent_m64[sp.ent_off + e] * sqrt(n2);
    }
    const double tl = block_sum(sl, sh);
    const double tm = block_sum(sm, sh);
    if (threadIdx.x == 0) part_lp[p] = tl + (double)(sp.K - 1) * log(tm);
}

__global__ void __launch_bounds__(kRedThreads) k_refresh_total(const double* part_ll, int n_ll, const double* part_lp,
                                                              int n_lp, double* out, const int* out_index)
{
    __shared__ double sh[kRedThreads];
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < n_ll; k += kRedThreads) a += part_ll[k];
    for (int k = threadIdx.x; k < n_lp; k += kRedThreads) b += part_lp[k];
    const double ta = block_sum(a, sh);
    const double tb = block_sum(b, sh);
    if (threadIdx.x == 0) out[out_index ? *out_index : 0] = ta + tb;
}

template <typename T>
cudaError_t launch_refresh(const Image& im, const Chain& ch, double* scratch, int write_state, double* out_logpost,
                    const int* out_index, int* err, cudaStream_t st, int64_t* launches)
{
    const int nblk = refresh_blocks(im.H, im.W, im.f);
    double* part_ll = scratch;
    double* part_lp = scratch + nblk;
    if (im.f > 1) {
        k_refresh_mu_fine<T><<<nblk, kRedThreads, 0, st>>>(im, ch, part_ll, write_state, err);
    } else {
        const bool small = refresh_small(im.H, im.W);
        const void* fn = small ? (const void*)k_refresh_mu<T, 32, 4, 1> : (const void*)k_refresh_mu<T, 64, 4, 4>;
        const int TC = (small ? 32 : 64) + im.L - 1, TR = (small ? 4 : 16) + im.L - 1;
        const size_t sm = 8 * (size_t)(((im.L * im.L + 1) & ~1) + TC * TR);
        const cudaError_t e = raise_smem_limit(fn, sm);
        if (e != cudaSuccess) return e;
        if (small) k_refresh_mu<T, 32, 4, 1><<<nblk, 128, sm, st>>>(im, ch, part_ll, write_state, err);
        else k_refresh_mu<T, 64, 4, 4><<<nblk, 256, sm, st>>>(im, ch, part_ll, write_state, err);
    }
    // the patch and its row transforms in shared memory (24 bytes per patch pixel)
    const size_t smem = 8 * (size_t)(((size_t)im.S * im.S + 1) / 2 * 2) + 16 * (size_t)im.S * im.S;
    const cudaError_t e = raise_smem_limit((const void*)k_refresh_spec<T>, smem);
    if (e != cudaSuccess) return e;
    k_refresh_spec<T><<<im.n_patches, kRedThreads, smem, st>>>(im, ch, part_lp, write_state);
    k_refresh_total<<<1, kRedThreads, 0, st>>>(part_ll, nblk, part_lp, im.n_patches, out_logpost, out_index);
    *launches += 3;
    return cudaGetLastError();
}
template cudaError_t launch_refresh<float>(const Image&, const Chain&, double*, int, double*, const int*, int*, cudaStream_t,
                                           int64_t*);
template cudaError_t launch_refresh<double>(const Image&, const Chain&, double*, int, double*, const int*, int*, cudaStream_t,
                                            int64_t*);

// ------------------------------------------------- photon-count draw -----
__global__ void k_lgamma(double* out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kLgamma) out[k] = lgamma((double)k + 1.0);
}

void launch_lgamma(double* out, cudaStream_t st, int64_t* launches)
{
    k_lgamma<<<(kLgamma + 127) / 128, 128, 0, st>>>(out);
    ++*launches;
}

template <typename T>
__global__ void k_sample_phi(Image im, Chain ch, int t, int* err)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= im.H * im.W) return;
    const int a = idx / im.W, b = idx % im.W;
    const size_t k = (size_t)a * im.mu_pitch + b;
    const T mu = reinterpret_cast<const T*>(ch.mu)[k];
    const Dat4<T> dv = dat<T>(im)[idx];
    const uint4 x = philox4x32_10(make_uint4((uint32_t)idx, (uint32_t)t, (uint32_t)ch.chain, 1u), im.seed_lo,
                                  im.seed_hi);
    int status = 0;
    const int phi = sample_phi<T>(mu, dv.c, dv.is2, uniform23<T>(x.x), status);
    if (status) atomicOr(err, kErrNumeric);
    reinterpret_cast<T*>(ch.phi)[k] = (T)phi;
}

template <typename T>
void launch_sample_phi(const Image& im, const Chain& ch, int t, int* err, cudaStream_t st, int64_t* launches)
{
    const int n = im.H * im.W;
    k_sample_phi<T><<<(n + 255) / 256, 256, 0, st>>>(im, ch, t, err);
    ++*launches;
}
template void launch_sample_phi<float>(const Image&, const Chain&, int, int*, cudaStream_t, int64_t*);
template void launch_sample_phi<double>(const Image&, const Chain&, int, int*, cudaStream_t, int64_t*);

// ------------------------------------------------------------ reset -----
__global__ void k_reset(const Image* imgs, const Chain* chains, int n_slots)
{
    const Chain& ch = chains[blockIdx.x];
    const int np = imgs[ch.img].n_patches;
    for (int k = threadIdx.x; k < np; k += blockDim.x) ch.prog[(size_t)k * kProgStride] = 0;
    for (int k = threadIdx.x; k < n_slots * np; k += blockDim.x) ch.trace_part[k] = 0.0;
}

void launch_reset(const Image* d_imgs, const Chain* d_chains, int n_chains, int n_slots, cudaStream_t st,
                  int64_t* launches)
{
    k_reset<<<n_chains, 256, 0, st>>>(d_imgs, d_chains, n_slots);
    ++*launches;
}

// ------------------------------------------------------------ trace -----
// trace[t0 + s + 1] = trace[t0] + sum_{s' <= s} sum_p part[s'][p]: the double
// running sum of accepted dL + dP, per chain (one block per chain); t0 is the
// chain's sweep counter, which this kernel then advances by n.
__global__ void __launch_bounds__(kRedThreads) k_trace(const Image* imgs, const Chain* chains, int n)
{
    __shared__ double sh[kRedThreads];
    const Chain& ch = chains[blockIdx.x];
    const int np = imgs[ch.img].n_patches;
    const int t0 = *ch.tdev;
    double cum = ch.trace[t0];
    for (int s = 0; s < n; ++s) {
        double a = 0.0;
        for (int p = threadIdx.x; p < np; p += kRedThreads) a += ch.trace_part[(size_t)s * np + p];
        cum += block_sum(a, sh);
        if (threadIdx.x == 0) ch.trace[t0 + s + 1] = cum;
    }
    __syncthreads();
    if (threadIdx.x == 0) *ch.tdev = t0 + n;
}

void launch_trace(const Image* d_imgs, const Chain* d_chains, int n_chains, int n_sweeps, cudaStream_t st,
                  int64_t* launches)
{
    k_trace<<<n_chains, kRedThreads, 0, st>>>(d_imgs, d_chains, n_sweeps);
    ++*launches;
}

__global__ void k_set_counters(const Chain* chains, int n, int value)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) *chains[k].tdev = value;
}

void launch_set_counters(const Chain* d_chains, int n_chains, int value, cudaStream_t st, int64_t* launches)
{
    k_set_counters<<<(n_chains + 127) / 128, 128, 0, st>>>(d_chains, n_chains, value);
    ++*launches;
}

// --------------------------------------------------------- conversions --
template <typename T>
__global__ void k_to_double(const T* src, double* dst, int rows, int cols, int pitch)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)rows * cols) return;
    const int r = (int)(idx / cols), c = (int)(idx % cols);
    dst[idx] = (double)src[(size_t)r * pitch + c];
}

template <typename T>
void launch_convert(const void* src, double* dst, int64_t n, int rows, int cols, int src_pitch, cudaStream_t st,
                    int64_t* launches)
{
    (void)n;
    const int64_t tot = (int64_t)rows * cols;
    k_to_double<T><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(reinterpret_cast<const T*>(src), dst, rows, cols,
                                                                   src_pitch);
    ++*launches;
}
template void launch_convert<float>(const void*, double*, int64_t, int, int, int, cudaStream_t, int64_t*);
template void launch_convert<double>(const void*, double*, int64_t, int, int, int, cudaStream_t, int64_t*);

template <typename T>
__global__ void k_from_double(const double* src, T* dst, int64_t n)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) dst[idx] = (T)src[idx];
}

template <typename T>
void launch_set_rho(const double* src, void* dst, int64_t n, cudaStream_t st, int64_t* launches)
{
    k_from_double<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(src, reinterpret_cast<T*>(dst), n);
    ++*launches;
}
template void launch_set_rho<float>(const double*, void*, int64_t, cudaStream_t, int64_t*);
template void launch_set_rho<double>(const double*, void*, int64_t, cudaStream_t, int64_t*);

template <typename T>
__global__ void k_fill(T* dst, int64_t n, T value)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) dst[idx] = value;
}

template <typename T>
void launch_fill(void* dst, int64_t n, double value, cudaStream_t st, int64_t* launches)
{
    k_fill<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(reinterpret_cast<T*>(dst), n, (T)value);
    ++*launches;
}
template void launch_fill<float>(void*, int64_t, double, cudaStream_t, int64_t*);
template void launch_fill<double>(void*, int64_t, double, cudaStream_t, int64_t*);

// posterior mean (variance, standard deviation, coefficient of variation)
// pooled over the chains of one problem
__global__ void k_mean(const double* sum, int n_chains, int64_t stride, int Wo, int crop_r, int oh, int ow,
                       double inv_n, double* out, const double* sq, int kind)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= oh * ow) return;
    const int y = idx / ow + crop_r, x = idx % ow + crop_r;
    const size_t m = (size_t)y * Wo + x;
    double s = 0.0, q = 0.0;
    for (int c = 0; c < n_chains; ++c) {
        s += sum[c * stride + m];
        if (kind) q += sq[c * stride + m];
    }
    const double mean = s * inv_n;
    if (kind == 0) {
        out[idx] = mean;
        return;
    }
    const double var = fmax(q * inv_n - mean * mean, 0.0);
    out[idx] = kind == 1 ? var : kind == 2 ? sqrt(var) : sqrt(var) / mean;
}

void launch_mean(const double* sum, int n_chains_img, int64_t chain_stride_elems, int Ho, int Wo, int crop_r,
                 int out_h, int out_w, double inv_n, double* out, const double* sq, int kind, cudaStream_t st,
                 int64_t* launches)
{
    (void)Ho;
    const int n = out_h * out_w;
    k_mean<<<(n + 255) / 256, 256, 0, st>>>(sum, n_chains_img, chain_stride_elems, Wo, crop_r, out_h, out_w, inv_n,
                                            out, sq, kind);
    ++*launches;
}

// ------------------------------------------------------------ quantiles --
// One block per output pixel: the pixel's kept values of every chain are
// loaded into shared memory, padded with +inf to a power of two, sorted by a
// bitonic network, and each requested quantile is read off the order
// statistics by linear interpolation at h = (n - 1) q.
template <typename T>
__global__ void __launch_bounds__(256) k_quantiles(const T* samples, int64_t chain_stride, int n_chains, int first,
                                                  int count, int64_t obj_pixels, int Wo, int crop_r, int out_w,
                                                  int64_t pix0, int npow2, const double* q, int nq, double* out,
                                                  int64_t npix)
{
    extern __shared__ double sv[];
    const int64_t i = blockIdx.x;
    const int64_t pix = pix0 + i;
    const int64_t y = pix / out_w + crop_r, x = pix % out_w + crop_r;
    const int64_t m = y * Wo + x;
    const int n = count * n_chains;
    for (int k = threadIdx.x; k < npow2; k += blockDim.x) {
        double v = INFINITY;
        if (k < n) {
            const int c = k / count, slot = first + (k - c * count);
            v = (double)samples[c * chain_stride + (int64_t)slot * obj_pixels + m];
        }
        sv[k] = v;
    }
    __syncthreads();
    for (int size = 2; size <= npow2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int k = threadIdx.x; k < npow2 / 2; k += blockDim.x) {
                // element pair (a, b) of this stage, ascending where (a & size) == 0
                const int a = 2 * k - (k & (stride - 1)), b = a + stride;
                const bool up = (a & size) == 0;
                const double va = sv[a], vb = sv[b];
                if ((va > vb) == up) {
                    sv[a] = vb;
                    sv[b] = va;
                }
            }
            __syncthreads();
        }
    for (int k = threadIdx.x; k < nq; k += blockDim.x) {
        const double h = (double)(n - 1) * q[k];
        int lo = (int)floor(h);
        lo = lo < 0 ? 0 : lo > n - 1 ? n - 1 : lo;
        const int hi = lo + 1 < n ? lo + 1 : n - 1;
        out[(int64_t)k * npix + i] = sv[lo] + (h - (double)lo) * (sv[hi] - sv[lo]);
    }
}

// Up to 32 E values a pixel: one warp sorts a pixel's values in registers, E a
// lane (element i of the sequence in register i % E of lane i / E), exchanging
// across lanes by shuffles, in the samples' own type.  A block takes kQuantPix
// consecutive pixels, so that the kept objects are read (pixel fastest) and the
// quantile maps written in whole sectors; the sorted values meet the
// interpolation in shared memory.  Bound by its compare-exchanges (issue), not
// by the samples' bytes.  100 kept objects of a 512 x 512 frame, five
// quantiles: 1.33 ms in the block-per-pixel form below, whose double-precision
// exchanges all go through shared memory and barriers, and 0.39 ms here.
constexpr int kQuantPix = 32;

template <typename T, int E>
__global__ void __launch_bounds__(256) k_quantiles_warp(const T* samples, int64_t chain_stride, int n_chains, int first,
                                                       int count, int64_t obj_pixels, int Wo, int crop_r, int out_w,
                                                       int64_t pix0, const double* q, int nq, double* out, int64_t npix)
{
    __shared__ T sv[32 * E * (kQuantPix + 1)];       // [value][pixel]
    constexpr int P = kQuantPix + 1;
    const int n = count * n_chains, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * kQuantPix;
    const int np = (int)(npix - i0 < kQuantPix ? npix - i0 : kQuantPix);
    {
        const int p = lane;
        const int64_t pix = pix0 + i0 + p, m = (pix / out_w + crop_r) * Wo + pix % out_w + crop_r;
        for (int k = warp; k < n && p < np; k += 8) {
            const int c = k / count, slot = first + (k - c * count);
            sv[k * P + p] = samples[c * chain_stride + (int64_t)slot * obj_pixels + m];
        }
    }
    __syncthreads();
    for (int p = warp; p < np; p += 8) {
        T v[E];
#pragma unroll
        for (int r = 0; r < E; ++r) v[r] = lane * E + r < n ? sv[(lane * E + r) * P + p] : (T)INFINITY;
#pragma unroll
        for (int size = 2; size <= 32 * E; size <<= 1) {
#pragma unroll
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                if (stride >= E) {   // partner in another lane
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        const T o = __shfl_xor_sync(0xffffffffu, v[r], stride / E);
                        const bool up = ((lane * E + r) & size) == 0, low = (lane & (stride / E)) == 0;
                        v[r] = (up == low) ? (o < v[r] ? o : v[r]) : (o < v[r] ? v[r] : o);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        if ((r & stride) == 0) {
                            const bool up = ((lane * E + r) & size) == 0;
                            const T x = v[r], y = v[r + stride];
                            const bool sw = (x > y) == up;
                            v[r] = sw ? y : x;
                            v[r + stride] = sw ? x : y;
                        }
                    }
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < E; ++r)
            if (lane * E + r < n) sv[(lane * E + r) * P + p] = v[r];
    }
    __syncthreads();
    for (int x = threadIdx.x; x < nq * kQuantPix; x += blockDim.x) {
        const int k = x / kQuantPix, p = x - k * kQuantPix;
        if (p >= np) continue;
        const double h = (double)(n - 1) * q[k];
        int lo = (int)floor(h);
        lo = lo < 0 ? 0 : lo > n - 1 ? n - 1 : lo;
        const int hi = lo + 1 < n ? lo + 1 : n - 1;
        const double a = (double)sv[lo * P + p], b = (double)sv[hi * P + p];
        out[(int64_t)k * npix + i0 + p] = a + (h - (double)lo) * (b - a);
    }
}

template <typename T>
cudaError_t launch_quantiles(const void* samples, int64_t chain_stride, int n_chains, int first, int count,
                             int64_t obj_pixels, int Wo, int crop_r, int out_w, int64_t pix0, int64_t npix,
                             const double* q, int nq, double* out, cudaStream_t st, int64_t* launches)
{
    // warp form while the block's values fit static shared memory (33 KB at 256
    // values a pixel in float and 128 in double; twice as many would pass 48 KB)
    const int n = count * n_chains;
    const unsigned wb = (unsigned)((npix + kQuantPix - 1) / kQuantPix);
    const T* sp = reinterpret_cast<const T*>(samples);
#define BD_QWARP(E)                                                                                                       \
    k_quantiles_warp<T, E><<<wb, 256, 0, st>>>(sp, chain_stride, n_chains, first, count, obj_pixels, Wo, crop_r, out_w, pix0, \
                                               q, nq, out, npix)
    if (n <= (sizeof(T) == 4 ? 256 : 128)) {
        if (n <= 32) BD_QWARP(1);
        else if (n <= 64) BD_QWARP(2);
        else if (n <= 128) BD_QWARP(4);
        else if constexpr (sizeof(T) == 4) BD_QWARP(8);
        ++*launches;
        return cudaGetLastError();
    }
#undef BD_QWARP
    int npow2 = 2;
    while (npow2 < n) npow2 <<= 1;
    const size_t smem = sizeof(double) * (size_t)npow2;
    const cudaError_t e = raise_smem_limit((const void*)k_quantiles<T>, smem);
    if (e != cudaSuccess) return e;
    k_quantiles<T><<<(unsigned)npix, 256, smem, st>>>(reinterpret_cast<const T*>(samples), chain_stride, n_chains,
                                                      first, count, obj_pixels, Wo, crop_r, out_w, pix0, npow2, q,
                                                      nq, out, npix);
    ++*launches;
    return cudaGetLastError();
}
template cudaError_t launch_quantiles<float>(const void*, int64_t, int, int, int, int64_t, int, int, int, int64_t,
                                             int64_t, const double*, int, double*, cudaStream_t, int64_t*);
template cudaError_t launch_quantiles<double>(const void*, int64_t, int, int, int, int64_t, int, int, int, int64_t,
                                              int64_t, const double*, int, double*, cudaStream_t, int64_t*);

}  // namespace bd
