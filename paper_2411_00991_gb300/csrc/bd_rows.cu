// bd_rows.cu -- row-run form of the sweep kernel (float: marginal on any object
// lattice, augmented on the camera grid).
//
// The classes of a sweep are taken S at a time, one class row u at a time:
// within a row the offsets v = 0..S-1 follow each other, and a block scores a
// run of up to V consecutive classes (u, v0..v0+n-1) of one patch at once from
// the state before the run.  If none is accepted (in a long chain all but a
// percent of them) the whole run is decided by one exchange of partial sums,
// one neighbour wait and one published word; otherwise the first accepted
// update is written and the run's later classes are scored again.  Either way
// every decision is taken on exactly the state the sequential raster scan
// gives it, and the cells and entries of an update are summed by the same
// threads in the same order as in bd_sweep.cu, so chains are bit-identical.
//
// Which neighbours a run waits for.  Two updates touch a common camera pixel
// only when their object pixels are less than L apart in rows and in columns,
// and a class pixel of the patch at offset (di, dj) lies di S + (u' - u) rows
// and dj S + (v' - v) columns away, S >= L.  Of the updates that come earlier
// in the raster scan, update (u, v) therefore meets
//   the right patch's only up to (u, v - 1)              (v' < v),
//   the left and the three lower patches' only up to row u - 1,
//   the three upper patches' only of the previous sweep   (u' > u).
// Within a row a patch depends on its right neighbour alone: a block takes the
// patches of its tile from right to left, and waits per run for the right tile
// to have finished the run's classes but the last, for the left and lower
// tiles to have finished the previous row, and for the upper tiles to have
// finished the previous sweep -- waits that are normally long satisfied.
//
// The union of the run's windows (L rows of L + V - 1 columns of the expected
// image and the photon cumulants) is copied once per run and patch into shared
// memory by the TMA engine while the block scores the run's prior changes, so
// the chain's state is read S / V times less often than class by class.
//
// What bounds it: instruction issue and its latency (no pipe near its peak).
// Against the general form: warp instructions per update 3.3k -> 1.7k on the
// 512 x 512 frame (L = 17), whose partial sums are exchanged, neighbours polled
// and window bounds worked out once per run; DRAM reads per update 31 -> 8 KB
// on the 2048 x 2048 frame (L = 31).  ms per sweep, before and after (50, 2 and
// 10 sweeps of long chains, with refresh and read-out): 512 x 512 L = 17 1.29
// and 0.91; 2048 x 2048 L = 31 x 4 chains 189 and 97; six frames 128..768
// x 4 chains 52 and 22; 64 x 64 L = 9 0.30 and 0.12; 150 x 150 on a twice finer
// lattice 1.13 and 0.40.
#include "bd_device.cuh"
#include "bd_update.cuh"

namespace bd {

namespace {

// x[i] summed over the warp, P (a power of two) values at once: at each of the
// first log2 P steps a lane keeps half of its values and hands over the other
// half, so P values take P + 4 - log2 P shuffles instead of 5 P.  The pairs
// added at every step are those of warp_sum, so each sum has the same bits.
// Returns the sum of value lane >> (5 - log2 P).
template <int P>
__device__ __forceinline__ float warp_sum_many(float (&x)[P])
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = P; n > 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const float keep = up ? x[i + n / 2] : x[i], give = up ? x[i] : x[i + n / 2];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    float v = x[0];
#pragma unroll
    for (; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__host__ __device__ constexpr int pow2_at_least(int n) { return n <= 1 ? 1 : 2 * pow2_at_least((n + 1) / 2); }
__host__ __device__ constexpr int log2_of(int p) { return p <= 1 ? 0 : 1 + log2_of(p / 2); }

}  // namespace

// One run's entry tables of a full patch: frequency (k << 16 | l, bit 31 set
// for multiplicity 2) and weight.
struct RowEnt { int kl; float wa; };

constexpr uint32_t kUndecided = 0x80000000u;   // in place of a run's accept mask: the right tile is not done

// FINE: an object lattice f times finer than the camera.  A class offset v is
// then a lattice column; its window starts at camera column (j0 + v) / f, and
// its kernel entries depend on the phase (j0 + v) mod f.
template <bool AUG, bool FINE, int VG, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_sweep_rows(SweepArgs a)
{
    using P = Prec<float>;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_ci, s_abort, s_right;
    __shared__ uint32_t s_mask, s_cnt;
    __shared__ short s_v0[kMaxS + 2];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ __align__(16) uint32_t s_chd[sizeof(Chain) / 4];
    __shared__ __align__(16) uint32_t s_imd[sizeof(Image) / 4];
    __shared__ double s_phid[AUG ? kRowMaxTeams : 1][8];   // [team][warp]

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) {
        int lo = 0, hi = a.n_chains - 1;
        while (lo < hi) {   // last chain with cta_base <= blockIdx.x
            const int mid = (lo + hi + 1) >> 1;
            if (a.chains[mid].cta_base <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        s_ci = lo;
        s_abort = 0;
        s_right = 0;
        s_cnt = 0;
        mbar_init(&s_bar, 1);
    }
    __syncthreads();
    {
        const uint32_t* gc = reinterpret_cast<const uint32_t*>(&a.chains[s_ci]);
        const uint32_t* gi = reinterpret_cast<const uint32_t*>(&a.imgs[a.chains[s_ci].img]);
        for (int k = tid; k < (int)(sizeof(Chain) / 4); k += blockDim.x) s_chd[k] = gc[k];
        for (int k = tid; k < (int)(sizeof(Image) / 4); k += blockDim.x) s_imd[k] = gi[k];
    }
    const char* tmap = reinterpret_cast<const char*>(a.rmaps) + (size_t)s_ci * kRowMapBytes;
    __syncthreads();
    const Chain& ch = *reinterpret_cast<const Chain*>(s_chd);
    const Image& im = *reinterpret_cast<const Image*>(s_imd);
    const int t0 = *ch.tdev;
    const int tl = (int)blockIdx.x - ch.cta_base;
    const int ti = tl / ch.ntj, tj = tl - (tl / ch.ntj) * ch.ntj;
    // L: side of an update's camera window; f, Le: lattice cells a camera pixel, side of the kernel
    const int S = im.S, L = FINE ? im.Lc : im.L, LL = L * L, f = FINE ? im.f : 1;
    auto Le = [&]() { return FINE ? im.Le : L; };
    const int pi0 = ti * ch.tpi, pj0 = tj * ch.tpj;
    const int tw_ = min(ch.tpj, im.npj - pj0), th_ = min(ch.tpi, im.npi - pi0), npt = th_ * tw_;
    // the block: G update teams of NT threads, each scoring VG classes of a run
    const int NT = im.team, G = blockDim.x / NT, V = G * VG, nwt = NT >> 5;
    const int g = tid / NT, lt = tid - g * NT, gw = lt >> 5, vb = g * VG;
    const int RN = (S + V - 1) / V;                 // runs per class row
    constexpr int RH = rows_ring_half(VG);          // ring slots drawn at a time
    const int BW = rows_box_w(L, V, f);
    const int VR = rows_ring_slots(V), DP = RH / VR; // proposal ring: slots per patch-run, patch-runs per draw
    const Shape& sh0 = im.shape[0];
    const RowsSmem sp = rows_smem(L, Le(), f, V, G, nwt, im.n_tw, sh0.nhalf, AUG, a.resident ? im.max_nhalf : 0);
    float* Ks = reinterpret_cast<float*>(smem + sp.K);
    float2* tws = reinterpret_cast<float2*>(smem + sp.tw);
    RowEnt* ent0 = reinterpret_cast<RowEnt*>(smem + sp.ent);
    float4* ring = reinterpret_cast<float4*>(smem + sp.ring);
    float* red = reinterpret_cast<float*>(smem + sp.red);
    const int RS = nwt * 3 * (V + G);           // one set of partial sums
    float* wmu = reinterpret_cast<float*>(smem + sp.mu);
    float4* wcum = reinterpret_cast<float4*>(smem + sp.cum);
    float2* wcum2 = reinterpret_cast<float2*>(smem + sp.cum2);
    float* wphi = reinterpret_cast<float*>(smem + sp.cum);
    float2* spec_s = reinterpret_cast<float2*>(smem + sp.spec);

    float* rho_g = reinterpret_cast<float*>(ch.rho);
    float* mu_g = reinterpret_cast<float*>(ch.mu);
    float2* spec_g = reinterpret_cast<float2*>(ch.spec);
    const Dat4<float>* dat_g = dat<float>(im);

    for (int k = tid; k <= RN; k += blockDim.x) s_v0[k] = (short)(k * S / RN);   // first class of each run
    for (int k = tid; k < Le() * Le(); k += blockDim.x) Ks[k] = im.Ke32[k];
    for (int k = tid; k < im.n_tw; k += blockDim.x) tws[k] = reinterpret_cast<const float2*>(im.tw32)[k];
    for (int k = tid; k < sh0.nhalf; k += blockDim.x)   // full patches' entries (others are read from global memory)
        ent0[k] = {im.ent_kl[sh0.ent_off + k] | (im.ent_m32[sh0.ent_off + k] > 1.0f ? (int)0x80000000 : 0),
                   im.ent_wa32[sh0.ent_off + k]};
    if (a.resident) {   // one patch per block: its spectrum stays in shared memory
        const Shape& sh = im.shape[shape_index(im, pi0, pj0)];
        for (int e = tid; e < sh.nhalf; e += blockDim.x) spec_s[e] = spec_g[im.patch_off[pi0 * im.npj + pj0] + e];
    }
    // where the patches' spectra start: every row of patches but a partial last one is alike
    const bool rpart = im.npi * S > im.Ho, cpart = im.npj * S > im.Wo;
    const int sz_f = (sh0.nhalf + 1) & ~1, sz_b = (im.shape[2].nhalf + 1) & ~1;
    const int sz_row = (im.npj - (cpart ? 1 : 0)) * sz_f + (cpart ? (im.shape[1].nhalf + 1) & ~1 : 0);
    // this thread's first window cell and its step from cell to cell in the box
    const int kc0 = lt - (lt / L) * L, idx0 = (lt / L) * BW + kc0;
    const int dkc = NT - (NT / L) * L, didx = (NT / L) * BW + dkc, dwrap = BW - L;
    // the service warp (the last: the first has the most cells and entries)
    // waits for the neighbours and issues the window copies; its lane k < 8
    // watches neighbour k: the progress word, and what a run waits for it to
    // have finished (kind 0, right: the run's classes but the last; 1: the
    // previous class row; 2: the previous sweep)
    const bool service = warp == nw - 1;
    if (service && lane == 0) {
        tensormap_acquire(tmap);
        tensormap_acquire(tmap + 128);
        if constexpr (!AUG) tensormap_acquire(tmap + 256);
    }
    const uint32_t* nword = nullptr;
    int nkind = 0;
    if (lane < 8) {
        const int d = lane < 4 ? lane : lane + 1, di = d / 3 - 1, dj = d - (d / 3) * 3 - 1;
        const int ni = ti + di, nj = tj + dj;
        if (ni >= 0 && ni < ch.nti && nj >= 0 && nj < ch.ntj)
            nword = reinterpret_cast<const uint32_t*>(ch.prog) + (size_t)(ni * ch.ntj + nj) * kProgStride;
        nkind = di < 0 ? 2 : (di == 0 && dj > 0) ? 0 : 1;
    }
    uint32_t nseen = 0;      // changes of the neighbour this block has acquired
    uint32_t my_word = 0;    // this block's last published word (thread 0)
    uint32_t par = 0;        // phase of s_bar
    int n_acc = 0;
    const int nsw = ch.n_sweeps > 0 ? ch.n_sweeps : a.n_sweeps;
    const int S2 = S * S, SS = AUG ? S2 + 1 : S2;
    const int NPR = S * RN * npt;                   // patch-runs per sweep
    const int NE = nsw * NPR;
    // draws up to 2 DP - 1 patch-runs ahead must not include a pixel whose
    // update in the sweep before is still to come
    const bool ahead = NPR >= 2 * DP;

    // the proposals of patch-runs e0 .. e0 + cnt - 1 (lane: one class of one
    // patch-run), into ring slots base ..
    auto draw = [&](int e0, int cnt, int base) {
        const int q_ = lane / VR, v_ = lane - q_ * VR, e = e0 + q_;
        if (q_ >= cnt || e >= NE) return;
        int x = e / npt;
        const int q = e - x * npt;
        const int rn = x - (x / RN) * RN;
        x /= RN;
        const int sw = x / S, u = x - sw * S;
        const int pi = pi0 + q / tw_, pj = pj0 + tw_ - 1 - (q - (q / tw_) * tw_);
        const Shape& sh = im.shape[shape_index(im, pi, pj)];
        const int v0 = s_v0[rn], v = v0 + v_;
        if (v >= s_v0[rn + 1] || u >= sh.ph || v >= sh.pw) return;
        const int m = (pi * S + u) * im.Wo + pj * S + v;
        float4 d;
        proposal<float>(im, ch, m, t0 + 1 + sw, __ldcg(rho_g + m), d.x, d.y, d.z, d.w);
        ring[base + lane] = d;
    };
    __syncthreads();
    if (ahead && warp == 0) draw(0, DP, 0);
    __syncthreads();

    // one poll of this lane's neighbour word until it shows `need` steps (bounded)
    auto poll = [&](uint32_t need, uint32_t& w) -> bool {
        w = (uint32_t)ld_relaxed(reinterpret_cast<const int*>(nword));
        if ((w >> kRowChgBits) >= need) return true;
        const uint64_t b = global_ns();
        uint32_t it = 0;
        while (((w = (uint32_t)ld_relaxed(reinterpret_cast<const int*>(nword))) >> kRowChgBits) < need) {
            ++it;
            if ((it & 31u) == 0u) {
                if (ld_relaxed(a.err) != 0) return false;
                if (global_ns() - b > a.wait_ns || it > kWaitPolls) {
                    atomicOr(a.err, kErrTimeout);
                    return false;
                }
            }
            if (it > 64u) __nanosleep(32);
        }
        return true;
    };
    // service warp: waits until the neighbours have finished the given steps
    // (by kind), then orders their changes before this block's reads.  right:
    // whether the right tile has also finished right_fin.
    auto wait_nbrs = [&](uint32_t sweep_s, uint32_t row_s, uint32_t right_s, uint32_t right_fin, bool& right, bool& fence_copy) -> bool {
        bool ok = true, chg = false, fin = true;
        if (nword != nullptr) {
            uint32_t w;
            ok = poll(nkind == 0 ? right_s : nkind == 1 ? row_s : sweep_s, w);
            chg = ok && (w & kRowChgMask) != nseen;   // a change this block has not acquired yet
            nseen = w & kRowChgMask;
            fin = nkind != 0 || (w >> kRowChgBits) >= right_fin;
        }
        if (__any_sync(0xffffffffu, chg)) {
            fence_acq_rel_gpu();
            fence_copy = true;
        }
        right = __all_sync(0xffffffffu, fin);
        return __all_sync(0xffffffffu, ok);
    };
    bool fence_copy = true;   // changes since the last window copy: order them before the next (async proxy)
    auto publish = [&](uint32_t steps, bool changed) {
        if (tid == 0 && (int)blockIdx.x != a.silent_block) {
            const uint32_t w = (steps << kRowChgBits) | ((my_word + (changed ? 1u : 0u)) & kRowChgMask);
            int* p = ch.prog + (size_t)tl * kProgStride;
            if (changed) red_add_release(p, (int)(w - my_word));
            else red_add_relaxed(p, (int)(w - my_word));
            my_word = w;
        }
    };

    int e = 0, epos = 0, ebase = 0;   // patch-run ordinal, its place in the current draw, the draw's ring half
    for (int slot = 0; slot < nsw; ++slot) {
        const int t = t0 + 1 + slot;
        const uint32_t sweep_s = (uint32_t)slot * SS + (AUG ? 1u : 0u);   // steps before the sweep's first class
        if constexpr (AUG) {
            // a0: the photon counts of the camera pixels centred on the tile's
            // patches, after every neighbour finished the previous sweep
            if (slot > 0) {
                bool right;
                if (service && !wait_nbrs(sweep_s - 1, sweep_s - 1, sweep_s - 1, 0, right, fence_copy) && lane == 0) s_abort = 1;
                __syncthreads();
                if (s_abort) return;
            }
            for (int q0 = 0; q0 < npt; q0 += G) {
                const int q = q0 + g;
                int pi = 0, pj = 0;
                if (q < npt) {
                    pi = pi0 + q / tw_;
                    pj = pj0 + q - (q / tw_) * tw_;
                    const double dj = phi_step_partial<float>(im, ch, pi, pj, t, lt, NT, dat_g, a.err);
                    if (lane == 0) s_phid[g][gw] = dj;
                }
                __syncthreads();
                if (q < npt && lt == 0) {
                    double tot = 0.0;
                    for (int w = 0; w < nwt; ++w) tot += s_phid[g][w];
                    ch.trace_part[(size_t)slot * im.n_patches + pi * im.npj + pj] += tot;
                }
                __syncthreads();
            }
            // the next window copies read these counts through the async proxy,
            // also where no neighbour's change would ask for the fence
            fence_copy = true;
            publish(sweep_s, true);
        }
        uint32_t row_s = sweep_s;
        for (int u = 0; u < S; ++u, row_s += (uint32_t)S) {
            for (int rn = 0; rn < RN; ++rn) {
                const int v0 = s_v0[rn], n = s_v0[rn + 1] - v0;
                bool waited = false, changed = false;
                bool right_ok = false;   // service warp: the right tile's part of this run is final and acquired
                for (int pr = 0; pr < th_; ++pr) {
                    const int pi = pi0 + pr, i = pi * S + u;
                    const bool pe = rpart && pi == im.npi - 1;
                    for (int pj = pj0 + tw_ - 1; pj >= pj0; --pj) {
                        const int sidx = (pe ? 2 : 0) | (cpart && pj == im.npj - 1 ? 1 : 0);
                        const Shape& sh = im.shape[sidx];
                        const int nv = u < sh.ph ? min(n, sh.pw - v0) : 0;   // classes of the run this patch has
                        const int j0 = pj * S + v0;
                        const int rbase = ebase + epos * VR;
                        if (!ahead) {
                            if (warp == 0) draw(e, 1, rbase);
                            __syncthreads();
                        }
                        float* rdP = red + ((e & 1) ? RS : 0);
                        float* rdS = rdP + V * nwt;
                        float* rdL = rdS + V * nwt;
                        float* rdA = rdL + V * nwt;
                        uint32_t* rdB = reinterpret_cast<uint32_t*>(rdA + G * nwt);
                        const int xb = j0 / f - (L - 1), y0 = i / f - (L - 1), dx = xb & 3;   // window of the run's first class
                        // (FINE) kernel rows and columns of a window cell: f kr + po, f kc + po - phase
                        const int po = FINE ? Le() - 1 - f * (L - 1) : 0;
                        auto copy_window = [&]() {   // one thread
                            const int x0 = xb & ~3;
                            if (fence_copy) fence_proxy_async_all();
                            mbar_arrive_expect_tx(&s_bar, (uint32_t)(AUG ? 8 : 28) * (uint32_t)(BW * L));
                            tma_load_2d(wmu, tmap, x0, y0, &s_bar);
                            if constexpr (AUG) {
                                tma_load_2d(wphi, tmap + 128, x0, y0, &s_bar);
                            } else {
                                tma_load_2d(wcum, tmap + 128, 4 * x0, y0, &s_bar);
                                tma_load_2d(wcum2, tmap + 256, 2 * x0, y0, &s_bar);
                            }
                        };
                        if (nv > 0) {
                            if (service) {
                                bool ok = true;
                                if (!waited)
                                    ok = wait_nbrs(sweep_s, row_s, row_s + (uint32_t)v0, row_s + (uint32_t)(v0 + n - 1), right_ok, fence_copy);
                                __syncwarp();
                                if (lane == 0) {
                                    if (ok) {
                                        copy_window();
                                        fence_copy = false;
                                    } else {
                                        s_abort = 1;
                                        mbar_arrive_expect_tx(&s_bar, 0);
                                    }
                                }
                                __syncwarp();
                            }
                            waited = true;
                        }
                        float2* spec_p = a.resident ? spec_s : spec_g + (pi * sz_row + pj * (pe ? sz_b : sz_f));
                        const float2* twh = tws + sh.twh_off;
                        const float2* tww = tws + sh.tww_off;
                        // entry x of the patch's spectrum tables
                        auto entry = [&](int x, int& kk, int& ll, float& wa, float& mult) {
                            if (sidx == 0) {
                                const RowEnt en = ent0[x];
                                kk = (en.kl >> 16) & 0x7fff;
                                ll = en.kl & 0xffff;
                                wa = en.wa;
                                mult = en.kl < 0 ? 2.0f : 1.0f;
                            } else {
                                const int kl = im.ent_kl[sh.ent_off + x];
                                kk = kl >> 16;
                                ll = kl & 0xffff;
                                wa = im.ent_wa32[sh.ent_off + x];
                                mult = im.ent_m32[sh.ent_off + x];
                            }
                        };
                        bool prior = true, load = nv > 0;   // this pass: score the prior; the window copy is to be awaited
                        int lo = 0;      // classes lo .. nv-1 of the run are still to be decided
                        for (;;) {
                            uint32_t bad = 0;
                            const bool mine = vb < nv && vb + VG > lo;   // this team has classes to score
                            float del[VG];
#pragma unroll
                            for (int k = 0; k < VG; ++k) del[k] = vb + k >= lo && vb + k < nv ? ring[rbase + vb + k].w : 0.0f;
                            if (mine && prior) {
                                // a4: prior changes of the team's classes, entry by entry
                                constexpr int NP = pow2_at_least(2 * VG + 1);
                                float acc[NP];
#pragma unroll
                                for (int k = 0; k < NP; ++k) acc[k] = 0.0f;
                                float2 Xn = lt < sh.nhalf ? spec_p[lt] : make_float2(0.0f, 0.0f);
                                for (int x = lt; x < sh.nhalf; x += NT) {
                                    const float2 X = Xn;
                                    if (x + NT < sh.nhalf) Xn = spec_p[x + NT];
                                    int kk, ll;
                                    float wa, mult;
                                    entry(x, kk, ll, wa, mult);
                                    const float2 eh = twh[small_mod(kk * u, sh.ph, sh.inv_ph)];
                                    int li = small_mod(ll * (v0 + vb), sh.pw, sh.inv_pw);
                                    const PriorHead hd = prior_head(X.x, X.y);
                                    acc[2 * VG] = fmaf(mult, hd.mo, acc[2 * VG]);
                                    float lg[VG];
                                    bool rare = false;
#pragma unroll
                                    for (int k = 0; k < VG; ++k) {
                                        float wr, wi;
                                        twiddle_mul(eh, tww[li], wr, wi);
                                        li += ll;
                                        li -= li >= sh.pw ? sh.pw : 0;
                                        lg[k] = prior_tail(X.x, X.y, hd, wr, wi, del[k], mult, acc[VG + k], rare);
                                    }
                                    if (rare) {   // a coefficient that shrinks by more than 1/sqrt 2, or vanishes
                                        li = small_mod(ll * (v0 + vb), sh.pw, sh.inv_pw);
#pragma unroll
                                        for (int k = 0; k < VG; ++k) {
                                            float wr, wi;
                                            twiddle_mul(eh, tww[li], wr, wi);
                                            li += ll;
                                            li -= li >= sh.pw ? sh.pw : 0;
                                            bool b = false;
                                            prior_rare(X.x, X.y, hd, wr, wi, del[k], lg[k], b);
                                            bad |= b ? 1u << k : 0u;
                                        }
                                    }
#pragma unroll
                                    for (int k = 0; k < VG; ++k) acc[k] = fmaf(wa, lg[k], acc[k]);
                                }
                                const float s = warp_sum_many<NP>(acc);
                                constexpr int sft = 5 - log2_of(NP);
                                const int vi = lane >> sft;
                                if ((lane & ((1 << sft) - 1)) == 0) {
                                    if (vi < VG) rdP[(vb + vi) * nwt + gw] = s;
                                    else if (vi < 2 * VG) rdS[(vb + vi - VG) * nwt + gw] = s;
                                    else if (vi == 2 * VG) rdA[g * nwt + gw] = s;
                                }
                                bad = __reduce_or_sync(0xffffffffu, bad);
                                if (lane == 0) rdB[g * nwt + gw] = bad;
                            }
                            if (load) {
                                load = false;
                                if (!mbar_wait(&s_bar, par, a.wait_ns)) {
                                    atomicOr(a.err, kErrTimeout);
                                    s_abort = 1;
                                }
                                par ^= 1u;
                            }
                            if (mine) {
                                // a3: likelihood changes over the windows, cell by cell
                                constexpr int NL = pow2_at_least(VG);
                                float acc[NL];
#pragma unroll
                                for (int k = 0; k < NL; ++k) acc[k] = 0.0f;
                                uint32_t badL = 0;
                                int kc = kc0, idx = idx0 + dx + (FINE ? 0 : vb);
                                int cs[FINE ? VG : 1], qo[FINE ? VG : 1], kr = FINE ? lt / L : 0;
                                if constexpr (FINE) {
#pragma unroll
                                    for (int k = 0; k < VG; ++k) {
                                        cs[k] = (j0 + vb + k) / f - j0 / f;
                                        qo[k] = po - (j0 + vb + k) % f;
                                    }
                                }
                                // box index and kernel entry (0 outside the kernel) of this cell for class k
                                auto cell = [&](int k) { return idx + (FINE ? cs[FINE ? k : 0] : k); };
                                auto kern = [&](int c, int k) -> float {
                                    if constexpr (!FINE) return Ks[c];
                                    const int p = f * kr + po - i % f, q = f * kc + qo[FINE ? k : 0];
                                    return (unsigned)p < (unsigned)im.Le && (unsigned)q < (unsigned)im.Le ? Ks[p * im.Le + q] : 0.0f;
                                };
                                for (int c = lt; c < LL; c += NT) {
                                    const float K0 = FINE ? 0.0f : Ks[c];
                                    float val[VG];
                                    bool slow = false;
#pragma unroll
                                    for (int k = 0; k < VG; ++k) {
                                        const float xk = mul_rn(del[k], FINE ? kern(c, k) : K0);
                                        if constexpr (AUG) {
                                            const float d = xk / wmu[cell(k)];
                                            val[k] = wphi[cell(k)] * log1p_small(d) - xk;
                                            slow = slow || !(fabsf(d) <= 0.05f);
                                        } else {
                                            const float d = xk * P::rcp(wmu[cell(k)]);
                                            val[k] = cgf_delta(xk, log1p_small(d), wcum[cell(k)], wcum2[cell(k)]);
                                            slow = slow || !(fabsf(d) <= 0.05f);
                                        }
                                    }
                                    if (slow) {
                                        // cells outside the frame (mu = 0: no change), and larger changes:
                                        // the library log1p, or the exact sum of Eq. 6
                                        uint32_t todo = 0;
#pragma unroll
                                        for (int k = 0; k < VG; ++k) {
                                            const float mu = wmu[cell(k)];
                                            if (!(mu > 0.0f)) val[k] = 0.0f;
                                            else todo |= 1u << k;
                                        }
                                        while (todo) {
                                            const int k = __ffs(todo) - 1;
                                            todo &= todo - 1;
                                            float dk = del[0], Kk = FINE ? kern(c, 0) : K0;
                                            int ix = cell(0);
#pragma unroll
                                            for (int z = 1; z < VG; ++z) {
                                                dk = k == z ? del[z] : dk;
                                                ix = k == z ? cell(z) : ix;
                                                if constexpr (FINE) Kk = k == z ? kern(c, z) : Kk;
                                            }
                                            const float mu = wmu[ix], xk = mul_rn(dk, Kk);
                                            float y;
                                            if constexpr (AUG) {
                                                const float d = xk / mu;
                                                if (!(d > -1.0f)) {
                                                    badL |= 1u << k;
                                                    y = 0.0f;
                                                } else {
                                                    y = wphi[ix] * log1p_cum(d) - xk;
                                                }
                                            } else {
                                                const float d = xk * P::rcp(mu);
                                                if (fabsf(d) <= kCumEval) {
                                                    y = cgf_delta(xk, log1p_cum(d), wcum[ix], wcum2[ix]);
                                                } else {
                                                    // (after a wait that failed the window is another run's, and a
                                                    // positive mu no sign that the cell lies in the frame)
                                                    const int rr = c / L, aa = y0 + rr;
                                                    const int bb = (j0 + vb + k) / f - (L - 1) + (c - rr * L);
                                                    y = 0.0f;
                                                    if ((unsigned)aa < (unsigned)im.H && (unsigned)bb < (unsigned)im.W) {
                                                        const Dat4<float> dv = dat_g[(size_t)aa * im.W + bb];
                                                        int b = 0;
                                                        y = dl_pixel_call(mu, xk, dv.c, dv.is2, dv.beta, &b);
                                                        badL |= b ? 1u << k : 0u;
                                                    }
                                                }
                                            }
#pragma unroll
                                            for (int z = 0; z < VG; ++z) val[z] = k == z ? y : val[z];
                                        }
                                    }
#pragma unroll
                                    for (int k = 0; k < VG; ++k) acc[k] += val[k];
                                    kc += dkc;
                                    idx += didx;
                                    if constexpr (FINE) kr += NT / L;
                                    if (kc >= L) {
                                        kc -= L;
                                        idx += dwrap;
                                        if constexpr (FINE) ++kr;
                                    }
                                }
                                const float s = warp_sum_many<NL>(acc);
                                constexpr int sft = 5 - log2_of(NL);
                                const int vi = lane >> sft;
                                if ((lane & ((1 << sft) - 1)) == 0 && vi < VG) rdL[(vb + vi) * nwt + gw] = s;
                                badL = __reduce_or_sync(0xffffffffu, badL);
                                if (lane == 0) rdB[(G + g) * nwt + gw] = badL;
                            }
                            // Before a run is decided the right tile must have finished its own
                            // part of it: its service lane looks once more (s_right: 0 finished
                            // and unchanged since the window was copied, 1 finished with a change,
                            // 2 not finished yet)
                            if (service) {
                                int st = 0;
                                if (nv > 0 && !right_ok && nkind == 0 && nword != nullptr) {
                                    const uint32_t w = (uint32_t)ld_relaxed(reinterpret_cast<const int*>(nword));
                                    st = (w >> kRowChgBits) < row_s + (uint32_t)(v0 + n - 1) ? 2 : (w & kRowChgMask) != nseen ? 1 : 0;
                                }
                                st = __reduce_max_sync(0xffffffffu, st);
                                if (st == 0) right_ok = true;
                                if (lane == 0) s_right = st;
                            }
                            // a5: the decisions, by the warp that finishes last, lane v for class v
                            bool last = true;
                            if (nw > 1) {
                                __syncwarp();
                                uint32_t c = 0;
                                if (lane == 0) {
                                    __threadfence_block();
                                    c = atomicAdd(&s_cnt, 1u);
                                    if (c == (uint32_t)nw - 1) {
                                        s_cnt = 0;
                                        __threadfence_block();
                                    }
                                }
                                last = __shfl_sync(0xffffffffu, c, 0) == (uint32_t)nw - 1;
                            } else {
                                __syncwarp();
                            }
                            auto decide = [&]() {
                                float dL = 0, dP = 0;
                                bool accept = false, nonfin = false;
                                if (lane >= lo && lane < nv) {
                                    const int vg = lane / VG;
                                    float sP = 0, sS = 0, sA = 0;
                                    uint32_t b = 0;
                                    for (int w = 0; w < nwt; ++w) {
                                        sP += rdP[lane * nwt + w];
                                        sS += rdS[lane * nwt + w];
                                        sA += rdA[vg * nwt + w];
                                        b |= rdB[vg * nwt + w] | rdB[(G + vg) * nwt + w];
                                        dL += rdL[lane * nwt + w];
                                    }
                                    const float4 prop = ring[rbase + lane];
                                    dP = fmaf((float)(sh.K - 1), P::log1p(sS / sA), sP);
                                    const float tot = dL + dP;
                                    const bool bd_ = (b >> (lane - vg * VG) & 1u) != 0;
                                    nonfin = !bd_ && !(fabsf(tot) <= P::kMaxFinite);
                                    accept = !bd_ && !nonfin && prop.y < tot + prop.x;
                                }
                                const uint32_t mask = __ballot_sync(0xffffffffu, accept);
                                // classes up to the first accepted one are decided
                                const int fin = mask ? __ffs(mask) - 1 : nv - 1;
                                if (lane >= lo && lane <= fin) {
                                    const int m = i * im.Wo + j0 + lane;
                                    if (nonfin) report_nonfinite(a.err, ch.chain, m, t, (double)dL, (double)dP);
                                    if (accept) {
                                        ch.trace_part[(size_t)slot * im.n_patches + pi * im.npj + pj] += (double)dL + (double)dP;
                                        rho_g[m] = ring[rbase + lane].z;
                                    }
                                    if (ch.acc_log != nullptr) ch.acc_log[(size_t)(t - 1) * im.Ho * im.Wo + m] = accept ? 1 : 0;
                                    if (ch.steps != nullptr && t <= im.burn_in) {
                                        float* sg = reinterpret_cast<float*>(ch.steps);
                                        const float sn = sg[m] * (float)im.adapt_fac[2 * (t - 1) + (accept ? 0 : 1)];
                                        sg[m] = sn < 1e-4f ? 1e-4f : sn > 4.0f ? 4.0f : sn;
                                    }
                                }
                                if (lane == 0) s_mask = mask;
                            };
                            if (last) {
                                if (s_right == 0) decide();
                                else if (lane == 0) s_mask = kUndecided;
                            }
                            __syncthreads();
                            if (s_abort) {
                                // (a copy still in flight gets one more bounded wait before
                                // the block's shared memory is released)
                                if (nv > 0) (void)mbar_wait(&s_bar, par ^ 1u, a.wait_ns);
                                return;
                            }
                            if (s_mask == kUndecided) {
                                // wait for the right tile; a change there is acquired, the window
                                // copied again and the likelihood scored again
                                __syncthreads();   // every thread has read s_mask
                                if (service) {
                                    bool ok = true, chg = false;
                                    if (nkind == 0 && nword != nullptr) {
                                        uint32_t w;
                                        ok = poll(row_s + (uint32_t)(v0 + n - 1), w);
                                        chg = ok && (w & kRowChgMask) != nseen;
                                        nseen = w & kRowChgMask;
                                    }
                                    ok = __all_sync(0xffffffffu, ok);
                                    chg = __any_sync(0xffffffffu, chg);
                                    if (chg) fence_acq_rel_gpu();
                                    fence_copy = true;
                                    __syncwarp();
                                    right_ok = true;
                                    if (!ok && lane == 0) s_abort = 1;
                                    if (ok && chg && lane == 0) copy_window();
                                    if (ok && !chg) decide();
                                }
                                __syncthreads();
                                if (s_abort) return;
                                if (s_mask == kUndecided) {
                                    prior = false;
                                    load = true;
                                    continue;
                                }
                            }
                            const uint32_t mask = s_mask;
                            if (lo == 0 && ahead && epos == 0 && warp == 0) draw(e + DP, DP, ebase ^ RH);
                            if (!mask) break;
                            // write the accepted update: window (global and staged), spectrum
                            const int fin = __ffs(mask) - 1;
                            changed = true;
                            fence_copy = true;
                            ++n_acc;
                            const float delta = ring[rbase + fin].w;
                            for (int c = tid; c < LL; c += blockDim.x) {
                                const int kr = c / L, kc = c - kr * L, xf = (j0 + fin) / f - (L - 1);
                                const int idx = kr * BW + kc + dx + (xf - xb);
                                const float old = wmu[idx];
                                if (!(old > 0.0f)) continue;   // outside the frame
                                int kw = c;
                                if constexpr (FINE) {
                                    const int p = f * kr + po - i % f, q = f * kc + po - (j0 + fin) % f;
                                    if ((unsigned)p >= (unsigned)im.Le || (unsigned)q >= (unsigned)im.Le) continue;   // outside the kernel
                                    kw = p * im.Le + q;
                                }
                                const size_t gx = (size_t)(y0 + kr) * im.mu_pitch + (xf + kc);
                                const float xk = mul_rn(delta, Ks[kw]), nmu = add_rn(old, xk);
                                __stcg(mu_g + gx, nmu);
                                wmu[idx] = nmu;
                                if constexpr (!AUG) {
                                    const float d = xk * P::rcp(old);
                                    Cum6 nq;
                                    if (fabsf(d) <= kCumShift) {
                                        nq = cgf_shift(wcum[idx], wcum2[idx], log1p_small(d));
                                    } else {
                                        const Dat4<float> dv = dat_g[(size_t)(y0 + kr) * im.W + (xf + kc)];
                                        nq = photon_cumulants_call(nmu, dv.c, dv.is2, dv.beta);
                                    }
                                    __stcg(ch.cum + gx, nq.a);
                                    __stcg(ch.cum2 + gx, nq.b);
                                    wcum[idx] = nq.a;
                                    wcum2[idx] = nq.b;
                                }
                            }
                            for (int x = tid; x < sh.nhalf; x += blockDim.x) {
                                int kk, ll;
                                float wa, mult, wr, wi;
                                entry(x, kk, ll, wa, mult);
                                twiddle_mul(twh[small_mod(kk * u, sh.ph, sh.inv_ph)],
                                            tww[small_mod(ll * (v0 + fin), sh.pw, sh.inv_pw)], wr, wi);
                                const float2 X = spec_p[x];
                                spec_p[x] = make_float2(fmaf(delta, wr, X.x), fmaf(delta, wi, X.y));
                            }
                            fence_proxy_async_all();   // before the next copy into (and of) what was written here
                            __syncthreads();
                            prior = true;
                            lo = fin + 1;
                            if (lo >= nv) break;
                        }
                        ++e;
                        if (ahead) {
                            if (++epos == DP) {
                                epos = 0;
                                ebase ^= RH;
                            }
                        } else {
                            ebase ^= RH;
                        }
                    }
                }
                publish(row_s + (uint32_t)(v0 + n), changed);
            }
        }
        // a7: after the sweep, the object into the running sums (own patches)
        // and, every sample_every-th sweep, into the kept objects
        if (t > im.burn_in) {
            const int ks = t - im.burn_in;
            const int slot_k = (ch.samples != nullptr && ks % im.sample_every == 0) ? ks / im.sample_every - 1 : -1;
            float* keep = slot_k >= 0 && slot_k < im.n_samples
                              ? reinterpret_cast<float*>(ch.samples) + (size_t)slot_k * im.Ho * im.Wo
                              : nullptr;
            const int r0 = pi0 * S, c0 = pj0 * S;
            const int nr = min(im.Ho - r0, th_ * S), nc = min(im.Wo - c0, tw_ * S);
            for (int x = tid; x < nr * nc; x += blockDim.x) {
                const int rr = x / nc;
                const size_t mm = (size_t)(r0 + rr) * im.Wo + c0 + (x - rr * nc);
                const float rv = __ldcg(rho_g + mm);
                ch.rho_sum[mm] += (double)rv;
                if (ch.rho_sq) ch.rho_sq[mm] += (double)rv * (double)rv;
                if (keep) keep[mm] = rv;
            }
        }
        if (tid == 0 && n_acc) atomicAdd(ch.acc_count + (t - 1), (unsigned long long)n_acc);
        n_acc = 0;
    }
    if (a.resident) {
        __syncthreads();
        const Shape& sh = im.shape[shape_index(im, pi0, pj0)];
        for (int x = tid; x < sh.nhalf; x += blockDim.x) spec_g[im.patch_off[pi0 * im.npj + pj0] + x] = spec_s[x];
    }
}

namespace {

template <bool AUG, bool FINE>
const void* rows_fn_of(int vg, int threads)
{
    switch (vg) {
    case 1: return (const void*)k_sweep_rows<AUG, FINE, 1, 320, 2>;
    case 4: return (const void*)k_sweep_rows<AUG, FINE, 4, 128, 5>;
    case 5: return (const void*)k_sweep_rows<AUG, FINE, 5, 128, 5>;
    default:
        return threads <= 224 ? (const void*)k_sweep_rows<AUG, FINE, 3, 224, 4> : (const void*)k_sweep_rows<AUG, FINE, 3, 256, 3>;
    }
}

// (the augmented sampler on a finer lattice keeps the general form)
const void* rows_fn(bool aug, bool fine, int vg, int threads)
{
    return aug ? rows_fn_of<true, false>(vg, threads)
               : fine ? rows_fn_of<false, true>(vg, threads) : rows_fn_of<false, false>(vg, threads);
}

}  // namespace

cudaError_t launch_sweep_rows(const SweepArgs& a, int grid, int threads, size_t smem, cudaStream_t st)
{
    SweepArgs args = a;
    void* kargs[] = {&args};
    const void* fn = rows_fn(a.aug != 0, a.fine != 0, a.row_vg, threads);
    cudaError_t e = raise_smem_limit(fn, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, kargs);
}

int rows_blocks_per_sm(bool aug, bool fine, int vg, int threads, size_t smem)
{
    const void* fn = rows_fn(aug, fine, vg, threads);
    int n = 0;
    if (raise_smem_limit(fn, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace bd
