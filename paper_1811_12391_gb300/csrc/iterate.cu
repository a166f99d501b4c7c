// Scattering-source update, FP64 reductions (residual, balance), dose tally
// and fluence extraction.
//
// Eq. 2's scattering term with the kernel as a Legendre expansion reduces, in
// moment form, to s_lm[g](v) = rho_v sum_{g'} sigma_s,l(g' -> g) phi_lm[g'](v)
// (downscatter only, self-scatter included).  The first-collision source is
// the same map applied to the uncollided moments (Sec. II.A).  Eq. 3's scalar
// fluence is the lm = 00 moment.  The dose tally multiplies the group fluence
// by group-wise conversion factors (Sec. II.A, III.A) and is accumulated in
// FP64, like the residual norm and the particle balance.
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "doctors_internal.h"

namespace doctors {

cudaError_t launch_sweep_m1_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_m4_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_m9_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_m16_entry(const SweepArgs& a, int mode, cudaStream_t s);

int sweep_chain_blocks_m1(int ab, bool ct, int threads, size_t smem);
int sweep_chain_blocks_m4(int ab, bool ct, int threads, size_t smem);
int sweep_chain_blocks_m9(int ab, bool ct, int threads, size_t smem);
int sweep_chain_blocks_m16(int ab, bool ct, int threads, size_t smem);

cudaError_t launch_sweep_flow_m1_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_flow_m4_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_flow_m9_entry(const SweepArgs& a, int mode, cudaStream_t s);
cudaError_t launch_sweep_flow_m16_entry(const SweepArgs& a, int mode, cudaStream_t s);
int sweep_flow_blocks_m1(int ab, int threads, size_t smem, bool split, bool dd);
cudaError_t launch_split_sweep_m1_entry(const SweepArgs& a, cudaStream_t s, int* count);
int sweep_flow_blocks_m4(int ab, int threads, size_t smem, bool split, bool dd);
cudaError_t launch_split_sweep_m4_entry(const SweepArgs& a, cudaStream_t s, int* count);
int sweep_flow_blocks_m9(int ab, int threads, size_t smem, bool split, bool dd);
cudaError_t launch_split_sweep_m9_entry(const SweepArgs& a, cudaStream_t s, int* count);
int sweep_flow_blocks_m16(int ab, int threads, size_t smem, bool split, bool dd);
cudaError_t launch_split_sweep_m16_entry(const SweepArgs& a, cudaStream_t s, int* count);

cudaError_t upload_tables_m1(const float* R, const float* w);
cudaError_t upload_tables_m4(const float* R, const float* w);
cudaError_t upload_tables_m9(const float* R, const float* w);
cudaError_t upload_tables_m16(const float* R, const float* w);

namespace {
std::mutex g_table_mu;
bool g_table_done[64] = {};
const int kOrders[6] = {2, 4, 6, 8, 12, 16};
}  // namespace

// The level-symmetric sets and their harmonics depend only on N, so one
// concatenated table (S2, S4, S6, S8, S12, S16) serves every problem.
cudaError_t ensure_direction_tables(int device, int N, int* base) {
    int off = 0, found = -1;
    for (int q = 0; q < 6; ++q) {
        if (kOrders[q] == N) found = off;
        off += kOrders[q] * (kOrders[q] + 2);
    }
    if (found < 0 || device < 0 || device >= 64) return cudaErrorInvalidValue;
    *base = found;
    std::lock_guard<std::mutex> lock(g_table_mu);
    if (g_table_done[device]) return cudaSuccess;
    std::vector<float> R, w;
    for (int q = 0; q < 6; ++q) {
        std::vector<double> dirs, wt;
        std::string err;
        if (!build_quadrature(kOrders[q], dirs, wt, err)) return cudaErrorInvalidValue;
        for (size_t n = 0; n < wt.size(); ++n) {
            double r[16];
            real_harmonics(3, dirs[3 * n], dirs[3 * n + 1], dirs[3 * n + 2], r);
            for (int m = 0; m < 16; ++m) R.push_back((float)r[m]);
            w.push_back((float)wt[n]);
        }
    }
    cudaError_t e = upload_tables_m1(R.data(), w.data());
    if (e == cudaSuccess) e = upload_tables_m4(R.data(), w.data());
    if (e == cudaSuccess) e = upload_tables_m9(R.data(), w.data());
    if (e == cudaSuccess) e = upload_tables_m16(R.data(), w.data());
    if (e == cudaSuccess) g_table_done[device] = true;
    return e;
}

bool sweep_supported(int ab, int M) {
    const int abs_ok[] = {1, 2, 3, 4, 5, 6, 7, 9, 10, 12};
    bool ok = false;
    for (int x : abs_ok) ok |= (x == ab);
    return ok && (M == 1 || M == 4 || M == 9 || M == 16);
}

int sweep_chain_blocks_per_sm(int ab, bool ct, int M, int threads, size_t smem) {
    switch (M) {
        case 1: return sweep_chain_blocks_m1(ab, ct, threads, smem);
        case 4: return sweep_chain_blocks_m4(ab, ct, threads, smem);
        case 9: return sweep_chain_blocks_m9(ab, ct, threads, smem);
        case 16: return sweep_chain_blocks_m16(ab, ct, threads, smem);
        default: return 0;
    }
}

int sweep_flow_blocks_per_sm(int ab, int M, int threads, size_t smem, bool split, bool dd) {
    switch (M) {
        case 1: return sweep_flow_blocks_m1(ab, threads, smem, split, dd);
        case 4: return sweep_flow_blocks_m4(ab, threads, smem, split, dd);
        case 9: return sweep_flow_blocks_m9(ab, threads, smem, split, dd);
        case 16: return sweep_flow_blocks_m16(ab, threads, smem, split, dd);
        default: return 0;
    }
}

cudaError_t launch_split_sweep(const SweepArgs& a, int M, cudaStream_t s, int* count) {
    switch (M) {
        case 1: return launch_split_sweep_m1_entry(a, s, count);
        case 4: return launch_split_sweep_m4_entry(a, s, count);
        case 9: return launch_split_sweep_m9_entry(a, s, count);
        case 16: return launch_split_sweep_m16_entry(a, s, count);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sweep_flow(const SweepArgs& a, int M, int mode, cudaStream_t s) {
    switch (M) {
        case 1: return launch_sweep_flow_m1_entry(a, mode, s);
        case 4: return launch_sweep_flow_m4_entry(a, mode, s);
        case 9: return launch_sweep_flow_m9_entry(a, mode, s);
        case 16: return launch_sweep_flow_m16_entry(a, mode, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sweep_stage(const SweepArgs& a, int M, int mode, cudaStream_t s) {
    switch (M) {
        case 1: return launch_sweep_m1_entry(a, mode, s);
        case 4: return launch_sweep_m4_entry(a, mode, s);
        case 9: return launch_sweep_m9_entry(a, mode, s);
        case 16: return launch_sweep_m16_entry(a, mode, s);
        default: return cudaErrorInvalidValue;
    }
}

namespace {

// Threads stride over (voxel, moment) pairs, moment fastest, so that a warp reads and
// writes contiguous memory.  A thread loads the moments of every source group
// it needs into registers once (all loads in flight together) and forms each
// destination group's sum from them; the group loops are unrolled up to
// GMAX (>= G) so that the moments stay in registers.  The scattering table
// is staged in shared memory when it fits.  Blocks stride over the
// (voxel, moment) range, so each stages the table once.
constexpr int kScatterThreads = 256;
constexpr size_t kScatterTableSmem = 100 * 1024;  // largest staged table

// staged table: [nmat][L+1] blocks of [GMAX (from)][GMAX (to)], so that every
// entry a thread reads is at a compile-time offset from its (material, degree)
// block; the block pitch GMAX^2 + 1 is odd, so the lanes of a warp (two voxels,
// up to eight blocks) read distinct shared-memory banks
template <int GMAX>
__host__ __device__ constexpr int scatter_block_pitch() { return GMAX * GMAX + 1; }
template <int GMAX>
size_t scatter_table_bytes(const ScatterArgs& a) {
    return (size_t)a.nmat * (a.L + 1) * scatter_block_pitch<GMAX>() * sizeof(float);
}

template <int GMAX>
__global__ void __launch_bounds__(kScatterThreads, 3) k_scatter(const ScatterCore a, int table_in_smem) {
    extern __shared__ float tab_s[];
    if (a.skip && *a.skip) return;
    const int G = a.G;
    if (table_in_smem) {
        constexpr int BP = scatter_block_pitch<GMAX>();
        const int nblk = a.nmat * (a.L + 1);
        for (int e = threadIdx.x; e < nblk * BP; e += blockDim.x) {
            const int blk = e / BP, r = e % BP, i = r / GMAX, j = r % GMAX;
            tab_s[e] = (r < GMAX * GMAX && i < G && j < G) ? __ldg(a.sigs + ((size_t)blk * G + i) * G + j) : 0.0f;
        }
        __syncthreads();
    }
    const size_t VM = a.V * a.M;
    const int g_beg = a.win ? a.win[0] : a.g0, g_end = a.win ? a.win[1] : (a.g1 > 0 ? a.g1 : G);
    // no barrier below: threads leave the grid-stride loop independently
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < VM; t += (size_t)gridDim.x * blockDim.x) {
        const size_t v = t / a.M;
        const int lm = (int)(t % a.M);
        const int l = degree_of_lm(lm_of_pos(lm, a.M));
        float ph[GMAX];
        float r = 0.0f;
        int mb = 0;
        if (a.phi) {
            mb = __ldg(a.mat + v) * (a.L + 1) + l;     // (material, degree) block of the table
            r = __ldg(a.rho + v);
            // every source group a destination group of the window needs
#pragma unroll
            for (int gp = 0; gp < GMAX; ++gp) {
                const bool need = a.transpose ? (gp >= g_beg && gp < G) : (gp < g_end);
                ph[gp] = need ? __ldg(a.phi + gp * VM + t) : 0.0f;
            }
        }
        // the fixed source of every destination group, also loaded up front
        float qb[GMAX];
#pragma unroll
        for (int g = 0; g < GMAX; ++g) qb[g] = (a.base && g >= g_beg && g < g_end) ? __ldg(a.base + g * VM + t) : 0.0f;
        const float* ts = tab_s + (size_t)mb * scatter_block_pitch<GMAX>();
        const float* tg = a.sigs + (size_t)mb * G * G;
#pragma unroll
        for (int g = 0; g < GMAX; ++g) {
            if (g < g_beg || g >= g_end) continue;
            float out = qb[g];
            if (lm == 0) {
                if (a.iso) out += __ldg(a.iso + g);
                if (a.iso_field) out += a.iso_field_scale * __ldg(a.iso_field + (size_t)g * a.V + v);
            }
            if (a.phi) {
                float acc = 0.0f;
                if (!a.transpose) {
                    // downscatter: g' <= g
                    if (table_in_smem) {
#pragma unroll
                        for (int gp = 0; gp <= g; ++gp) acc = fmaf(ts[gp * GMAX + g], ph[gp], acc);
                    } else {
#pragma unroll
                        for (int gp = 0; gp <= g; ++gp) acc = fmaf(__ldg(tg + gp * G + g), ph[gp], acc);
                    }
                } else {
                    // adjoint: g' >= g (zero padding beyond G in the staged table)
                    if (table_in_smem) {
#pragma unroll
                        for (int gp = g; gp < GMAX; ++gp) acc = fmaf(ts[g * GMAX + gp], ph[gp], acc);
                    } else {
#pragma unroll
                        for (int gp = g; gp < GMAX; ++gp)
                            if (gp < G) acc = fmaf(__ldg(tg + g * G + gp), ph[gp], acc);
                    }
                }
                out = fmaf(r, acc, out);
            }
            a.out[g * VM + t] = out;
        }
    }
}

// The iteration's form of the same map (a scattering term, no per-voxel
// isotropic field, fewer than 2^31 entries) with no branch in its group
// loops (ISO: the first-collision form, with the volume sources' isotropic
// term and no fixed source, added to the l = 0 entries): the
// direction of the sum (downscatter or its transpose) and the presence of a
// fixed source are template parameters, the group window only predicates the
// loads of the fixed source and the stores, and entry indices are 32-bit.  The
// inner sums are those of k_scatter term by term, so the two kernels give
// identical results.  Every source group below G is needed by some group of
// the window (the forward window only retires leading groups, the adjoint
// window trailing ones), so all G source moments are loaded; padding groups up
// to GMAX read group G-1's row again and are zeroed.
__device__ __forceinline__ float ldg_if(const float* p, bool pred) {
    float x = 0.0f;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.f32 %0, [%1];\n\t}"
        : "+f"(x)
        : "l"(p), "r"((unsigned)pred));
    return x;
}

// staged table of k_scatter_fast: per (material, degree) block GMAX rows of
// GMAX entries, row g holding the entries destination group g sums over in
// ascending source order (forward: sigma(g' -> g) for g' = 0..GMAX-1, the
// table's column g; adjoint: sigma(g -> g'), its row g), so that a thread
// reads them as 16-byte vectors.  The block pitch GMAX^2 + 4 is 4 or 20 mod
// 32 words for every GMAX used, so eight consecutive blocks (the degrees of
// two voxels of neighbouring materials, as one warp reads them) start in
// distinct 16-byte bank groups.
template <int GMAX>
__host__ __device__ constexpr int scatter_fast_pitch() { return GMAX * GMAX + 4; }
template <int GMAX>
size_t scatter_fast_table_bytes(const ScatterArgs& a) {
    return (size_t)a.nmat * (a.L + 1) * scatter_fast_pitch<GMAX>() * sizeof(float);
}

template <int GMAX, bool TR, bool HAS_BASE, bool ISO = false, bool ZERO = false>
__global__ void __launch_bounds__(kScatterThreads, GMAX <= 24 ? 2 : 1) k_scatter_fast(const std::conditional_t<ZERO, ScatterArgs, ScatterCore> a) {
    extern __shared__ float4 tab4_s[];
    float* tab_s = reinterpret_cast<float*>(tab4_s);
    static_assert(GMAX % 4 == 0, "rows of whole 16-byte vectors");
    if (a.skip && *a.skip) return;
    const int G = a.G;
    constexpr int BP = scatter_fast_pitch<GMAX>();
    const int nblk = a.nmat * (a.L + 1);
    for (int e = threadIdx.x; e < nblk * BP; e += blockDim.x) {
        const int blk = e / BP, r = e % BP, i = r / GMAX, j = r % GMAX;   // row i, entry j
        const int from = TR ? i : j, to = TR ? j : i;
        tab_s[e] = (r < GMAX * GMAX && i < G && j < G) ? __ldg(a.sigs + ((size_t)blk * G + from) * G + to) : 0.0f;
    }
    __syncthreads();
    const unsigned VM = (unsigned)(a.V * a.M), M = (unsigned)a.M;
    const int g_beg = a.win ? a.win[0] : a.g0, g_end = a.win ? a.win[1] : (a.g1 > 0 ? a.g1 : G);
    int z_beg = 0, z_end = 0;
    if constexpr (ZERO) {
        z_beg = a.zero_win[0];
        z_end = a.zero_win[1];
        if (blockIdx.x == 0) {
            for (int g = threadIdx.x; g < 2 * G; g += blockDim.x) a.zero_red[G + g] = 0.0;
            for (int g = z_beg + threadIdx.x; g < z_end; g += blockDim.x) a.zero_red[g] = 0.0;
        }
    }
    const int L1 = a.L + 1;
    // no barrier below: threads leave the grid-stride loop independently
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < VM; t += gridDim.x * blockDim.x) {
        const unsigned v = t / M;
        const int lm = (int)(t - v * M);
        const int mb = __ldg(a.mat + v) * L1 + degree_of_lm(lm_of_pos(lm, (int)M));
        const float r = __ldg(a.rho + v);
        float ph[GMAX];
        const float* pp = a.phi + t;
#pragma unroll
        for (int gp = 0; gp < GMAX; ++gp) {
            float x;
            if constexpr (ZERO) x = pp[(size_t)(gp < G ? gp : G - 1) * VM];
            else x = __ldg(pp + (size_t)(gp < G ? gp : G - 1) * VM);
            ph[gp] = gp < G ? x : 0.0f;
        }
        if constexpr (ZERO) {
            // read by no other thread: ready for the next sweep to add to
            float* pz = a.zero_mom + t;
#pragma unroll
            for (int gp = 0; gp < GMAX; ++gp)
                if (gp >= z_beg && gp < z_end) pz[(size_t)gp * VM] = 0.0f;
        }
        float qb[GMAX];
        const float* pb = a.base + t;
#pragma unroll
        for (int g = 0; g < GMAX; ++g) qb[g] = HAS_BASE ? ldg_if(pb + (size_t)g * VM, g >= g_beg && g < g_end) : 0.0f;
        if (ISO && lm == 0) {
#pragma unroll
            for (int g = 0; g < GMAX; ++g)
                if (g < G) qb[g] += __ldg(a.iso + g);
        }
        const float4* ts4 = reinterpret_cast<const float4*>(tab_s + mb * BP);
        float* po = a.out + t;
#pragma unroll
        for (int g = 0; g < GMAX; ++g) {
            // the same sums as k_scatter, source groups ascending: forward
            // g' = 0..g, adjoint g' = g..GMAX-1, read four entries at a time
            float acc = 0.0f;
            constexpr int R4 = GMAX / 4;
#pragma unroll
            for (int c = TR ? g / 4 : 0; c < (TR ? R4 : g / 4 + 1); ++c) {
                const float4 t4 = ts4[g * R4 + c];
                const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int gp = 4 * c + k;
                    if (TR ? gp >= g : gp <= g) acc = fmaf(tv[k], ph[gp], acc);
                }
            }
            const float out = fmaf(r, acc, qb[g]);
            if (g >= g_beg && g < g_end) po[(size_t)g * VM] = out;
        }
    }
}

// Update a live instance's iteration count and residual (max over groups of
// sqrt(sum (dphi)^2 / sum phi^2)), retire it when the relative change is below
// its tolerance or not finite or the cap is reached, else shrink its active group window: a
// group whose relative change is below tol and whose sources are all final is
// final too (forward: leading groups, adjoint: trailing groups).  One warp; its
// lanes form the changes of groups lane and lane + 32.
__device__ void advance_loop(LoopCtl& c) {
    static_assert(kMaxG <= 64, "two groups per lane");
    const int lane = threadIdx.x & 31;
    double e[2];
    unsigned below[2];
    bool nan = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int g = lane + 32 * h;
        double num = 0.0, den = 0.0;
        if (g < c.G) {
            num = __ldcg(c.res + 2 * g);
            den = __ldcg(c.res + 2 * g + 1);
        }
        e[h] = den == 0.0 ? 0.0 : sqrt(num / den);       // NaN sums stay NaN
        nan = nan || e[h] != e[h];
        below[h] = __ballot_sync(0xffffffffu, e[h] < c.tol);
    }
    double eps = e[1] > e[0] ? e[1] : e[0];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_xor_sync(0xffffffffu, eps, off);
        eps = o > eps ? o : eps;
    }
    if (__any_sync(0xffffffffu, nan)) eps = __longlong_as_double(0x7ff8000000000000LL);
    if (lane != 0) return;
    c.iters += 1;
    c.resid = eps;
    c.group_sweeps += c.use_window ? c.win[1] - c.win[0] : c.G;
    c.swept[0] = c.win[0];
    c.swept[1] = c.win[1];
    if (eps < c.tol || c.iters >= c.max_iters || !isfinite(eps)) {
        c.done = 1;
    } else if (c.use_window) {
        auto final_group = [&](int g) { return (below[g >> 5] >> (g & 31)) & 1u; };
        if (!c.reverse)
            while (c.win[0] < c.win[1] - 1 && final_group(c.win[0])) ++c.win[0];
        else
            while (c.win[1] - 1 > c.win[0] && final_group(c.win[1] - 1)) --c.win[1];
    }
}

// The adjoint's fixed source: scale * field in the l = 0 moment, nothing else
// (one 16-byte store per thread and pass; M = 1, 9: one entry).  Floor: the
// moments written once, 25 us at 19 groups x 64x64x32, P3; the general kernel,
// which loops over groups per entry, takes 231 us.
template <int VEC>
__global__ void __launch_bounds__(256) k_iso_source(size_t GV, int M, const float* field, float scale, float* out) {
    const unsigned per = (unsigned)M / VEC;              // vectors per record
    const size_t n = GV * per;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x) {
        const size_t e = t / per;
        const float x = t - e * per == 0 ? scale * __ldg(field + e) : 0.0f;
        if constexpr (VEC == 4) reinterpret_cast<float4*>(out)[t] = make_float4(x, 0.0f, 0.0f, 0.0f);
        else out[t] = x;
    }
}

template <int NV>
__device__ __forceinline__ void block_reduce_add(double (&x)[NV], double* dst) {
    __shared__ double red[NV][32];
#pragma unroll
    for (int q = 0; q < NV; ++q)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x[q] += __shfl_down_sync(0xffffffffu, x[q], off);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) red[q][wid] = x[q];
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            double y = lane < nw ? red[q][lane] : 0.0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) y += __shfl_down_sync(0xffffffffu, y, off);
            if (lane == 0 && y != 0.0) atomicAdd(dst + q, y);
        }
    }
}

// grid: (blocks over V, G).  The four elements of one pass are differenced
// and squared in FP32 (a relative error near 1e-7 in a convergence norm that
// is compared against tolerances of 1e-6 and above); the passes, the threads
// and the blocks are summed in FP64, so that few FP64 operations are issued:
// their rate on this part is a small fraction of the FP32 rate.
// rho sigma_t of every cell and group, the product the sweep would form per cell step
__global__ void __launch_bounds__(256) k_total_xs(size_t V, int G, const uint8_t* mat, const float* rho,
                                                  const float* sigt, float* out) {
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x) {
        const float r = rho ? rho[v] : 1.0f;
        const int m = mat[v];
        for (int g = 0; g < G; ++g) out[(size_t)g * V + v] = r * __ldg(sigt + m * G + g);
    }
}

// loop: the last block also advances the loop and leaves a copy of its state in pinned host memory.
__global__ void __launch_bounds__(256) k_residual(size_t V, int M, const float* mom, float* prev,
                                                  double* res, const int* skip, int g0, const int* win,
                                                  LoopCtl* loop, LoopCtl* host_copy) {
    if (skip && *skip) return;
    const int g = g0 + blockIdx.y;
    if (win && (g < win[0] || g >= win[1])) {            // retired group (whole block)
        if (!loop) return;
        V = 0;
    }
    double x[2] = {0.0, 0.0};
    // four voxels per thread and pass, their loads issued together
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t v0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v0 < V; v0 += 4 * stride) {
        float cur[4], old[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const size_t v = v0 + u * stride;
            cur[u] = v < V ? mom[((size_t)g * V + v) * M] : 0.0f;
            old[u] = v < V ? prev[(size_t)g * V + v] : 0.0f;
        }
        float dd = 0.0f, cc = 0.0f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const size_t v = v0 + u * stride;
            if (v < V) {
                const float d = cur[u] - old[u];
                dd = fmaf(d, d, dd);
                cc = fmaf(cur[u], cur[u], cc);
                prev[(size_t)g * V + v] = cur[u];
            }
        }
        x[0] += (double)dd;
        x[1] += (double)cc;
    }
    block_reduce_add<2>(x, res + 2 * g);
    if (loop && threadIdx.x < 32) {
        __threadfence();                                 // this block's sums before its arrival
        unsigned before = 0;
        if (threadIdx.x == 0) before = atomicAdd(&loop->arrived, 1u);
        before = __shfl_sync(0xffffffffu, before, 0);
        if (before == gridDim.x * gridDim.y - 1) {
            __threadfence();
            advance_loop(*loop);
            __syncwarp();
            if (threadIdx.x == 0) {
                loop->arrived = 0;
                *host_copy = *loop;
                __threadfence_system();
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_balance(size_t V, int G, int M, const uint8_t* mat,
                                                 const float* rho, const float* sigt, const float* src,
                                                 const float* mom, double vol, double* bal) {
    const int g = blockIdx.y;
    double x[2] = {0.0, 0.0};
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (size_t)gridDim.x * blockDim.x) {
        const double s00 = src[((size_t)g * V + v) * M];
        const double p00 = mom[((size_t)g * V + v) * M];
        const double st = (double)rho[v] * (double)sigt[mat[v] * G + g];
        x[0] += vol * s00;
        x[1] += vol * st * p00;
    }
    block_reduce_add<2>(x, bal + 2 * g);
}

__global__ void __launch_bounds__(256) k_dose(size_t V, int G, int M, const uint8_t* mat, const float* rho,
                                              const double* k, const float* phi_u, const float* mom,
                                              double* dose) {
    const size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    const int m = mat[v];
    double acc = 0.0;
    for (int g = 0; g < G; ++g) {
        const double phi = (double)phi_u[(size_t)g * V + v] + (double)mom[((size_t)g * V + v) * M];
        acc += k[m * G + g] * phi;
    }
    dose[v] = acc * (double)rho[v];
}

__global__ void __launch_bounds__(256) k_extract(size_t V, int G, int M, int which, const float* phi_u,
                                                 const float* mom, float* out) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= V * G) return;
    float x = 0.0f;
    if (which & 1) x += phi_u[t];
    if (which & 2) x += mom[t * M];
    out[t] = x;
}

template <class T>
__global__ void __launch_bounds__(256) k_zero(T* p, size_t n, const int* skip) {
    if (skip && *skip) return;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        p[t] = T(0);
}

// One warp: advance every live instance and stop the graph's while loop once
// all instances are retired.
__global__ void __launch_bounds__(32) k_decide(LoopCtl* ctl, int n, cudaGraphConditionalHandle h) {
    bool all = true;
    for (int q = 0; q < n; ++q) {
        const bool live = !ctl[q].done;
        __syncwarp();
        if (live) advance_loop(ctl[q]);
        __syncwarp();
        all = all && ctl[q].done;
    }
    if (all && threadIdx.x == 0) cudaGraphSetConditional(h, 0);
}

// The window's moments and leakage and every residual sum to zero, in one
// launch (per_group = V * M floats)
__global__ void __launch_bounds__(256) k_zero_iteration(float* mom, size_t per_group, double* red, int G, const int* win,
                                                        const int* skip) {
    if (skip && *skip) return;
    const int g0 = win[0], g1 = win[1];
    const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const size_t beg = (size_t)g0 * per_group, end = (size_t)g1 * per_group;
    // whole 16-byte vectors, then the unaligned ends
    const size_t b4 = (beg + 3) / 4, e4 = end / 4;
    float4* m4 = reinterpret_cast<float4*>(mom);
    for (size_t t = b4 + first; t < e4; t += stride) m4[t] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (first < 4) {
        if (beg + first < 4 * b4 && beg + first < end) mom[beg + first] = 0.0f;
        if (4 * e4 + first < end && 4 * e4 >= beg) mom[4 * e4 + first] = 0.0f;
    }
    for (size_t g = first; g < (size_t)(2 * G); g += stride) red[G + g] = 0.0;
    for (size_t g = g0 + first; g < (size_t)g1; g += stride) red[g] = 0.0;
}

template <class T>
__global__ void __launch_bounds__(256) k_zero_window(T* p, size_t per_group, const int* win, const int* skip) {
    if (skip && *skip) return;
    const size_t beg = (size_t)win[0] * per_group, end = (size_t)win[1] * per_group;
    for (size_t t = beg + (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < end; t += (size_t)gridDim.x * blockDim.x)
        p[t] = T(0);
}

unsigned blocks_for(size_t n, int bs, unsigned cap = 0) {
    size_t b = (n + bs - 1) / bs;
    if (cap && b > cap) b = cap;
    return (unsigned)(b ? b : 1);
}

}  // namespace

// one resident wave of k_scatter_fast
template <int GMAX, bool TR, bool HAS_BASE, bool ISO = false, bool ZERO = false>
cudaError_t launch_scatter_fast(const ScatterArgs& a, size_t smem, cudaStream_t s) {
    auto kern = k_scatter_fast<GMAX, TR, HAS_BASE, ISO, ZERO>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int nb = 0, dev = 0, nsm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kScatterThreads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const unsigned grid = blocks_for(a.V * a.M, kScatterThreads, (unsigned)(nsm * (nb > 0 ? nb : 1)));
    kern<<<grid, kScatterThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int GMAX>
cudaError_t launch_scatter_g(const ScatterArgs& a, cudaStream_t s, int* count) {
    const size_t tab_bytes = scatter_table_bytes<GMAX>(a);
    const int staged = tab_bytes <= kScatterTableSmem ? 1 : 0;
    const size_t smem = staged ? tab_bytes : 0;
    const size_t fast_bytes = scatter_fast_table_bytes<GMAX>(a);
    const bool fast = fast_bytes <= kScatterTableSmem && a.phi && !a.iso_field && a.V * a.M < ((size_t)1 << 31);
    if (fast && a.iso && !a.transpose && !a.base)
        return launch_scatter_fast<GMAX, false, false, true>(a, fast_bytes, s);
    if (a.zero_mom) {
        // small moment arrays: zeroed by the threads that have read them, one launch
        // fewer (16^3 cube, S4 P1: 0.86 -> 0.74 ms per solve together with the
        // residual's last block deciding the loop); large ones in a launch of their
        // own, which streams the stores (cylinder S8 P3, 160 MB: 16.5 ms against 17.2)
        const bool small = a.V * a.M * a.G * sizeof(float) <= ((size_t)24 << 20);
        if (small && fast && !a.iso && a.base)
            return a.transpose ? launch_scatter_fast<GMAX, true, true, false, true>(a, fast_bytes, s)
                               : launch_scatter_fast<GMAX, false, true, false, true>(a, fast_bytes, s);
        ScatterArgs b = a;
        b.zero_mom = nullptr;
        cudaError_t e = launch_scatter_g<GMAX>(b, s, nullptr);
        if (e != cudaSuccess) return e;
        if (count) *count = 2;
        k_zero_iteration<<<blocks_for((a.V * a.M * a.G + 15) / 16, 256, 152 * 8), 256, 0, s>>>(
            a.zero_mom, a.V * a.M, a.zero_red, a.G, a.zero_win, a.skip);
        return cudaGetLastError();
    }
    if (fast && !a.iso) {
        if (a.transpose)
            return a.base ? launch_scatter_fast<GMAX, true, true>(a, fast_bytes, s)
                          : launch_scatter_fast<GMAX, true, false>(a, fast_bytes, s);
        return a.base ? launch_scatter_fast<GMAX, false, true>(a, fast_bytes, s)
                      : launch_scatter_fast<GMAX, false, false>(a, fast_bytes, s);
    }
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_scatter<GMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_scatter<GMAX><<<blocks_for(a.V * a.M, kScatterThreads, 152 * 8), kScatterThreads, smem, s>>>(a, staged);
    return cudaGetLastError();
}

cudaError_t launch_scatter(const ScatterArgs& a, cudaStream_t s, int* count) {
    if (count) *count = 1;
    if (!a.phi && !a.base && !a.iso && a.iso_field && !a.skip && !a.win && a.g0 == 0 && (a.g1 == 0 || a.g1 == a.G)) {
        const size_t GV = (size_t)a.G * a.V;
        if (a.M % 4 == 0)
            k_iso_source<4><<<blocks_for(GV * a.M / 4, 256, 152 * 16), 256, 0, s>>>(GV, a.M, a.iso_field, a.iso_field_scale, a.out);
        else
            k_iso_source<1><<<blocks_for(GV * a.M, 256, 152 * 16), 256, 0, s>>>(GV, a.M, a.iso_field, a.iso_field_scale, a.out);
        return cudaGetLastError();
    }
    if (a.G <= 8) return launch_scatter_g<8>(a, s, count);
    if (a.G <= 16) return launch_scatter_g<16>(a, s, count);
    if (a.G <= 20) return launch_scatter_g<20>(a, s, count);
    if (a.G <= 24) return launch_scatter_g<24>(a, s, count);
    if (a.G <= 32) return launch_scatter_g<32>(a, s, count);
    if (a.G <= 64) return launch_scatter_g<64>(a, s, count);
    return cudaErrorInvalidValue;
}

cudaError_t launch_residual(size_t V, int G, int M, const float* mom, float* prev, double* res,
                            cudaStream_t s, const int* skip, int g0, int gcount, const int* win, LoopCtl* loop,
                            LoopCtl* host_copy) {
    // sixteen voxels per thread (four passes)
    dim3 grid(blocks_for((V + 15) / 16, 256, 152), gcount < 0 ? G : gcount);
    k_residual<<<grid, 256, 0, s>>>(V, M, mom, prev, res, skip, g0, win, loop, host_copy);
    return cudaGetLastError();
}

cudaError_t launch_total_xs(size_t V, int G, const uint8_t* mat, const float* rho, const float* sigt, float* out,
                            cudaStream_t s) {
    k_total_xs<<<blocks_for(V, 256, 152 * 16), 256, 0, s>>>(V, G, mat, rho, sigt, out);
    return cudaGetLastError();
}

cudaError_t launch_zero_window(float* p, size_t per_group, int G, const int* win, const int* skip, cudaStream_t s) {
    k_zero_window<float><<<blocks_for((per_group * G + 3) / 4, 256, 152 * 16), 256, 0, s>>>(p, per_group, win, skip);
    return cudaGetLastError();
}

cudaError_t launch_zero_window(double* p, size_t per_group, int G, const int* win, const int* skip, cudaStream_t s) {
    k_zero_window<double><<<blocks_for((per_group * G + 3) / 4, 256, 152 * 16), 256, 0, s>>>(p, per_group, win, skip);
    return cudaGetLastError();
}

cudaError_t launch_zero(float* p, size_t n, const int* skip, cudaStream_t s) {
    k_zero<float><<<blocks_for((n + 3) / 4, 256, 152 * 16), 256, 0, s>>>(p, n, skip);
    return cudaGetLastError();
}

cudaError_t launch_zero(double* p, size_t n, const int* skip, cudaStream_t s) {
    k_zero<double><<<blocks_for((n + 3) / 4, 256, 152 * 16), 256, 0, s>>>(p, n, skip);
    return cudaGetLastError();
}

cudaError_t launch_decide(LoopCtl* ctl, int n, unsigned long long cond_handle, cudaStream_t s) {
    k_decide<<<1, 32, 0, s>>>(ctl, n, (cudaGraphConditionalHandle)cond_handle);
    return cudaGetLastError();
}

cudaError_t launch_balance(size_t V, int G, int M, const uint8_t* mat, const float* rho, const float* sigt,
                           const float* src, const float* mom, double vol, double* bal, cudaStream_t s) {
    dim3 grid(blocks_for(V, 256, 296), G);
    k_balance<<<grid, 256, 0, s>>>(V, G, M, mat, rho, sigt, src, mom, vol, bal);
    return cudaGetLastError();
}

cudaError_t launch_dose(size_t V, int G, int M, const uint8_t* mat, const float* rho, const double* k,
                        const float* phi_u, const float* mom, double* dose, cudaStream_t s) {
    k_dose<<<blocks_for(V, 256), 256, 0, s>>>(V, G, M, mat, rho, k, phi_u, mom, dose);
    return cudaGetLastError();
}

cudaError_t launch_extract(size_t V, int G, int M, int which, const float* phi_u, const float* mom,
                           float* out, cudaStream_t s) {
    k_extract<<<blocks_for(V * G, 256), 256, 0, s>>>(V, G, M, which, phi_u, mom, out);
    return cudaGetLastError();
}

}  // namespace doctors
