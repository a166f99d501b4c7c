// Dataflow octant wavefront sweep: the step-differenced cell update of
// k_sweep_chain (whole octants per CTA; the first octant's direction rows,
// coefficients and moment tables are kernel parameters, read through the
// constant bank at compile-time offsets) with the tile stages replaced by a
// task queue in one launch.  S12 and S16 run as whole octants (21 and 36
// directions per cell step); S16 also as three launches, one per block of
// 12 directions of every octant, each with that block's table.
//
// The tasks (tile, octant, group) are numbered stage by stage (the tile
// diagonal of the octant's reflected tile grid).  Each CTA takes the next
// task from a global counter, sweeps it through its hyperplane pipeline and
// takes another, until the queue is empty; there is one launch per sweep and
// no barrier between stages.  A task needs the fluxes leaving its upstream
// x and y tiles, which other CTAs may still be producing: every face record
// (the AB fluxes of one column face and plane) starts the sweep as NaN, the
// producer overwrites it with the fluxes, and the consumer's face warp (one
// more warp per CTA; the column threads run no face code) fetches it a few
// steps ahead with cp.async (L2, not L1), reads it again while any value is
// still NaN, moves it into the halo of the plane buffers and writes NaN back,
// so the face buffers are ready for the next sweep without a reset pass.
//
// Waiting is bounded and cannot deadlock: a CTA holds the task it sweeps and
// at most one later task, taken a few steps before the first ends.  It waits
// only on tasks with smaller numbers than the one it sweeps, so the lowest
// unfinished task is always being swept and waits on nothing unfinished.  A
// wait that exceeds kFlowSpinLimit polls records the failure in the problem's
// flag word, uses zero fluxes and goes on (later waits of the sweep then give
// up at once); the host turns the flag into DOCTORS_ERR_TIMEOUT and resets
// the buffers.
//
// What bounds it, and the layout taken for that (water cylinder 64x64x32, S8
// P3, 19 groups, 8x8 tiles, one full sweep):
//   * with one 64-byte record (the 16 moments of a cell) per thread, each of
//     its quarters went out as its own request: 191 M L2 requests a sweep, L1
//     request port 65 % and L2 tags 64 % busy, and 59 M of the 110 M
//     shared-memory wavefronts were bank conflicts (64-byte slots read as
//     16-byte vectors).  Now four lanes move one record (one request of two
//     full sectors): 75 M requests; the slots are swizzled, the plane records
//     are read and written as vectors.  1.04 -> 0.81 ms (all groups active, under
//     ncu; 0.97 -> 0.76 on average over a solve).
//   * source records, cross sections and face records are fetched up to four
//     steps ahead into shared memory (SweepArgs::depth), for every number of
//     moments; the step no longer ends with a wait for L2.  The paper's coarse
//     mesh (64x64x16, S6 P0, 7 groups), whose 144 dependent steps are latency:
//     0.222 -> 0.100 ms per sweep; the 16^3 cube, S4 P1: 46 -> 25 us.
//   * the task queue's counter is read ahead and the boundary current is added
//     once per task (it was a shared-memory FP64 addition per finishing column
//     between two steps: 0.386 -> 0.297 ms for the twelve sweeps of the cube).
//   * the register bound follows the tile (template NT): with one bound for
//     CTAs of 288 threads (96 registers) the cooperative addresses spilled in
//     the 8x8 tile too (0.748 against 0.703 ms; six CTAs of 96 registers spill
//     and take 0.930, four of up to 168 take 0.742).
// Together, average over a solve: cylinder 0.97 -> 0.68 ms per sweep, diamond 0.77;
// the abdomen (128x128x48, S16 P3, 19 groups) 12.0 -> 10.0.  A P3 step is bound by
// the issue of its instructions (about a quarter of them packed FMAs), a P0 or P1
// step on a small mesh by the latency of its chain.
#pragma once

#include <algorithm>

#include "sweep_chain.cuh"

namespace doctors {

constexpr int kFlowSpinLimit = 1 << 19;
constexpr int kFlowMinCtas = 5;

// floats per face record: AB fluxes padded to a multiple of 4 (16-byte copies)
__host__ __device__ constexpr int flow_abp(int ab) { return (ab + 3) & ~3; }

__device__ __forceinline__ void cp_async_cg16(void* dst_smem, const void* src_gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(dst_smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src_gmem) : "memory");
}

// the hyperplane step's barrier of the column warps and the face warp (reached
// from two places)
__device__ __forceinline__ void flow_step_barrier() {
    asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
}

// 16 bytes another CTA may be writing (each word is checked by itself)
__device__ __forceinline__ float4 ld_relaxed4(const float* p) {
    float4 t;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "l"(p) : "memory");
    return t;
}

__device__ __forceinline__ void red_add_v4(float* p, float4 t) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(p), "f"(t.x), "f"(t.y), "f"(t.z), "f"(t.w)
                 : "memory");
}

// PW floats of a plane record as one shared-memory access
template <int PW>
__device__ __forceinline__ void plane_load(const float* p, float (&x)[PW]) {
    if constexpr (PW == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
    } else if constexpr (PW == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        x[0] = t.x; x[1] = t.y;
    } else {
        x[0] = p[0];
    }
}
template <int PW>
__device__ __forceinline__ void plane_store_w(float* p, const float* x) {
    if constexpr (PW == 4) *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
    else if constexpr (PW == 2) *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
    else p[0] = x[0];
}
// a whole plane record
template <int AB>
__device__ __forceinline__ void plane_store(float* p, const float (&v)[flow_abp(AB)]) {
#pragma unroll
    for (int q = 0; q < flow_rs(AB); q += flow_pw(AB)) plane_store_w<flow_pw(AB)>(p + q, v + q);
}
// a face or angular record in global memory: AB fluxes, zero padding
template <int AB>
__device__ __forceinline__ void store_record(float* p, const float (&v)[AB]) {
    float4* dst = reinterpret_cast<float4*>(p);
#pragma unroll
    for (int c4 = 0; c4 < flow_abp(AB) / 4; ++c4)
        dst[c4] = make_float4(4 * c4 < AB ? v[4 * c4 < AB ? 4 * c4 : 0] : 0.0f,
                              4 * c4 + 1 < AB ? v[4 * c4 + 1 < AB ? 4 * c4 + 1 : 0] : 0.0f,
                              4 * c4 + 2 < AB ? v[4 * c4 + 2 < AB ? 4 * c4 + 2 : 0] : 0.0f,
                              4 * c4 + 3 < AB ? v[4 * c4 + 3 < AB ? 4 * c4 + 3 : 0] : 0.0f);
}

// sum of N products, two at a time: the two lanes of packed operations (even
// and odd terms), and their sum.  FP64 results of a solve (J, the view weights)
// show this order in their tenth digit: sums of a pair of directions and their
// differences (the harmonics are even or odd under x <-> y) need fewer terms, but
// moved them by up to 1e-8 and were taken back (with them a sweep of the cylinder
// took 4 % less, a S16 P3 solve of 96x80x24 22.7 ms instead of 28.1)
template <int N>
__device__ __forceinline__ float2 dot2(const float* c, const float* x) {
    float2 t = N == 1 ? make_float2(c[0] * x[0], 0.0f) : make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k + 1 < N; k += 2) t = __ffma2_rn(make_float2(c[k], c[k + 1]), make_float2(x[k], x[k + 1]), t);
    if constexpr (N % 2 == 1 && N > 1) t.x = fmaf(c[N - 1], x[N - 1], t.x);
    return t;
}
template <int N>
__device__ __forceinline__ float dot(const float* c, const float* x) {
    if constexpr (N == 1) return c[0] * x[0];
    const float2 t = dot2<N>(c, x);
    return t.x + t.y;
}

// column (li, lj) of column thread t: the tile's columns in diagonal order
__device__ __forceinline__ void flow_column(int t, int tx, int ty, int& li, int& lj) {
    int base = 0;
    for (int dd = 0; dd <= tx + ty - 2; ++dd) {
        const int lo = dd > ty - 1 ? dd - (ty - 1) : 0;
        const int hi = dd < tx - 1 ? dd : tx - 1;
        const int cnt = hi - lo + 1;
        if (t < base + cnt) {
            li = lo + (t - base);
            lj = dd - li;
            return;
        }
        base += cnt;
    }
}

// place of plane k's face record in its column's run of nz.  The 16-byte records
// of S2 and S4 lie two to a 32-byte sector, and one that shares its sector with
// the one its producer writes next is slow to read: so the first and the second
// half of the planes take the sectors' halves in turn, and a sector's two records
// are nz / 2 steps apart
template <int AB>
__device__ __forceinline__ int flow_face_slot(int k, int nz) {
    if constexpr (flow_abp(AB) > 4) return k;
    const int half = (nz + 1) >> 1;
    return k < half ? 2 * k : 2 * (k - half) + 1;
}

// tiles of stage s of an ntx x nty tile grid
__device__ __forceinline__ int flow_stage_tiles(int s, int ntx, int nty) {
    const int lo = s - (nty - 1) > 0 ? s - (nty - 1) : 0;
    const int hi = s < ntx - 1 ? s : ntx - 1;
    return hi - lo + 1;
}

// SPLIT = true: the transforms run in separate passes (k_split_m2d before,
// k_split_d2m after); the sweep reads each cell's angular-source record
// a.qang and writes its angular-fluence record a.pang, with no moments and
// no reductions (mode 0 only).
//
// DD = true: diamond differencing (no negative-flux fixup).  The direction
// table then holds 2 c_x, 2 c_y, 2 c_z and their sum, so the cell solve
// (q + sum 2 c psi_in) / (sigma + 2 sum c) is the step formula's; each face
// leaves with 2 psi - psi_in.  The x-going and y-going face fluxes of a cell
// differ, so they are kept in two planes (x: buf, y: bufy), and the face
// records and the leakage carry the face fluxes, not the cell flux.
//
// NT: the largest CTA of the instantiation: 96 threads (tiles of up to 64
// columns) or 288 (one has 160, flow_mid_cta).  The register file is shared out by warps per scheduler, so
// a bound of 288 threads leaves at most 168 registers (96 for two CTAs).
// The bound of the instantiations for 96 threads, in CTAs per SM: five up to 12
// directions; three at S12 (four: the same at step, diamond P3 solves of 96x80x24
// 22.1 against 21.2 ms); at S16 two (step P0 to P2 12.2, 13.3, 24.3 ms; four: 12.9,
// 14.6, 27.6; step P3 takes 166 registers, so four CTAs are resident all the same),
// but four for diamond P0 to P2 (17.2, 18.8, 31.6 ms; two: 21.1, 23.7, 36.4), which
// otherwise take so many registers that too few warps are resident.
// Step S16 P3 has a third instantiation, for 97 to 160 threads (tiles of up to 128
// columns): two warps per scheduler leave it 255 registers (16x8 tiles, six
// iterations of 64x60x20, 8 groups: 5.0 ms, 7.2 with the bound for 288 threads).
constexpr bool flow_mid_cta(int AB, int M, int threads, bool DD) { return AB == 36 && M == 16 && !DD && threads > 96 && threads <= 160; }
constexpr int flow_min_ctas(int AB, int M, bool DD, int NT) {
    if (NT > 96) return AB > 12 ? 1 : 2;
    return AB <= 12 ? kFlowMinCtas : AB <= 21 ? 3 : DD && M < 16 ? 4 : 2;
}
template <int AB, int M, int MODE, bool SPLIT, bool DD, int NT>
__global__ void __launch_bounds__(NT, flow_min_ctas(AB, M, DD, NT))
    k_sweep_flow(const SweepArgs a, const ChainDirTable dt) {
    static_assert(!SPLIT || MODE == 0, "split transforms sweep in mode 0 only");
    static_assert(!DD || !SPLIT, "diamond differencing in the fused kernel only");
    constexpr int ABP = flow_abp(AB);
    constexpr int RS = flow_rs(AB), PW = flow_pw(AB);   // plane record: floats, vector width
    constexpr int RF = SPLIT ? ABP : M;                 // floats of a cell's source record
    constexpr bool COOP = RF == 16;                     // record moved by four lanes
    // S16 P3: lane sums, and signs, of two directions or moments in one packed
    // operation, which keeps the 36 x 16 products out of local memory (28.1 ms
    // against 55.9 for a step solve of 96x80x24; six iterations of 64x60x20 diamond,
    // 16x16 tiles: 8.1 against 11.4).  Not in step CTAs of up to 288 threads, whose
    // 168 registers it overflows (16x16 tiles 9.8 against 7.3); elsewhere one by one
    // is as fast or faster (S8 P3 11.98 against 12.38, S6 P3 10.2 against 10.7)
    constexpr bool PAIRED = !SPLIT && AB == 36 && M == 16 && (DD || NT < 288);
    constexpr bool FUSED = !SPLIT && flow_fused_sig(DD, M);   // denominator fma(rho, sigma_t, sum c)
    extern __shared__ float4 sm4[];
    if (a.skip && *a.skip) return;          // retired instance of a batched loop
    const int PX = chain_px(a.tx);
    const int P = PX * (a.ty + 1);
    const int T = a.tx * a.ty;                                // column threads
    const int D = a.depth, PD = a.fdepth;   // steps held of source records (2 or 4) and of face records (also 1)
    float* ring = reinterpret_cast<float*>(sm4);              // [D][T][RF] source records
    float* sring = ring + flow_up4(D * T * RF);               // [D][T] rho sigma_t (FUSED: sigma_t, then [D][T] rho)
    float* landx = sring + flow_up4((FUSED ? 2 : 1) * D * T);                   // [PD][ty][ABP] fetched x-face records
    float* landy = landx + PD * a.ty * ABP;                   // [PD][tx][ABP] fetched y-face records
    float* buf = landy + PD * a.tx * ABP;                     // [2][P][RS]
    float* bufy = DD ? buf + 2 * P * RS : buf;                // [2][P][RS] y-going faces (diamond)
    double* leak_s = reinterpret_cast<double*>(buf + flow_up4((DD ? 4 : 2) * P * RS));   // [gcount]
    int* task_s = reinterpret_cast<int*>(leak_s + a.gcount);

    // groups swept: [g0, g0 + gcount), from device memory in a batched
    // graph loop (a.g0, a.gcount then size the buffers only)
    int g0 = a.g0, gcount = a.gcount;
    if (a.win) {
        g0 = a.win[0];
        gcount = a.win[1] - a.win[0];
    }
    for (int e = threadIdx.x; e < gcount; e += blockDim.x) leak_s[e] = 0.0;
    for (int e = threadIdx.x; e < (DD ? 4 : 2) * P * RS; e += blockDim.x) buf[e] = 0.0f;

    // The face warp is the CTA's first or last warp, by the warp slot the CTA
    // starts at: the slots go round the SM's four schedulers, and this way the
    // column warps of successive three-warp CTAs take schedulers 1, 2 and 3, 0
    // in turn, so that an even number of CTAs loads them evenly
    unsigned wslot;
    asm volatile("mov.u32 %0, %%warpid;" : "=r"(wslot));
    if (threadIdx.x == 0) task_s[1] = (int)(wslot & 1);
    __syncthreads();
    const int nwarps = (int)(blockDim.x >> 5), wid = (int)(threadIdx.x >> 5);
    const int fwarp = task_s[1] ? nwarps - 1 : 0;
    const bool fw = wid == fwarp;
    const int tid = (int)threadIdx.x - (wid > fwarp ? 32 : 0), lane = threadIdx.x & 31;   // column threads: 0 .. T - 1
    const unsigned nxy = (unsigned)a.nx * a.ny;
    const size_t V = (size_t)nxy * a.nz;
    const int ntxf = a.ntx > 1 ? a.ntx - 1 : 0, ntyf = a.nty > 1 ? a.nty - 1 : 0;
    const size_t xslab = (size_t)a.ny * a.nz * ABP, yslab = (size_t)a.nx * a.nz * ABP;
    const int ntasks = a.ntx * a.nty * 8 * gcount;
    const int hend = a.nz + a.tx + a.ty - 2;                  // steps of a task

    // threads own the tile's columns in diagonal order (li + lj ascending)
    const bool colthread = !fw && tid < T;
    int li = 0, lj = 0;
    if (colthread) flow_column(tid, a.tx, a.ty, li, lj);
    const int d = li + lj;
    const int cs = (lj + 1) * PX + li + 1;
    const int xs = (cs - 1) * RS, ys = (cs - PX) * RS, os = cs * RS;
    // cooperative records: this lane moves the 16-byte quarter lane & 3 of the
    // records of lanes 8 i + lane / 4, i = 0..3, of its warp.  A record's
    // quarter c lies at position c ^ ((owner / 2) & 3) of the owner's 64-byte
    // slot, so that own-record reads (eight lanes, eight slots) and
    // quarter-wise reads (two whole slots) both fall in distinct banks
    const int qown = lane >> 2;
    const int qoff = ((tid & ~31) + qown) * 16 + (((lane & 3) ^ ((qown >> 1) & 3)) << 2);   // floats, owner qown
    const int soff = COOP ? tid * 16 + (((tid >> 1) & 3) << 2) : tid * RF;                  // own record's quarter 0
    const float qnan = __int_as_float(0x7fffffff);

    float zc[AB];                             // z inflow of the column's next cell
    float lk = 0.0f;
    int stage = 0, sbase = 0;                 // stage of the CTA's current task and its first task
    const int hook = a.flow[3] - 1;           // test hook: this task owes no faces
    if (threadIdx.x == 0) *task_s = atomicAdd(a.flow + 0, 1);
    __syncthreads();
    for (;;) {
        const int t = *task_s;
        if (t >= ntasks) break;
        const bool withhold = hook == t;
        // task t: stage, then tile fastest, octant, group (a CTA's tasks ascend)
        int ntiles = flow_stage_tiles(stage, a.ntx, a.nty);
        while (t >= sbase + ntiles * 8 * gcount) {
            sbase += ntiles * 8 * gcount;
            ntiles = flow_stage_tiles(++stage, a.ntx, a.nty);
        }
        int r = t - sbase;
        const int ti = r % ntiles;
        r /= ntiles;
        const int o = r & 7, gi = r >> 3;
        const int g = g0 + gi;
        const int at = max(0, stage - (a.nty - 1)) + ti, bt = stage - at;
        const int oe = a.reverse ? (o ^ 7) : o;     // octant of the directions
        const size_t gV = (size_t)g * V;
        const size_t og = (size_t)o * a.G + g;
        // the next task is taken a few steps before this one ends (the counter's
        // round trip is then off the critical path).  A CTA then holds at most the
        // task it sweeps and a later one: the lowest unfinished task is always
        // being swept, so the waits below still end
        const int htake = max(-1, hend - 6), hgive = max(0, hend - 3);

        if (fw) {
            // ---- face warp: the incoming face records ----
            // lane r owns x-face row r (r < ty: the record entering column (0, r))
            // and y-face column r - ty (entering column (r - ty, 0)), and again r + 32
            int next = 0;
            struct Rec {
                float* src;      // record of plane 0 (null on the mesh boundary: zero inflow)
                int idx, land, halo, lstride;
                bool ok;
            };
            auto rec = [&](int q) {
                Rec c;
                if (q < a.ty) {
                    const int jr2 = bt * a.ty + q;
                    c.idx = q;
                    c.ok = jr2 < a.ny;
                    c.src = at > 0 ? a.xface + (og * ntxf + at - 1) * xslab + (size_t)jr2 * a.nz * ABP : nullptr;
                    c.land = (int)(landx - ring) + q * ABP;
                    c.lstride = a.ty * ABP;
                    c.halo = (int)(buf - ring) + (q + 1) * PX * RS;
                } else {
                    c.idx = q - a.ty;
                    const int ir2 = at * a.tx + c.idx;
                    c.ok = ir2 < a.nx;
                    c.src = bt > 0 ? a.yface + (og * ntyf + bt - 1) * yslab + (size_t)ir2 * a.nz * ABP : nullptr;
                    c.land = (int)(landy - ring) + c.idx * ABP;
                    c.lstride = a.tx * ABP;
                    c.halo = (int)(bufy - ring) + (c.idx + 1) * RS;
                }
                return c;
            };
            const int nrec = a.tx + a.ty;
            Rec first = rec(lane < nrec ? lane : 0);
            first.ok = first.ok && lane < nrec;
            // fetch the records used at step st (plane st - idx of each edge column)
            auto issue1 = [&](const Rec& c, int st) {
                const int pf = st - c.idx;
                if (c.ok && c.src && (unsigned)pf < (unsigned)a.nz) {
                    float* land = ring + c.land + (st & (PD - 1)) * c.lstride;
                    const float* s0 = c.src + (size_t)flow_face_slot<AB>(pf, a.nz) * ABP;
#pragma unroll
                    for (int c4 = 0; c4 < ABP / 4; ++c4) cp_async_cg16(land + 4 * c4, s0 + 4 * c4);
                }
            };
            auto issue = [&](int st) {
                issue1(first, st);
                for (int q = lane + 32; q < nrec; q += 32) issue1(rec(q), st);
                asm volatile("cp.async.commit_group;\n" ::: "memory");
            };
            // the records of step st (fetched PD steps ago): wait until the producer
            // has written every flux (no NaN left), move into the halo of plane
            // buffer cbf, hand back to the next sweep as NaN; zero inflow on the
            // mesh boundary
            auto fill1 = [&](const Rec& c, int st, int cbf) {
                const int pf = st - c.idx;
                if (!c.ok || (unsigned)pf >= (unsigned)a.nz) return;
                float v[ABP];
                if (!c.src) {
#pragma unroll
                    for (int q = 0; q < ABP; ++q) v[q] = 0.0f;
                } else {
                    const float4* land = reinterpret_cast<const float4*>(ring + c.land + (st & (PD - 1)) * c.lstride);
                    float* s0 = c.src + (size_t)flow_face_slot<AB>(pf, a.nz) * ABP;
#pragma unroll
                    for (int c4 = 0; c4 < ABP / 4; ++c4) {
                        const float4 t4 = land[c4];
                        v[4 * c4] = t4.x; v[4 * c4 + 1] = t4.y; v[4 * c4 + 2] = t4.z; v[4 * c4 + 3] = t4.w;
                    }
                    bool got = false;
                    for (int it = 0; it < kFlowSpinLimit; ++it) {
                        got = true;
#pragma unroll
                        for (int q = 0; q < AB; ++q) got = got && !isnan(v[q]);
                        if (got) break;
                        // once any wait of this sweep has given up, give up at once
                        if ((it & 63) == 63 && *reinterpret_cast<volatile int*>(a.flow + 2)) break;
                        __nanosleep(20);
#pragma unroll
                        for (int c4 = 0; c4 < ABP / 4; ++c4) {
                            const float4 t4 = ld_relaxed4(s0 + 4 * c4);
                            v[4 * c4] = t4.x; v[4 * c4 + 1] = t4.y; v[4 * c4 + 2] = t4.z; v[4 * c4 + 3] = t4.w;
                        }
                    }
                    if (!got) {
                        atomicExch(a.flow + 2, 1);
#pragma unroll
                        for (int q = 0; q < ABP; ++q) v[q] = 0.0f;
                    }
                    float4* back = reinterpret_cast<float4*>(s0);
#pragma unroll
                    for (int c4 = 0; c4 < ABP / 4; ++c4) back[c4] = make_float4(qnan, qnan, qnan, qnan);
                }
                plane_store<AB>(ring + c.halo + cbf * P * RS, v);
            };
            for (int st = 0; st < PD - 1; ++st) issue(st);
#pragma unroll 1
            for (int h = -1; h < hend; ++h) {
                if (h == htake && lane == 0) next = atomicAdd(a.flow + 0, 1);
                issue(h + PD);
                if (PD == 4) asm volatile("cp.async.wait_group 3;\n" ::: "memory");
                else if (PD == 2) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                fill1(first, h + 1, h & 1);
                for (int q = lane + 32; q < nrec; q += 32) fill1(rec(q), h + 1, h & 1);
                if (h == hgive && lane == 0) *task_s = next;
                flow_step_barrier();
            }
            continue;
        }

        // ---- column warps ----
        const int sx = (o & 1) ? -1 : 1, sy = (o & 2) ? -1 : 1, sz = (o & 4) ? -1 : 1;
        const float fx = (oe & 1) ? -1.0f : 1.0f, fy = (oe & 2) ? -1.0f : 1.0f, fz = (oe & 4) ? -1.0f : 1.0f;
        const int ir = at * a.tx + li, jr = bt * a.ty + lj;
        const bool col = colthread && ir < a.nx && jr < a.ny;
        const unsigned nzc = col ? a.nz : 0;        // planes of this thread's column
        // cells are stepped by +-nxy; index of the cell of step h = -1 (out of the
        // mesh until the column starts; only used where 0 <= plane < nz)
        const int szn = sz > 0 ? (int)nxy : -(int)nxy;
        unsigned v = (unsigned)((sy > 0 ? jr : a.ny - 1 - jr) * a.nx + (sx > 0 ? ir : a.nx - 1 - ir)) +
                     (sz > 0 ? 0u : (unsigned)(a.nz - 1) * nxy) - (unsigned)((1 + d) * szn);
        int kr = -1 - d;                            // plane (in sweep order) of this step
        const bool xout = li == a.tx - 1 && at < a.ntx - 1 && !withhold;
        const bool yout = lj == a.ty - 1 && bt < a.nty - 1 && !withhold;
        const bool xleak = ir == a.nx - 1, yleak = jr == a.ny - 1;
        float* const xo = a.xface + (og * ntxf + at) * xslab + (size_t)jr * a.nz * ABP;
        float* const yo = a.yface + (og * ntyf + bt) * yslab + (size_t)ir * a.nz * ABP;
        const size_t ang0 = ((size_t)g * 8 + oe) * V;       // angular records of (group, direction octant)
        const float* const srcg = SPLIT ? a.qang + ang0 * ABP : a.src + gV * M;
        const float* const sigg = dt.sig + gV;
        float* const momg = SPLIT ? a.pang + ang0 * ABP : a.mom + gV * M;
        // cooperative records: cell of each owner at the step of the prefetch, so
        // that the reductions' base is D - 1 cells back
        int vo[COOP ? 4 : 1];
        const float* const srcq = srcg + ((lane & 3) << 2);
        float* const momq = momg + ((lane & 3) << 2) - (ptrdiff_t)(D - 1) * szn * 16;
        if constexpr (COOP) {
#pragma unroll
            for (int i = 0; i < 4; ++i) vo[i] = __shfl_sync(0xffffffffu, (int)v, 8 * i + qown) + (D - 1) * szn;
        }
        // fetch the source record and the cross section of the cell D - 1 steps
        // ahead into ring slot `slot`
        auto prefetch = [&](int ahead, int slot) {
            const bool pre = (unsigned)(kr + ahead) < nzc;
            const unsigned vp = v + (unsigned)(ahead * szn);
            if constexpr (COOP) {
                const unsigned mp = __ballot_sync(0xffffffffu, pre) >> qown;
                float* dst = ring + slot * T * 16 + qoff;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if ((mp >> (8 * i)) & 1u)
                        cp_async_cg16(dst + 128 * i, srcq + ((ptrdiff_t)vo[i] + (ahead - (D - 1)) * szn) * 16);
            } else if (pre) {
                float* dst = ring + slot * T * RF + soff;
                const float* s0 = srcg + (size_t)vp * RF;
                if constexpr (RF % 4 == 0) {
#pragma unroll
                    for (int c4 = 0; c4 < RF / 4; ++c4) cp_async_cg16(dst + 4 * c4, s0 + 4 * c4);
                } else {
#pragma unroll
                    for (int m = 0; m < RF; ++m) cp_async_f32(dst + m, s0 + m);
                }
            }
            if (pre) cp_async_f32(sring + slot * T + tid, sigg + vp);
            if (FUSED && pre) cp_async_f32(sring + (D + slot) * T + tid, a.rho + vp);
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        for (int st = 0; st < D - 2; ++st) prefetch(st + 1, st & (D - 1));   // steps 0 .. D - 3
#pragma unroll
        for (int q = 0; q < AB; ++q) zc[q] = 0.0f;
#pragma unroll 1
        for (int h = -1; h < hend; ++h) {
            const int cb = h & 1, pb = cb ^ 1;
            const int slot = h & (D - 1);
            prefetch(D - 1, (h + D - 1) & (D - 1));
            const bool act = (unsigned)kr < nzc;
            if (act) {
                const bool last = kr == a.nz - 1;
                const float sig = sring[slot * T + tid];
                const float rho = FUSED ? sring[(D + slot) * T + tid] : 1.0f;
                const float* rs = ring + slot * T * RF;
                float s[RF];
                if constexpr (RF % 4 == 0) {
#pragma unroll
                    for (int c4 = 0; c4 < RF / 4; ++c4) {
                        const float4 t4 = *reinterpret_cast<const float4*>(rs + (COOP ? soff ^ (c4 << 2) : soff + 4 * c4));
                        s[4 * c4] = t4.x; s[4 * c4 + 1] = t4.y; s[4 * c4 + 2] = t4.z; s[4 * c4 + 3] = t4.w;
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < RF; ++m) s[m] = rs[soff + m];
                }
                float st4[MODE == 2 ? ABP : 1];     // stored angular fluence (mode 2), read ahead of its use
                if constexpr (MODE == 2) {
                    const float4* rec =
                        reinterpret_cast<const float4*>(a.psi + ((ang0 + v) * a.nab + a.blk) * ABP);
#pragma unroll
                    for (int c4 = 0; c4 < ABP / 4; ++c4) {
                        const float4 t4 = __ldg(rec + c4);
                        st4[4 * c4] = t4.x; st4[4 * c4 + 1] = t4.y; st4[4 * c4 + 2] = t4.z; st4[4 * c4 + 3] = t4.w;
                    }
                }
                // moments -> directions (split: the record already holds them)
                float psi[AB];
                if constexpr (SPLIT) {
#pragma unroll
                    for (int q = 0; q < AB; ++q) psi[q] = s[q];
                } else if constexpr (PAIRED) {
#pragma unroll
                    for (int m = 0; m < M; m += 2) {
                        const float2 r2 = __fmul2_rn(make_float2(s[m], s[m + 1]),
                                                     make_float2(octant_sign<M>(m, fx, fy, fz), octant_sign<M>(m + 1, fx, fy, fz)));
                        s[m] = r2.x;
                        s[m + 1] = r2.y;
                    }
#pragma unroll
                    for (int q = 0; q < AB; q += 2) {
                        const float2 ta = dot2<M>(dt.mop + q * 16, s), tb = dot2<M>(dt.mop + (q + 1) * 16, s);
                        const float2 p2 = __fadd2_rn(make_float2(ta.x, tb.x), make_float2(ta.y, tb.y));
                        psi[q] = p2.x;
                        psi[q + 1] = p2.y;
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < M; ++m) s[m] *= octant_sign<M>(m, fx, fy, fz);
#pragma unroll
                    for (int q = 0; q < AB; ++q) psi[q] = dot<M>(dt.mop + q * 16, s);
                }
                // cell solve, PW directions at a time (the plane records' vector width)
                const float* pv = buf + pb * P * RS;
                float* cv = buf + cb * P * RS;
                const float* pvy = bufy + pb * P * RS;    // step: the same plane
                float* cvy = bufy + cb * P * RS;
#pragma unroll
                for (int q0 = 0; q0 < AB; q0 += PW) {
                    float px[PW], py[PW];
                    plane_load<PW>(pv + xs + q0, px);
                    plane_load<PW>(pvy + ys + q0, py);
#pragma unroll
                    for (int e = 0; e + 1 < PW; e += 2) {
                        const int q = q0 + e;
                        if (q + 1 < AB) {
                            // two directions per packed operation
                            float2 n2 = __ffma2_rn(make_float2(dt.cx[q], dt.cx[q + 1]), make_float2(px[e], px[e + 1]),
                                                   make_float2(psi[q], psi[q + 1]));
                            n2 = __ffma2_rn(make_float2(dt.cy[q], dt.cy[q + 1]), make_float2(py[e], py[e + 1]), n2);
                            n2 = __ffma2_rn(make_float2(dt.cz[q], dt.cz[q + 1]), make_float2(zc[q], zc[q + 1]), n2);
                            const float2 cs2 = make_float2(dt.csum[q], dt.csum[q + 1]);
                            const float2 d2 = FUSED ? __ffma2_rn(make_float2(rho, rho), make_float2(sig, sig), cs2)
                                                    : __fadd2_rn(make_float2(sig, sig), cs2);
                            psi[q] = n2.x * rcp_approx(d2.x);
                            psi[q + 1] = n2.y * rcp_approx(d2.y);
                        }
                    }
                    if (q0 + PW > AB || PW == 1) {
                        if constexpr (AB % 2 == 1) {
                            constexpr int q = AB - 1;
                            const int e = q - q0;
                            const float num = fmaf(dt.cz[q], zc[q], fmaf(dt.cy[q], py[e], fmaf(dt.cx[q], px[e], psi[q])));
                            psi[q] = num * rcp_approx(FUSED ? fmaf(rho, sig, dt.csum[q]) : sig + dt.csum[q]);
                        }
                    }
#pragma unroll
                    for (int e = 0; e < PW; ++e) {
                        const int q = q0 + e;
                        if (q < AB) {
                            if constexpr (DD) {
                                px[e] = fmaf(2.0f, psi[q], -px[e]);
                                py[e] = fmaf(2.0f, psi[q], -py[e]);
                                zc[q] = fmaf(2.0f, psi[q], -zc[q]);
                            } else {
                                px[e] = psi[q];
                                zc[q] = psi[q];
                            }
                        } else {
                            px[e] = py[e] = 0.0f;     // record padding
                        }
                    }
                    plane_store_w<PW>(cv + os + q0, px);
                    if constexpr (DD) plane_store_w<PW>(cvy + os + q0, py);
                }
                // stored angular fluence, laid out for this kernel as one 16-byte
                // aligned record of ABP floats per (group, direction octant, voxel,
                // direction block): [G][8][V][nab][ABP] (the stage kernels use [G][V][A]).
                // A record need not fill its last 32-byte sector; this way the x
                // neighbour, one step later, fills it while it is still in L2 (with the
                // octants of a voxel side by side it was written back half full)
                if constexpr (MODE == 1)
                    store_record<AB>(a.psi + ((ang0 + v) * a.nab + a.blk) * ABP, psi);
                if constexpr (MODE == 2) {
                    float pacc = 0.0f;
#pragma unroll
                    for (int q = 0; q < AB; ++q) pacc = fmaf(dt.w[q] * psi[q], st4[q], pacc);
                    red_add_f32(a.prod + gV + v, pacc);
                }
                // outgoing face records of plane kr and the boundary currents
                if constexpr (DD) {
                    // the x and y face fluxes, read back from this thread's plane entries
                    const float* fxo = cv + os;
                    const float* fyo = cvy + os;
                    float f[AB];
                    if (xout) {
#pragma unroll
                        for (int q = 0; q < AB; ++q) f[q] = fxo[q];
                        store_record<AB>(xo + (size_t)flow_face_slot<AB>(kr, a.nz) * ABP, f);
                    }
                    if (yout) {
#pragma unroll
                        for (int q = 0; q < AB; ++q) f[q] = fyo[q];
                        store_record<AB>(yo + (size_t)flow_face_slot<AB>(kr, a.nz) * ABP, f);
                    }
                    if (xleak || yleak || last) {
#pragma unroll
                        for (int q = 0; q < AB; ++q) {
                            if (xleak) lk = fmaf(dt.lx[q], fxo[q], lk);
                            if (yleak) lk = fmaf(dt.ly[q], fyo[q], lk);
                            if (last) lk = fmaf(dt.lz[q], zc[q], lk);
                        }
                    }
                } else {
                    if (xout) store_record<AB>(xo + (size_t)flow_face_slot<AB>(kr, a.nz) * ABP, psi);
                    if (yout) store_record<AB>(yo + (size_t)flow_face_slot<AB>(kr, a.nz) * ABP, psi);
                    if (xleak || yleak || last) {
#pragma unroll
                        for (int q = 0; q < AB; ++q) {
                            float f = 0.0f;
                            if (xleak) f += dt.lx[q];
                            if (yleak) f += dt.ly[q];
                            if (last) f += dt.lz[q];
                            lk = fmaf(f, psi[q], lk);
                        }
                    }
                }
                if constexpr (SPLIT) {
                    // the cell's angular fluence record, for k_split_d2m
                    store_record<AB>(momg + (size_t)v * ABP, psi);
                } else {
                    // directions -> moments (Eq. 3 for lm = 00): table rows hold w R_lm
                    float acc[M];
                    if constexpr (PAIRED) {
#pragma unroll
                        for (int m = 0; m < M; m += 2) {
                            const float2 ta = dot2<AB>(dt.dop + m * kFlowMaxAB, psi), tb = dot2<AB>(dt.dop + (m + 1) * kFlowMaxAB, psi);
                            const float2 r2 = __fmul2_rn(__fadd2_rn(make_float2(ta.x, tb.x), make_float2(ta.y, tb.y)),
                                                         make_float2(octant_sign<M>(m, fx, fy, fz), octant_sign<M>(m + 1, fx, fy, fz)));
                            acc[m] = r2.x;
                            acc[m + 1] = r2.y;
                        }
                    } else {
#pragma unroll
                        for (int m = 0; m < M; ++m)
                            acc[m] = dot<AB>(dt.dop + m * kFlowMaxAB, psi) * octant_sign<M>(m, fx, fy, fz);
                    }
                    if constexpr (COOP) {
                        // into the consumed source slot, from where four lanes reduce each record
                        float* ws = ring + slot * T * 16;
#pragma unroll
                        for (int c4 = 0; c4 < 4; ++c4)
                            *reinterpret_cast<float4*>(ws + (soff ^ (c4 << 2))) =
                                make_float4(acc[4 * c4], acc[4 * c4 + 1], acc[4 * c4 + 2], acc[4 * c4 + 3]);
                    } else {
                        add_moments<M>(momg + (size_t)v * M, acc);
                    }
                }
            }
            if constexpr (COOP && !SPLIT) {
                const unsigned ma = __ballot_sync(0xffffffffu, act) >> qown;
                __syncwarp();
                const float* rq = ring + slot * T * 16 + qoff;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if ((ma >> (8 * i)) & 1u)
                        red_add_v4(momq + (ptrdiff_t)vo[i] * 16, *reinterpret_cast<const float4*>(rq + 128 * i));
#pragma unroll
                for (int i = 0; i < 4; ++i) vo[i] += szn;
            }
            v += (unsigned)szn;
            ++kr;
            // the next step's source records have landed
            if (D == 4) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
            else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            flow_step_barrier();
        }
        // the task's boundary current: one addition per warp (an FP64 shared-memory
        // addition is a compare-and-swap loop, so the columns of a finishing
        // diagonal must not each do one between two steps)
        if (__any_sync(0xffffffffu, lk != 0.0f)) {
            double x = lk;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
            if (lane == 0) atomicAdd(leak_s + gi, x);
            lk = 0.0f;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < gcount; e += blockDim.x)
        if (leak_s[e] != 0.0) atomicAdd(a.leak + g0 + e, leak_s[e]);
    // the last CTA out resets the queue for the next sweep
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.flow + 1, 1) == (int)gridDim.x - 1) {
            a.flow[0] = 0;
            a.flow[1] = 0;
        }
    }
}

// Moments -> angular source of every direction of every octant (the
// transform taken out of the split sweep): q[g][o][v][j] =
// sum_lm (2l+1)/(4 pi) R_lm(Omega_{o,j}) s_lm[g][v], with R of octant o the
// first octant's times the reflection signs.  One thread per (group, voxel),
// records written as 16-byte vectors; HBM-bound.
template <int M, int AB>
__global__ void __launch_bounds__(256) k_split_m2d(const float* src, float* qang, size_t V, int g0, int gcount,
                                                  const int* skip) {
    constexpr int ABP = flow_abp(AB);
    constexpr int rb = chain_row_base(AB) * 16;
    if (skip && *skip) return;
    const size_t n = (size_t)gcount * V;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const int g = g0 + (int)(e / V);
        const size_t v = e % V;
        float s[M];
        load_moments<M>(src + ((size_t)g * V + v) * M, s);
#pragma unroll 1
        for (int o = 0; o < 8; ++o) {
            const float fx = (o & 1) ? -1.0f : 1.0f, fy = (o & 2) ? -1.0f : 1.0f, fz = (o & 4) ? -1.0f : 1.0f;
            float so[M];
#pragma unroll
            for (int m = 0; m < M; ++m) so[m] = s[m] * octant_sign<M>(m, fx, fy, fz);
            float q[ABP];
#pragma unroll
            for (int j = 0; j < ABP; ++j) {
                float t = 0.0f;
                if (j < AB) {
#pragma unroll
                    for (int m = 0; m < M; ++m) t = fmaf(c_Mop1[rb + j * 16 + lm_of_pos(m, M)], so[m], t);
                }
                q[j] = t;
            }
            float4* out = reinterpret_cast<float4*>(qang + (((size_t)g * 8 + o) * V + v) * ABP);
#pragma unroll
            for (int c4 = 0; c4 < ABP / 4; ++c4) out[c4] = make_float4(q[4 * c4], q[4 * c4 + 1], q[4 * c4 + 2], q[4 * c4 + 3]);
        }
    }
}

// Angular fluence of every direction -> moments (Eq. 3 for lm = 00):
// mom[g][v][lm] = sum_o sum_j w_j R_lm(Omega_{o,j}) psi[g][o][v][j], written
// with plain stores (one thread per (group, voxel), no reductions).
template <int M, int AB>
__global__ void __launch_bounds__(256) k_split_d2m(const float* pang, float* mom, size_t V, int g0, int gcount,
                                                  const int* skip) {
    constexpr int ABP = flow_abp(AB);
    constexpr int rb = chain_row_base(AB) * 16;
    if (skip && *skip) return;
    const size_t n = (size_t)gcount * V;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const int g = g0 + (int)(e / V);
        const size_t v = e % V;
        float acc[M];
#pragma unroll
        for (int m = 0; m < M; ++m) acc[m] = 0.0f;
#pragma unroll 1
        for (int o = 0; o < 8; ++o) {
            const float fx = (o & 1) ? -1.0f : 1.0f, fy = (o & 2) ? -1.0f : 1.0f, fz = (o & 4) ? -1.0f : 1.0f;
            const float4* in = reinterpret_cast<const float4*>(pang + (((size_t)g * 8 + o) * V + v) * ABP);
            float ps[ABP];
#pragma unroll
            for (int c4 = 0; c4 < ABP / 4; ++c4) {
                const float4 t4 = __ldg(in + c4);
                ps[4 * c4] = t4.x; ps[4 * c4 + 1] = t4.y; ps[4 * c4 + 2] = t4.z; ps[4 * c4 + 3] = t4.w;
            }
#pragma unroll
            for (int m = 0; m < M; ++m) {
                float b = 0.0f;
#pragma unroll
                for (int j = 0; j < AB; ++j) b = fmaf(c_Dop1[rb + j * 16 + lm_of_pos(m, M)], ps[j], b);
                acc[m] = fmaf(octant_sign<M>(m, fx, fy, fz), b, acc[m]);
            }
        }
        float* out = mom + ((size_t)g * V + v) * M;
        if constexpr (M % 4 == 0) {
            float4* o4 = reinterpret_cast<float4*>(out);
#pragma unroll
            for (int c4 = 0; c4 < M / 4; ++c4) o4[c4] = make_float4(acc[4 * c4], acc[4 * c4 + 1], acc[4 * c4 + 2], acc[4 * c4 + 3]);
        } else {
#pragma unroll
            for (int m = 0; m < M; ++m) out[m] = acc[m];
        }
    }
}

template <int M>
int sweep_flow_blocks_per_sm(int ab, int threads, size_t smem, bool split, bool dd) {
    int b = 0;
    cudaError_t e = cudaErrorInvalidValue;
    auto query = [&](auto kern) {
        e = smem > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                             : cudaSuccess;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem);
    };
#define DOCTORS_FLOW_OCC(AB)                                                        \
    case AB:                                                                        \
        if (split) {                                                                \
            if constexpr (AB <= 10) query(k_sweep_flow<AB, M, 0, true, false, 288>);  \
        } else if (threads <= 96) {                                                 \
            if (dd) query(k_sweep_flow<AB, M, 0, false, true, 96>);                  \
            else query(k_sweep_flow<AB, M, 0, false, false, 96>);                    \
        } else if (flow_mid_cta(AB, M, threads, dd)) {                               \
            if constexpr (flow_mid_cta(AB, M, 160, false)) query(k_sweep_flow<AB, M, 0, false, false, 160>); \
        } else if (dd) query(k_sweep_flow<AB, M, 0, false, true, 288>);              \
        else query(k_sweep_flow<AB, M, 0, false, false, 288>);                       \
        break;
    switch (ab) {
        DOCTORS_FLOW_OCC(1)
        DOCTORS_FLOW_OCC(3)
        DOCTORS_FLOW_OCC(6)
        DOCTORS_FLOW_OCC(10)
        DOCTORS_FLOW_OCC(12)
        DOCTORS_FLOW_OCC(21)
        DOCTORS_FLOW_OCC(36)
        default: break;
    }
#undef DOCTORS_FLOW_OCC
    return e == cudaSuccess ? b : 0;
}

// m2d, split sweep, d2m: one full sweep with the transforms taken out
template <int M>
cudaError_t launch_split_sweep_m(const SweepArgs& a, cudaStream_t s, int* count) {
    *count = 0;
    if (a.gcount <= 0) return cudaSuccess;
    if (a.dir_table == nullptr || a.flow == nullptr || a.dir_table->sig == nullptr || !flow_depths_ok(a.depth, a.fdepth) || a.nab != 1 || !a.qang ||
        !a.pang)
        return cudaErrorInvalidValue;
    const size_t V = (size_t)a.nx * a.ny * a.nz;
    const size_t n = (size_t)a.gcount * V;
    const unsigned tgrid = (unsigned)std::min<size_t>((n + 255) / 256, 152 * 8);
    int ntasks = 0;
    for (int st = 0; st < a.ntx + a.nty - 1; ++st) {
        const int lo = st - (a.nty - 1) > 0 ? st - (a.nty - 1) : 0;
        const int hi = st < a.ntx - 1 ? st : a.ntx - 1;
        ntasks += (hi - lo + 1) * 8 * a.gcount;
    }
    // persistent CTAs: every resident slot, or its share when several instances sweep at once
    const int slots = std::max(1, a.chain_slots / std::max(1, a.slot_share));
    const int grid = ntasks < slots ? ntasks : slots;
    const int T = flow_threads(a.tx, a.ty);
    const size_t smem = sweep_flow_smem_bytes(a.ab, flow_abp(a.ab), a.tx, a.ty, a.gcount, a.depth, a.fdepth);
    cudaError_t e = cudaSuccess;
    // P3: the transforms on the tensor cores when the problem holds their tables
    const bool tc = M == 16 && a.tc_b1 && a.tc_b2;
    auto run = [&](auto m2d, auto sweep, auto d2m) {
        if (tc) {
            e = launch_m2d_tc(a, s);
        } else {
            m2d<<<tgrid, 256, 0, s>>>(a.src, const_cast<float*>(a.qang), V, a.g0, a.gcount, a.skip);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && smem > 48 * 1024)
            e = cudaFuncSetAttribute(sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) {
            sweep<<<grid, T, smem, s>>>(a, *a.dir_table);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) {
            if (tc) {
                e = launch_d2m_tc(a, s);
            } else {
                d2m<<<tgrid, 256, 0, s>>>(a.pang, a.mom, V, a.g0, a.gcount, a.skip);
                e = cudaGetLastError();
            }
        }
    };
    switch (a.ab) {
        case 1: run(k_split_m2d<M, 1>, k_sweep_flow<1, M, 0, true, false, 288>, k_split_d2m<M, 1>); break;
        case 3: run(k_split_m2d<M, 3>, k_sweep_flow<3, M, 0, true, false, 288>, k_split_d2m<M, 3>); break;
        case 6: run(k_split_m2d<M, 6>, k_sweep_flow<6, M, 0, true, false, 288>, k_split_d2m<M, 6>); break;
        case 10: run(k_split_m2d<M, 10>, k_sweep_flow<10, M, 0, true, false, 288>, k_split_d2m<M, 10>); break;
        default: return cudaErrorInvalidValue;
    }
    if (e == cudaSuccess) *count = 3;
    return e;
}

template <int M, int MODE>
cudaError_t launch_sweep_flow_m(const SweepArgs& a, cudaStream_t s) {
    if (a.gcount <= 0) return cudaSuccess;
    if (a.dir_table == nullptr || a.flow == nullptr || a.dir_table->sig == nullptr || !flow_depths_ok(a.depth, a.fdepth) || a.blk < 0 || a.blk >= a.nab ||
        a.ab * a.nab != a.A8)
        return cudaErrorInvalidValue;
    const bool dd = a.dd != 0;
    int ntasks = 0;
    for (int st = 0; st < a.ntx + a.nty - 1; ++st) {
        const int lo = st - (a.nty - 1) > 0 ? st - (a.nty - 1) : 0;
        const int hi = st < a.ntx - 1 ? st : a.ntx - 1;
        ntasks += (hi - lo + 1) * 8 * a.gcount;
    }
    // persistent CTAs: every resident slot, or its share when several instances sweep at once
    const int slots = std::max(1, a.chain_slots / std::max(1, a.slot_share));
    const int grid = ntasks < slots ? ntasks : slots;
    const int T = flow_threads(a.tx, a.ty);
    const size_t smem = sweep_flow_smem_bytes(a.ab, M, a.tx, a.ty, a.gcount, a.depth, a.fdepth, dd);
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        if (smem > 48 * 1024) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) kern<<<grid, T, smem, s>>>(a, *a.dir_table);
    };
#define DOCTORS_FLOW_CASE(AB)                                                        \
    case AB:                                                                         \
        if (T <= 96) {                                                               \
            if (dd) launch(k_sweep_flow<AB, M, MODE, false, true, 96>);               \
            else launch(k_sweep_flow<AB, M, MODE, false, false, 96>);                 \
        } else if (flow_mid_cta(AB, M, T, dd)) {                                     \
            if constexpr (flow_mid_cta(AB, M, 160, false)) launch(k_sweep_flow<AB, M, MODE, false, false, 160>); \
        } else if (dd) launch(k_sweep_flow<AB, M, MODE, false, true, 288>);           \
        else launch(k_sweep_flow<AB, M, MODE, false, false, 288>);                    \
        break;
    switch (a.ab) {
        DOCTORS_FLOW_CASE(1)
        DOCTORS_FLOW_CASE(3)
        DOCTORS_FLOW_CASE(6)
        DOCTORS_FLOW_CASE(10)
        DOCTORS_FLOW_CASE(12)
        DOCTORS_FLOW_CASE(21)
        DOCTORS_FLOW_CASE(36)
        default: return cudaErrorInvalidValue;
    }
#undef DOCTORS_FLOW_CASE
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace doctors
