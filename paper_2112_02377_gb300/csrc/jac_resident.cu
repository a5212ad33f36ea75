// FP64 sweeps of systems whose matrix fits in the chip's shared memory.
//
// One CTA per SM keeps its rows of S, their columns, b and its part of the
// iterate in shared memory for the whole launch; a sweep then moves only the
// iterate, through L2.  What is left of such a sweep is latency, and this
// kernel is arranged around the chain that every sweep has to go through:
// gather x, sum the row, store, pass the grid barrier (fence, arrival, poll:
// 1.3 us with one CTA per SM).  GB300's FP64 pipe takes 64 cycles per warp
// instruction and sub-partition, so the residual norm -- shuffle trees of
// FP64 adds, a square root, a division -- costs several times the row sums of
// a small system.  It is taken off the chain altogether:
//   sweep s      the math warps leave each thread's sum of r^2 and max |r| in
//                shared memory;
//   sweep s + 1  a spare warp adds them and publishes the CTA's partial sums;
//   sweep s + 2  a spare warp of CTA 0 adds all CTAs' partials (the barrier of
//                sweep s + 1 made them visible), takes the decision of sweep s and
//                publishes it as one word;
//   sweep s + 3  every CTA reads that word before it arrives at the barrier, or
//                already in sweep s + 2 where that is longer than the decision takes.
// The iterate rotates through five buffers, so the x^k that a stop returns is
// still there three sweeps later.  Iterates and infinity norms are those of the other
// kernels bit for bit; 2-norms are the same squares added in another order (2 n u
// apart at most), so a solve stops in the same sweep unless its test value lies that
// close to the tolerance.  The price of the late decision is two or three more sweeps
// after the one that passes: a solve that its first iterate ends takes 70 us at 70^3 (82
// with three), 59 in the pipelined kernel, and is even after two or three sweeps.
//
// Measured on GB300, 16^3 7-point: 2.3 to 2.4 us a sweep, of them 1.2 us in the grid
// barrier (a bare one takes 1.4 us; splitting its counter over several lines or
// polling differently changes less than 3 %); 2.75 with every CTA taking the
// decisions itself, 7.0 in the pipelined kernel.  64^3: 5.9 us against 10.7, of
// which 3.4 are the FP64 pipe's.  More sizes at the rule in jac_api.cu
// (resident_plan).
#include <cuda_runtime.h>

#include "jac_device.cuh"
#include "jac_launch.h"

namespace jac {

namespace {

constexpr int CH = 8;                           // entries whose gathers are issued together
constexpr int NBUF = 5;                         // iterate buffers
constexpr int NPART = 4;                        // sweeps whose partial sums are kept

// Math warps; two spare warps follow.  (20 with two lanes per row: 27-point 32^3
// 4.54 -> 4.21 us a sweep, but the 33^3 Q1 replay 3.74 -> 3.94: every idle warp
// costs the barriers something.)
constexpr int MW = 16;
constexpr int RT = (MW + 2) * 32;

// A CTA's sums cost the first spare warp up to 21 FP64 instructions, all on the
// sub-partition of the warps 0, 4, 8, ...; a slice of short rows costs its warp 8.
// So the first slices go to the warps of the other three only (7-point 48^3
// 3.92 -> 3.67 us a sweep, 64^3 6.33 -> 5.92; with two lanes, whose slices cost
// 16, 27-point 32^3 4.1 -> 4.5: none there).
template <int L>
constexpr int uneven_slices() { return L == 1 ? 9 : 0; }

struct ResidentDecision {
    long long k, k_limit, hist_at, hist_cap;    // iterate of the launch's first sweep; limits
    double tol, bnorm, pass;
    double* hist;
    int kind, test;
    double relres, res2, resinf;
    long long k_eval;
    int loc_part;                               // local stopping: the partition that passed, its value
    double loc_val;
};

// Barrier of the math warps and the first spare warp.
template <int ID, int THREADS>
__device__ __forceinline__ void cta_sync()
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}

__device__ void init_decision(ResidentDecision& d, const volatile JacCtl* c)
{
    d.k = c->k;
    d.k_limit = c->k_limit;
    d.hist_at = c->evals;
    d.hist_cap = c->hist_cap;
    d.tol = c->tol;
    d.bnorm = c->bnorm;
    d.hist = c->hist;
    d.kind = c->norm_kind;
    d.test = c->test;
    d.relres = c->relres;
    d.res2 = c->res2;
    d.resinf = c->resinf;
    d.k_eval = c->k_eval;
    d.loc_part = -1;
    d.loc_val = 0.0;
    // A sum of squares above this fails the 2-norm test whatever decide()
    // rounds (the margin covers its roundings and ours), so most sweeps are
    // decided without its square root and division.  Where the product is too
    // small to carry the margin, decide() is always asked.
    const double v = d.bnorm > 0.0 ? d.tol * d.bnorm : d.tol;
    d.pass = v * v * (1.0 + 1e-12);
    if (!(d.pass > 1e-280)) d.pass = 1.7976931348623157e308;
}

// The decision of sweep j of the launch, by one warp, from every CTA's partial
// sums (in every lane).  LOC: the first partition whose own rows pass ends the
// solve too; its maxima are cleared for sweep j + NPART once they have been read.
template <bool LOC>
__device__ int take_decision(ResidentDecision& s, const Partial* part, unsigned long long* loc, int nloc, JacCtl* ctl,
                             int j, bool last)
{
    int done = DONE_RUNNING;
    [[maybe_unused]] unsigned long long lk = ~0ull;
    [[maybe_unused]] int lp = -1;
    if constexpr (LOC) {
        local_sets_min(loc, nloc, lk, lp);
        for (int i = threadIdx.x & 31; i < nloc; i += 32) __stcg(loc + i, 0ull);
    }
    // five partials of a lane are loaded together (one round trip for 160 CTAs)
    double tss = 0.0;
    unsigned long long tmx = 0;
    for (int i = threadIdx.x & 31; i < (int)gridDim.x; i += 160) {
        ulonglong2 w[5];
#pragma unroll
        for (int u = 0; u < 5; ++u)
            w[u] = i + 32 * u < (int)gridDim.x ? __ldcg(reinterpret_cast<const ulonglong2*>(part + i + 32 * u))
                                               : make_ulonglong2(0ull, 0ull);
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            tss += __longlong_as_double((long long)w[u].x);
            tmx = umax64(tmx, w[u].y);
        }
    }
    tss = warp_sum(tss);
    tmx = warp_max_all(tmx);
    if ((threadIdx.x & 31) == 0) {
        const long long k = s.k + j;
        const bool bad = !(tss <= 1.7976931348623157e308) || tmx >= KEY_INF;
        bool near = s.kind == 2 ? !(tss > s.pass) : abs_from_key(tmx) <= s.tol;
        // (NaN keys never pass)
        const bool local = LOC && s.test && nloc > 0 && lk <= KEY_INF && abs_from_key(lk) <= s.tol;
        if constexpr (LOC) near = near || local;
        if (last || s.hist || bad || (s.test && (k >= s.k_limit || near))) {
            const Decision d = decide(s.test, s.tol, s.k_limit, s.kind, s.bnorm, tss, tmx, k);
            s.relres = d.relres;
            s.res2 = d.res2;
            s.resinf = d.resinf;
            s.k_eval = k;
            done = d.done;
            if constexpr (LOC) {
                if (local && !d.numeric_bad) {
                    done = DONE_CONVERGED;
                    s.loc_part = lp;
                    s.loc_val = abs_from_key(lk);
                }
            }
            if (d.numeric_bad) atomicOr(&ctl->status, ST_NUMERIC);
            if (s.hist && s.hist_at + j < s.hist_cap) s.hist[s.hist_at + j] = d.relres;
        }
    }
    return __shfl_sync(0xffffffffu, done, 0);
}

// A CTA's partial sums of one sweep, by one warp: its math threads' sums
// (active: those that own rows), lane-strided, then a fixed tree.
__device__ void publish(const double* ss, const unsigned long long* mx, int active, Partial* slot)
{
    const int lane = threadIdx.x & 31;
    double a = 0.0;
    unsigned long long b = 0;
    for (int i = lane; i < active; i += 32) {
        a += ss[i];
        b = umax64(b, mx[i]);
    }
    a = warp_sum(a);
    b = warp_max_all(b);
    if (lane == 0) {
        __stcg(&slot->ss, a);
        __stcg(&slot->mx, b);
    }
}

}  // namespace

// Dynamic shared memory of a CTA: `words` 12-byte entry slots (32 per entry
// column of a slice), then b and the iterate of its rows, then each slice's
// offset and the lanes' entry counts.  Slices are 32 / L rows.
__host__ __device__ static inline long long resident_bytes(long long words, int rows, int slices)
{
    return words * 12 + 16ll * rows + 4ll * (slices + 1) + 64ll * slices + 32;
}

long long resident_smem_bytes(const int* rowptr, int r0, int r1, int lanes)
{
    const int rps = 32 / lanes;
    const int slices = (r1 - r0 + rps - 1) / rps;
    long long words = 0;
    for (int s = 0; s < slices; ++s) {
        int w = 0;
        for (int r = r0 + s * rps; r < r1 && r < r0 + (s + 1) * rps; ++r) {
            const int len = (rowptr[r + 1] - rowptr[r] + lanes - 1) / lanes;
            w = len > w ? len : w;
        }
        if (w > 65535) return -1;
        words += 32ll * w;
    }
    return resident_bytes(words, r1 - r0, slices);
}

// L lanes sum a row (1 or 2), as in the pipelined kernel: interleaved chains in
// stored order, then the pairwise add, so the iterates are the same bits.
//
// Entries are stored slice by slice, entry-major (entry e of lane l at
// 32 e + l): a warp's reads of S and col are consecutive.
//
// LOC also keeps each partition's max |r| (integer atomics on the sets holding a
// row, as in the pipelined kernel), in NPART slots of v.loc that start at zero:
// sweep s raises slot s % NPART, the decision of sweep s reads and clears it, and
// every CTA has seen that decision before it starts sweep s + NPART.
// Measured, 33^3 Q1 matrix, us per sweep, pipelined / resident: 8 bands 8.2 / 4.8,
// 8 boxes 10.3 / 7.0, 64 boxes 12.5 / 7.7 (the global test: 3.7); what it adds is
// the atomics and, where a warp's rows lie in several boxes, finding the peers.
template <int L, bool LOC>
__global__ void __launch_bounds__(RT, 1) k_resident(DevMat m, DevVec v, const int* __restrict__ cta_row, JacCtl* ctl,
                                                    int max_sweeps, int late)
{
    constexpr int SYNC = (MW + 1) * 32;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ double s_ss[2][MW * 32];
    __shared__ unsigned long long s_mx[2][MW * 32];
    __shared__ ResidentDecision s_dec;
    __shared__ int s_start, s_skip, s_xb, s_words, s_stop, s_done;
    __shared__ volatile int s_fail;          // written by thread 0 between the two CTA barriers of a sweep only
    __shared__ long long s_budget;
    __shared__ double* s_x[NBUF];            // (indexed in shared memory: a local copy would be re-read from L2)
    constexpr int RPS = 32 / L;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = cta_row[blockIdx.x], rows = cta_row[blockIdx.x + 1] - r0;
    const int ns = (rows + RPS - 1) / RPS;
    if (tid == 0) {
        const volatile JacCtl* c = ctl;
        init_decision(s_dec, c);
        s_xb = c->xbuf;
        s_budget = c->timeout;
        s_skip = c->fault_skip_cta;
        s_start = c->done == DONE_RUNNING && c->status == 0;
        s_fail = 0;
        s_stop = -1;
        for (int q = 0; q < NBUF; ++q) s_x[q] = v.x[q];
    }
    // ---- slice offsets: widths first (kept in the offsets' place), then their prefix sum.
    // The small arrays sit at the front, so that their places need no width.
    int* off = reinterpret_cast<int*>(smem);
    unsigned short* cnt = reinterpret_cast<unsigned short*>(off + ns + 1);
    double* sb = reinterpret_cast<double*>(smem + ((4 * (ns + 1) + 64 * ns + 15) & ~15));
    double* sy = sb + rows;
    double* sv = sy + rows;
    const bool front = 4ll * (ns + 1) + 64ll * ns + 16ll * rows + 32 <= (long long)dynamic_smem_bytes();
    __syncthreads();
    if (!s_start) return;
    if (front) {
        for (int s = warp; s < ns; s += MW + 2) {
            const int r = s * RPS + lane / L, q = lane % L;
            int my = 0;
            if (r < rows) {
                const int len = __ldg(m.rowptr + r0 + r + 1) - __ldg(m.rowptr + r0 + r);
                my = L == 1 ? len : (len > q ? (len - q + L - 1) / L : 0);
            }
            cnt[32 * s + lane] = (unsigned short)my;
            const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)my);
            if (lane == 0) off[s] = w;
        }
    }
    __syncthreads();
    if (warp == 0 && front) {
        int base = 0;
        for (int s0 = 0; s0 < ns; s0 += 32) {
            const int w = s0 + lane < ns ? off[s0 + lane] : 0;
            int inc = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            if (s0 + lane < ns) off[s0 + lane] = base + inc - w;
            base += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) {
            off[ns] = base;
            s_words = base * 32;
        }
    }
    __syncthreads();
    // the rows must fit the dynamic shared memory of the launch
    if (!front || resident_bytes(s_words, rows, ns) > (long long)dynamic_smem_bytes()) {
        if (tid == 0) atomicOr(&ctl->status, ST_CONFIG);
        return;
    }
    int* sc = reinterpret_cast<int*>(sv + s_words);
    const int xb0 = s_xb;
    for (int s = warp; s < ns; s += MW + 2) {
        const int r = s * RPS + lane / L, q = lane % L;
        if (r < rows) {
            const int kb = __ldg(m.rowptr + r0 + r) + q, my = cnt[32 * s + lane];
            double* dv = sv + 32 * off[s] + lane;
            int* dc = sc + 32 * off[s] + lane;
            for (int e = 0; e < my; ++e) {
                dv[32 * e] = __ldg(m.S64 + kb + e * L);
                dc[32 * e] = __ldg(m.col + kb + e * L);
            }
            if (q == 0) {
                sb[r] = __ldg(m.b + r0 + r);
                sy[r] = __ldcg(s_x[xb0] + r0 + r);
            }
        }
    }
    __syncthreads();

    int ksw = max_sweeps;
    if (!s_dec.test) {
        const long long rem = s_dec.k_limit - s_dec.k;
        ksw = (int)(rem < (long long)ksw ? (rem > 0 ? rem : 0) : ksw);
    }
    // slices of this math warp: one of the first X for the warps of sub-partitions
    // 1 to 3, then X + warp, X + warp + MW, ...
    constexpr int X = uneven_slices<L>();
    const int early = X && (warp & 3) ? (warp >> 2) * 3 + (warp & 3) - 1 : X;
    const bool has_early = warp < MW && early < X && early < ns;
    // math threads whose sums the spare warp adds: up to the last warp with rows
    const int nx = ns < X ? ns : X;
    const int last_early = nx ? ((nx - 1) / 3) * 4 + (nx - 1) % 3 + 1 : -1;
    const int last_round = ns - X < MW ? ns - X - 1 : MW - 1;
    const int active = 32 * ((last_early > last_round ? last_early : last_round) + 1);
    for (int i = tid; i < 2 * MW * 32; i += RT) {
        s_ss[i / (MW * 32)][i % (MW * 32)] = 0.0;
        s_mx[i / (MW * 32)][i % (MW * 32)] = 0ull;
    }
    __syncthreads();
    const long long budget = s_budget;
    unsigned long long arrivals = 0;
    unsigned long long tr_comp = 0, tr_wait = 0, tr_mark = 0;
    if (tid == 0) asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(tr_mark));
    // Bounded grid barrier by thread 0: release of the CTA's stores (ordered
    // before by the CTA barrier), arrival, acquire by the load that sees the
    // last arrival; the CTA barrier after it extends that to every thread.
    auto grid_barrier = [&]() {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        tr_comp += t - tr_mark;
        tr_mark = t;
        fence_acq_rel_gpu();
        if (s_skip != (int)blockIdx.x) atomicAdd(&ctl->bar, 1ull);
        arrivals += gridDim.x;
        const long long t0 = clock64();
        int spins = 0;
        while (ld_acquire_u64(&ctl->bar) < arrivals) {
            if ((++spins & 63) == 0) {
                if (ld_volatile_i32(&ctl->status) & ST_TIMEOUT) { s_fail = 1; break; }
                if (clock64() - t0 > budget) { atomicOr(&ctl->status, ST_TIMEOUT); s_fail = 1; break; }
            }
        }
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        tr_wait += t - tr_mark;
        tr_mark = t;
    };

    // ================================================= decisions (CTA 0's second spare warp)
    if (warp == MW + 1) {
        if (blockIdx.x != 0) return;
        for (int j = 0; j < ksw; ++j) {
            // sweep j's partials were published before the barrier of sweep j + 1
            int ok = 1;
            if (lane == 0) {
                const unsigned long long target = (unsigned long long)(j + 2) * gridDim.x;
                const long long t0 = clock64();
                while (ld_acquire_u64(&ctl->bar) < target) {
                    if (s_fail) { ok = 0; break; }
                    if (clock64() - t0 > budget) { atomicOr(&ctl->status, ST_TIMEOUT); ok = 0; break; }
                }
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            __syncwarp();                         // lane 0's acquire, for every lane
            const int done = take_decision<LOC>(s_dec, v.part + (j % NPART) * v.nslots,
                                                LOC ? v.loc + (size_t)(j % NPART) * v.nloc : nullptr, v.nloc, ctl, j,
                                                j + 1 >= ksw);
            if constexpr (LOC) __syncwarp();      // every lane's cleared maxima before the release
            // one word: the sweeps decided, and how the last of them ended
            if (lane == 0) st_release_u64(&ctl->dec_ready, (unsigned long long)(j + 1) | (unsigned long long)done << 32);
            if (done != DONE_RUNNING) break;
        }
        return;
    }
    // The word that decides sweep j, or the final one (by one lane); false on a
    // timeout.  It runs beside the math warps, which may still be reading s_fail, so
    // it leaves that flag alone: a CTA that got no decision goes on, each later wait
    // ends at once on ST_TIMEOUT, and thread 0 ends the CTA's loop, between the two
    // CTA barriers, in the first grid barrier that does not fill.
    auto await_decision = [&](int j, unsigned long long& word) -> bool {
        const long long t0 = clock64();
        int spins = 0;
        for (;;) {
            word = ld_acquire_u64(&ctl->dec_ready);
            if ((long long)(word & 0xffffffffull) > j || (word >> 32)) return true;
            if ((++spins & 63) == 0) {
                if (ld_volatile_i32(&ctl->status) & ST_TIMEOUT) return false;
                if (clock64() - t0 > budget) { atomicOr(&ctl->status, ST_TIMEOUT); return false; }
            }
        }
    };
    auto publish_sweep = [&](int j) {
        publish(s_ss[j & 1], s_mx[j & 1], active, v.part + (j % NPART) * v.nslots + blockIdx.x);
    };

    int xs_at = xb0;         // buffer of the iterate that the sweep reads
    int ran = 0;             // sweeps whose barrier has passed
    bool stopped = false;
    for (int s = 0; s < ksw; ++s) {
        const int xd_at = xs_at + 1 == NBUF ? 0 : xs_at + 1;
        if (warp < MW) {
            const double* xs = s_x[xs_at];
            double* xd = s_x[xd_at];
            double ss = 0.0;
            unsigned long long mx = 0;
            for (int sl = has_early ? early : X + warp; sl < ns; sl = sl < X ? X + warp : sl + MW) {
                const int base = 32 * off[sl] + lane, w = off[sl + 1] - off[sl];
                const int my = cnt[32 * sl + lane];
                const int r = sl * RPS + lane / L;
                const bool lead = r < rows && lane % L == 0;
                const double* pv = sv + base;
                const int* pc = sc + base;
                double acc = lead ? sb[r] : 0.0;
                [[maybe_unused]] int head = -1;
                if constexpr (LOC) head = lead ? __ldg(m.mem_head + r0 + r) : -1;
                for (int o = 0; o < w; o += CH) {
                    double xv[CH];
#pragma unroll
                    for (int u = 0; u < CH; ++u)
                        if (o + u < my) xv[u] = __ldca(xs + pc[32 * (o + u)]);
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        if (o + u >= w) break;
                        if (o + u < my) acc = __fma_rn(pv[32 * (o + u)], xv[u], acc);
                    }
                }
#pragma unroll
                for (int d = L / 2; d >= 1; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
                [[maybe_unused]] unsigned long long key = 0;
                if (lead) {
                    __stcg(xd + r0 + r, acc);
                    if constexpr (LOC) key = accumulate_residual_key(acc, sy[r], ss, mx);
                    else accumulate_residual(acc, sy[r], ss, mx);
                    sy[r] = acc;
                }
                if constexpr (LOC)
                    local_sets_update(v.loc + (size_t)(s % NPART) * v.nloc, m.mem_ptr, m.mem_part, lead ? r0 + r : -1,
                                      head, key);
            }
            if (has_early || X + warp < ns) {
                s_ss[s & 1][tid] = ss;
                s_mx[s & 1][tid] = mx;
            }
        } else {
            if (s >= 1) publish_sweep(s - 1);
            // every CTA stops in the same sweep: on the decision of sweep s - late,
            // although later ones may be known
            unsigned long long word = 0;
            if (s >= late && lane == 0 && await_decision(s - late, word) && (word >> 32) &&
                (int)(word & 0xffffffffull) - 1 == s - late) {
                s_stop = s - late;
                s_done = (int)(word >> 32);
            }
        }
        cta_sync<1, SYNC>();
        if ((stopped = s_stop >= 0)) break;
        if (tid == 0) grid_barrier();
        cta_sync<2, SYNC>();
        if (s_fail) break;
        ++ran;
        xs_at = xd_at;
    }
    if (!stopped && !s_fail && ksw > 0) {
        // the decisions of the last sweeps
        if (warp == MW) publish_sweep(ksw - 1);
        cta_sync<1, SYNC>();
        if (tid == 0) grid_barrier();
        cta_sync<2, SYNC>();
        unsigned long long word = 0;
        if (!s_fail && warp == MW && lane == 0 && await_decision(ksw - 1, word) && (word >> 32)) {
            s_stop = (int)(word & 0xffffffffull) - 1;
            s_done = (int)(word >> 32);
        }
        cta_sync<1, SYNC>();
    }
    if (tid == 0 && v.trace) {
        atomicAdd(v.trace + 4 * blockIdx.x + 0, tr_comp);
        atomicAdd(v.trace + 4 * blockIdx.x + 1, tr_wait);
        atomicAdd(v.trace + 4 * blockIdx.x + 2, (unsigned long long)ran);
    }
    if (blockIdx.x == 0 && tid == 0 && ksw > 0) {
        // x^{k+j} where sweep j's decision stopped the launch, else the last sweep's result
        const int stop_at = s_stop, j = stop_at >= 0 ? stop_at : ran;
        ctl->k = s_dec.k + j;
        ctl->xbuf = (xb0 + j) % NBUF;
        ctl->evals = s_dec.hist_at + (stop_at >= 0 ? stop_at + 1 : ran);
        if (stop_at >= 0) ctl->done = s_done;
        ctl->relres = s_dec.relres;
        ctl->res2 = s_dec.res2;
        ctl->resinf = s_dec.resinf;
        ctl->k_eval = s_dec.k_eval;
        if (LOC && s_dec.loc_part >= 0) {
            ctl->loc_part = s_dec.loc_part;
            ctl->loc_val = s_dec.loc_val;
        }
        __threadfence();
    }
}

const void* resident_kernel(int lanes, bool local_stop)
{
    if (lanes == 1)
        return local_stop ? reinterpret_cast<const void*>(&k_resident<1, true>)
                          : reinterpret_cast<const void*>(&k_resident<1, false>);
    if (lanes == 2)
        return local_stop ? reinterpret_cast<const void*>(&k_resident<2, true>)
                          : reinterpret_cast<const void*>(&k_resident<2, false>);
    return nullptr;
}

int resident_threads() { return RT; }

cudaError_t launch_resident(const void* fn, int grid, int smem, const DevMat& m, const DevVec& v, const int* cta_row,
                            JacCtl* ctl, int max_sweeps, cudaStream_t s)
{
    // the sweeps of a CTA with this much to sum (from 60^3 7-point on, 5.3 us) are longer
    // than the 3 us in which a decision is taken and read: us a sweep with two / three
    // sweeps' delay, 64^3 5.91 / 6.01, 70^3 7.04 / 7.08, 27-point 44^3 6.25 / 6.22
    int late = smem > 128 * 1024 ? 2 : 3;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(RT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {(void*)&m, (void*)&v, (void*)&cta_row, (void*)&ctl, (void*)&max_sweeps, (void*)&late};
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace jac
