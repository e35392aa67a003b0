// Adjoint g = A^T r and the fused quadratic-objective pass
//   d = A x,  f = sum_i w_i (d_i - p_i)^2,  g = A^T [2 w (d - p)]
// on the row-group layout (rg_layout.cu): the gradient of the dose objective
// that the optimiser needs every iteration (Sec. I; Sec. II-A).
//
// One CTA per SM.  Every worker warp streams its own packets of row groups
// through its own ring (rg_common.cuh) and owns a private shared-memory
// accumulator of the CTA's columns of the gradient.  Per packet:
//   1. the groups' row sums, as the dose SpMV forms them (rg_dot, rg_reduce),
//      into the warp's row buffer;
//   2. one lane per row of the packet: d, the double-float objective term
//      w (d - p)^2 and the residual r = 2 w (d - p), back into the buffer;
//   3. lane l takes union columns l, l + 32, ... of each group again: sum over
//      the group's rows of a r in packed FP32 pairs, and one read-modify-write of
//      the accumulator per column.
// The rows of a packet lie anywhere in the matrix, so their p and w (or r) are
// gathered: each lane loads those of its rows one packet ahead, with row numbers
// loaded two packets ahead, so that neither latency is waited for.  Rows without
// entries (88 % of the clinical beam's) only need d = 0 and w p^2: three more
// warps stream p and w for them while the workers compute.  A second small
// kernel (rg_finalize) adds up the CTAs' partials.
// Determinism (Sec. II-D: no float atomics, fixed reduction order): the union
// columns of a group are distinct, so no two lanes of a warp update one word
// in one instruction; each warp takes its groups in a fixed order; the CTA sums
// its warps' accumulators in warp order and the second kernel sums the CTAs'
// partials in CTA order.
#include "rg_common.cuh"

#include <algorithm>
#include <type_traits>

namespace dose {
namespace {

constexpr uint32_t kRgMaxChain = 64;                // passes of one chain
constexpr uint32_t kRgGradientSmem = 195 * 1024;
constexpr uint32_t kRgWarpBytes = kRgMaxRows * 4;   // a worker's row buffer: row sums, then residuals

struct RgParams {
    RgView A;
    const float* x;    // QUADRATIC
    const float* v0;   // QUADRATIC: p; ADJOINT: r
    const float* v1;   // QUADRATIC: w
    float* d;          // QUADRATIC, may be null
    float* g_part;     // one element per dict entry
    double* f_part;    // grid
    const uint32_t* mask;  // rows with entries
    uint32_t wmax, nw, depth, slot;
    uint32_t chain;        // RG_CHAIN_*
    int* err;
};

// Passes of different matrices that only share their inputs (the scenarios of a
// robust objective) may overlap: each lets the next start once the kernels before
// the first are done (so the next need not wait for anything), its CTAs take the
// SMs that the previous pass's have left, and it waits for the previous pass only
// before it ends, so that the last one's end is the end of all.  Three scenarios of
// an 80 x 80 x 50 plan: 105 us, 129 us with each pass finalised before the next began.
constexpr uint32_t RG_CHAIN_NEXT = 1;   // let the next pass start early
constexpr uint32_t RG_CHAIN_PREV = 2;   // started early: wait at the end

// Row numbers and per-row vectors of a warp's packets, ahead of their use: the
// packets with any flag of NEED, in the order the stream delivers them.  Lane l
// holds rows l and l + 32 of a packet (0xFFFFFFFF: none).
template <uint32_t NEED, bool QUAD>
struct RgVecs {
    const uint4* pk;
    uint32_t i, end;
    uint4 nxt;                  // entry of the packet whose row numbers are loaded next
    uint32_t row[2], rown[2];   // of the packet at hand, of the next
    float v0[2], v1[2], v0n[2], v1n[2];
    uint32_t rows2[2];          // of the one after the next

    __device__ __forceinline__ void numbers(const uint32_t* row_list, uint32_t lane, uint32_t (&r)[2]) {
        while (i < end && !(nxt.y & NEED)) {
            ++i;
            if (i < end) nxt = __ldg(pk + i);
        }
        r[0] = r[1] = 0xFFFFFFFFu;
        if (i >= end) return;
        if (lane < nxt.w) r[0] = __ldg(row_list + nxt.z + lane);
        if (nxt.w > 32 && lane + 32 < nxt.w) r[1] = __ldg(row_list + nxt.z + lane + 32);
        ++i;
        if (i < end) nxt = __ldg(pk + i);
    }
    __device__ __forceinline__ void values(const RgParams& p) {
        v0n[1] = v1n[1] = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (k && !__any_sync(0xffffffffu, rown[1] != 0xFFFFFFFFu)) break;  // most packets hold at most 32 rows
            v0n[k] = v1n[k] = 0.f;
            if (rown[k] != 0xFFFFFFFFu) {
                v0n[k] = p.v0[rown[k]];
                if (QUAD) v1n[k] = p.v1[rown[k]];
            }
        }
    }
    // From the stream's first entry on: the first two packets' row numbers.
    template <class S>
    __device__ __forceinline__ void start(const S& s, const RgView& v, uint32_t lane) {
        pk = s.pk;
        i = s.i;
        end = s.end;
        nxt = s.nxt;
        numbers(v.row_list, lane, rown);
        numbers(v.row_list, lane, rows2);
    }
    // Move on by one packet: the values loaded for it are taken over, the next
    // packet's are loaded, and the row numbers of the one after.
    __device__ __forceinline__ void next(const RgParams& p, uint32_t lane) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            row[k] = rown[k];
            v0[k] = v0n[k];
            v1[k] = v1n[k];
            rown[k] = rows2[k];
        }
        values(p);
        numbers(p.A.row_list, lane, rows2);
    }
};

// Rows without entries of the fused pass: their objective terms w p^2 (zero, and
// skipped, where p = 0 and w is finite).  Four rows per lane and step (16-byte
// loads of p and w), four steps' loads in flight; the CTA's share of the rows is
// contiguous, its row warps take it in turn.
__device__ __forceinline__ void rg_empty_rows(const RgParams& p, uint32_t z, uint32_t lane, float& hi, float& lo) {
    constexpr uint32_t U = 4;
    const uint32_t nq = (p.A.nrows + 3) / 4, full_q = p.A.nrows / 4;
    const uint32_t q0 = (uint32_t)((uint64_t)nq * blockIdx.x / gridDim.x), q1 = (uint32_t)((uint64_t)nq * (blockIdx.x + 1) / gridDim.x);
    const float4* p4 = reinterpret_cast<const float4*>(p.v0);
    const float4* w4 = reinterpret_cast<const float4*>(p.v1);
    for (uint32_t i0 = q0 + 32 * U * z + lane; i0 < q1; i0 += 32 * U * kRgRowWarps) {
        uint32_t m[U];
        float4 a[U], b[U];
#pragma unroll
        for (uint32_t k = 0; k < U; ++k) {
            const uint32_t i = i0 + 32 * k, r = 4 * i;
            m[k] = i < q1 ? (__ldg(p.mask + (r >> 5)) >> (r & 31)) & 0xFu : 0xFu;
            if (i < q1 && r + 4 > p.A.nrows) m[k] |= (0xFu << (p.A.nrows - r)) & 0xFu;  // rows past the end
            a[k] = b[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < q1 && i < full_q) {
                a[k] = p4[i];
                b[k] = w4[i];
            } else if (i < q1) {
                float t[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (uint32_t u = 0; u < 4; ++u)
                    if (r + u < p.A.nrows) {
                        t[u] = p.v0[r + u];
                        t[4 + u] = p.v1[r + u];
                    }
                a[k] = make_float4(t[0], t[1], t[2], t[3]);
                b[k] = make_float4(t[4], t[5], t[6], t[7]);
            }
        }
#pragma unroll
        for (uint32_t k = 0; k < U; ++k) {
            // nothing to add where every p is 0 and every w finite (w * 0 summed is 0
            // then, else NaN): most quads end here
            const float finite = __fmaf_rn(b[k].x, 0.f, __fmaf_rn(b[k].y, 0.f, __fmaf_rn(b[k].z, 0.f, __fmul_rn(b[k].w, 0.f))));
            const uint32_t any = (__float_as_uint(a[k].x) | __float_as_uint(a[k].y) | __float_as_uint(a[k].z) | __float_as_uint(a[k].w)) << 1;
            if (m[k] == 0xFu || (any == 0u && finite == 0.f)) continue;
            const float pv[4] = {a[k].x, a[k].y, a[k].z, a[k].w}, wv[4] = {b[k].x, b[k].y, b[k].z, b[k].w};
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u)
                if (!((m[k] >> u) & 1u) && (pv[u] != 0.0f || !(fabsf(wv[u]) < INFINITY)))
                    dev::df_add_wsq(hi, lo, wv[u], 0.0f, pv[u]);
        }
    }
}

// The accumulator updates of up to K steps of 32 union columns (the last one
// masked): all loads before the stores, since the columns are distinct.
template <int FMT, int HR, uint32_t IW, int K>
__device__ __forceinline__ void rg_scatter_steps(const unsigned char* cols, const unsigned char* vals, uint32_t n,
                                                 uint32_t lane, float* gw, const uint64_t (&r)[HR / 2]) {
    RgVal<FMT, HR> q[K];
    uint32_t c[K];
    const bool last = 32 * (K - 1) + lane < n;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t u = 32 * k + lane;
        c[k] = 0;
        q[k].zero();
        if (k < K - 1 || last) {
            c[k] = rg_col<IW>(cols, u);
            q[k].load(vals + u * RgVal<FMT, HR>::kBytes);
        }
    }
    float g[K];
#pragma unroll
    for (int k = 0; k < K; ++k) g[k] = gw[c[k]];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float lo, hi;
        if constexpr (HR == 4) {  // one after the other (the stored-row order's sums; no longer than packed pairs)
            float a[4], b[4];
            dev::f2_split(q[k].pair(0), a[0], a[1]);
            dev::f2_split(q[k].pair(1), a[2], a[3]);
            dev::f2_split(r[0], b[0], b[1]);
            dev::f2_split(r[1], b[2], b[3]);
            float t = __fmul_rn(a[0], b[0]);
            t = __fmaf_rn(a[1], b[1], t);
            t = __fmaf_rn(a[2], b[2], t);
            g[k] = __fadd_rn(g[k], __fmaf_rn(a[3], b[3], t));
        } else {
            uint64_t t = dev::f2_mul(q[k].pair(0), r[0]);
#pragma unroll
            for (int i = 1; i < HR / 2; ++i) t = dev::f2_fma(q[k].pair(i), r[i], t);
            dev::f2_split(t, lo, hi);
            g[k] = __fadd_rn(g[k], __fadd_rn(lo, hi));
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (k < K - 1 || last) gw[c[k]] = g[k];
}

template <int FMT, int HR, uint32_t IW>
__device__ __forceinline__ void rg_scatter(const unsigned char* cols, const unsigned char* vals, uint32_t n, uint32_t lane,
                                           float* gw, const uint64_t (&r)[HR / 2]) {
    constexpr uint32_t VB = RgVal<FMT, HR>::kBytes;
    while (n > 128) {
        rg_scatter_steps<FMT, HR, IW, 4>(cols, vals, 128, lane, gw, r);
        cols += 128 * IW;
        vals += 128 * VB;
        n -= 128;
    }
    switch ((n + 31) >> 5) {
        case 1: rg_scatter_steps<FMT, HR, IW, 1>(cols, vals, n, lane, gw, r); break;
        case 2: rg_scatter_steps<FMT, HR, IW, 2>(cols, vals, n, lane, gw, r); break;
        case 3: rg_scatter_steps<FMT, HR, IW, 3>(cols, vals, n, lane, gw, r); break;
        default: rg_scatter_steps<FMT, HR, IW, 4>(cols, vals, n, lane, gw, r); break;
    }
}

// Bound by issue (51 % active) and each warp's chain from load to scatter, at 3.7 warps
// per scheduler: more do not fit beside their private accumulators.  With rg_finalize,
// 6.3e7 entries (200 x 200 x 120 voxels) take 72 us and 1.5e8 (the clinical beam) 0.128
// ms, against 98 us and 0.168 ms with groups of four consecutive rows and one ring of
// stages per CTA (48 M warp instructions on the smaller beam, 39 M now).
template <int FMT, int HR, uint32_t IW, int MODE>
__global__ void __launch_bounds__((kRgMaxWarps + kRgRowWarps) * 32, 1) rg_kernel(const __grid_constant__ RgParams p) {
    constexpr bool QUAD = MODE == ADJ_MODE_QUADRATIC;
    constexpr bool FP8 = FMT == DOSE_FMT_FP8E4M3_ROWSCALE;
    constexpr uint32_t NEED = QUAD ? (RG_FORWARD | RG_SCATTER) : (uint32_t)RG_SCATTER;
    constexpr uint32_t VB = RgVal<FMT, HR>::kBytes;
    constexpr uint32_t RL = 32 / HR;  // lanes of a row
    extern __shared__ __align__(128) unsigned char smem[];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NW = p.nw;
    double* fred = reinterpret_cast<double*>(smem + 1024 + 512);  // per-warp objective
    unsigned char* zeros = smem + kRgHeader;                      // QUAD: read by the bulk stores of empty rows
    unsigned char* bufs = zeros + (QUAD ? kRgZeroBytes : 0);
    const uint32_t gstride = round_up(p.wmax, 32);
    float* gacc = reinterpret_cast<float*>(bufs + NW * kRgWarpBytes);  // NW x gstride
    float* xs = gacc + (size_t)NW * gstride;                           // QUAD: the CTA's x and a zero
    unsigned char* slot_base = reinterpret_cast<unsigned char*>(xs) + (QUAD ? round_up((p.wmax + 1) * 4, 128) : 0);
    const uint32_t cta = blockIdx.x, T = blockDim.x, t = threadIdx.x;
    RgStream<NEED> S;
    RgVecs<NEED, QUAD> V;
    RgDict C;
    C.range(p.A, cta);
    if (warp < NW) S.range(p.A, cta, NW, warp);
    if (QUAD) C.load(t, T);
    if (warp < NW) {
        S.entry();
        V.start(S, p.A, lane);
        S.start(warp, p.depth, p.slot, smem, slot_base, lane);
    }
    const uint32_t db = C.db, nc = C.nc;
    float4* g4 = reinterpret_cast<float4*>(gacc);
    for (uint32_t j = t; j < NW * gstride / 4; j += T) g4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!(p.chain & RG_CHAIN_PREV)) rg_wait_previous();
    if (p.chain & RG_CHAIN_NEXT) rg_let_next_start();
    if (QUAD) {
        C.each(t, T, [&](uint32_t c) { return __ldcg(p.x + c); }, [&](uint32_t j, float v) { xs[j] = v; });
        if (t == 0) xs[nc] = 0.f;
    }
    if (warp < NW) V.values(p);
    __syncthreads();

    float f_hi = 0.f, f_lo = 0.f;  // this lane's objective terms, double-float
    if (QUAD && warp >= NW) {
        if (p.d && warp == NW) {
            rg_fill_zeros(zeros, lane);
            rg_zero_rows(p.A.zero_runs, p.A.n_zero_runs, reinterpret_cast<unsigned char*>(p.d), 4, zeros, lane);
        }
        rg_empty_rows(p, warp - NW, lane, f_hi, f_lo);
    }
    if (warp < NW) {
        float* gw = gacc + (size_t)warp * gstride;
        float* rbuf = reinterpret_cast<float*>(bufs + warp * kRgWarpBytes);
        uint64_t acc[HR / 2];
        while (S.pending) {
            V.next(p, lane);
            if (!S.wait(p.err)) break;  // recorded in the error word; the results are then worthless but in bounds
            const RgSlotView<FMT, HR, IW> P(S.slot());
            if (rg_packet_ok(P, S.slot(), p.slot, p.A.nrows, nc, lane, p.err)) {
                const uint32_t fl = S.flag();
                if (QUAD && (fl & RG_FORWARD)) {
                    uint32_t u = 0;
                    for (uint32_t g = 0; g < P.ng; ++g) {
                        const uint32_t n = P.gn[g];
                        if (!(fl & RG_CARRY_IN)) {
#pragma unroll
                            for (int i = 0; i < HR / 2; ++i) acc[i] = 0ull;
                        }
                        rg_dot<FMT, HR, IW>(P.cols + u * IW, P.vals + u * VB, n, lane, xs, nc, acc);
                        u += n;
                        if (fl & RG_CARRY_OUT) break;  // a piece is alone in its packet
                        const float sum = rg_reduce<HR>(acc, lane);
                        if ((lane & (RL - 1)) == 0) rbuf[g * HR + lane / RL] = sum;
                    }
                    __syncwarp();
                }
                // one lane per row: residuals
                if (QUAD ? (fl & (RG_FORWARD | RG_CARRY_OUT)) == RG_FORWARD : true) {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const uint32_t i = lane + 32 * k;
                        if (32 * k < P.ng * HR && i < P.ng * HR) {
                            const bool has = V.row[k] != 0xFFFFFFFFu;
                            const float rsc = FP8 ? P.scales[i] : 1.f;
                            float rr;
                            if (QUAD) {
                                const float sum = rbuf[i], wv = V.v1[k], pv = V.v0[k];
                                const float dv = FMT == DOSE_FMT_U16_SCALE ? __fmul_rn(p.A.scale, sum)
                                                                           : (FP8 ? __fmul_rn(rsc, sum) : sum);
                                rr = __fmul_rn(__fmul_rn(__fmul_rn(2.0f, wv), __fsub_rn(dv, pv)), rsc);
                                if (has) {
                                    dev::df_add_wsq(f_hi, f_lo, wv, dv, pv);
                                    if (p.d) p.d[V.row[k]] = dv;
                                }
                            } else {
                                rr = FP8 ? __fmul_rn(V.v0[k], rsc) : V.v0[k];
                            }
                            rbuf[i] = has ? rr : 0.f;
                        }
                    }
                    __syncwarp();
                }
                if (fl & RG_SCATTER) {
                    uint32_t u = 0;
                    for (uint32_t g = 0; g < P.ng; ++g) {
                        const uint32_t n = P.gn[g];
                        uint64_t r[HR / 2];
#pragma unroll
                        for (int i = 0; i < HR / 4; ++i) {
                            const ulonglong2 t = reinterpret_cast<const ulonglong2*>(rbuf + g * HR)[i];
                            r[2 * i] = t.x;
                            r[2 * i + 1] = t.y;
                        }
                        rg_scatter<FMT, HR, IW>(P.cols + u * IW, P.vals + u * VB, n, lane, gw, r);
                        u += n;
                        __syncwarp();  // this group's updates precede the next group's
                    }
                }
            }
            S.done(lane);
        }
    }
    if (QUAD) {
        double f_lane = (double)f_hi + (double)f_lo;
        for (uint32_t o = 16; o > 0; o >>= 1) f_lane += __shfl_xor_sync(0xffffffffu, f_lane, o);
        if (lane == 0) fred[warp] = f_lane;
    }
    if (!(p.chain & RG_CHAIN_NEXT)) rg_let_next_start();
    __syncthreads();
    for (uint32_t j = t; j < nc; j += T) {
        float sum = gacc[j];
        for (uint32_t w2 = 1; w2 < NW; ++w2) sum = __fadd_rn(sum, gacc[(size_t)w2 * gstride + j]);
        p.g_part[db + j] = sum;
    }
    if (QUAD && t == 0) {
        double sum = 0.0;
        for (uint32_t w2 = 0; w2 < NW + kRgRowWarps; ++w2) sum += fred[w2];
        p.f_part[cta] = sum;
    }
    if (p.chain & RG_CHAIN_PREV) rg_wait_previous();
}

// Second kernel of the row-group passes: g_j = s * (sum of the partials of the CTAs
// that see column j, in CTA order), and the optional projected-gradient step on x;
// block 0 also writes f = the CTAs' objective partials, added in one fixed order.
struct RgFin {
    const float* g_part;
    const uint32_t* col_ptr;  // where column j's partials lie in g_part (CTA order)
    const uint32_t* col_pos;
    uint32_t nparts, ncols;
    float scale;
    float* g;
    float* x_update;
    float eta;
    const double* f_part;
    double* f;
};

template <uint32_t N>
struct RgFins {
    RgFin q[N];  // block row y finishes pass y
};

template <uint32_t N>
__global__ void __launch_bounds__(256) rg_finalize(const __grid_constant__ RgFins<N> all) {
    const RgFin& q = all.q[blockIdx.y];
    __shared__ float part[8][33];
    __shared__ double red[256];
    const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31, j = blockIdx.x * 32 + lane;
    uint32_t k = 0, k1 = 0;
    if (j < q.ncols && q.nparts) {
        k = __ldg(q.col_ptr + 8 * (size_t)j + w);
        k1 = __ldg(q.col_ptr + 8 * (size_t)j + w + 1);
    }
    rg_let_next_start();
    rg_wait_previous();  // the main kernel's partials (and it may update x, which that reads)
    // warp w adds the partials of CTAs w, w + 8, ... in order; four loads in flight
    float t = 0.f;
    for (; k + 4 <= k1; k += 4) {
        float v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) v[u] = __ldcg(q.g_part + __ldg(q.col_pos + k + u));
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) t = __fadd_rn(t, v[u]);
    }
    for (; k < k1; ++k) t = __fadd_rn(t, __ldcg(q.g_part + __ldg(q.col_pos + k)));
    part[w][lane] = t;
    __syncthreads();
    if (w == 0 && j < q.ncols) {
        float tot = part[0][lane];
        for (uint32_t i = 1; i < 8; ++i) tot = __fadd_rn(tot, part[i][lane]);
        tot = __fmul_rn(q.scale, tot);
        if (q.g) q.g[j] = tot;
        if (q.x_update) {
            const float xn = __fsub_rn(q.x_update[j], __fmul_rn(q.eta, tot));
            q.x_update[j] = xn > 0.f ? xn : 0.f;
        }
    }
    if (!q.f || blockIdx.x) return;
    double s = 0.0;
    for (uint32_t i = threadIdx.x; i < q.nparts; i += 256) s += __ldcg(q.f_part + i);
    red[threadIdx.x] = s;
    __syncthreads();
    for (uint32_t st = 128; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *q.f = red[0];
}

template <int FMT, int HR, uint32_t IW, int MODE>
cudaError_t launch_t(const dose_matrix* A, const RgParams& p, size_t smem, cudaStream_t s) {
    return rg_launch(rg_kernel<FMT, HR, IW, MODE>, p, A->rg.grid, 32 * (p.nw + (MODE == ADJ_MODE_QUADRATIC ? kRgRowWarps : 0)),
                     smem, s);
}

template <int FMT, int MODE>
cudaError_t launch_shape(const dose_matrix* A, const RgParams& p, size_t smem, cudaStream_t s) {
    const RowGroups& R = rg_of(A, MODE == ADJ_MODE_QUADRATIC ? RG_DEAL_FUSED : RG_DEAL_ADJOINT);
    if constexpr (value_bytes(FMT) <= 2) {
        if (R.hr == 8) return R.iw == 2 ? launch_t<FMT, 8, 2, MODE>(A, p, smem, s) : launch_t<FMT, 8, 4, MODE>(A, p, smem, s);
    }
    return R.iw == 2 ? launch_t<FMT, 4, 2, MODE>(A, p, smem, s) : launch_t<FMT, 4, 4, MODE>(A, p, smem, s);
}

template <int MODE>
cudaError_t launch_fmt(const dose_matrix* A, const RgParams& p, size_t smem, cudaStream_t s) {
    switch (A->fmt) {
        case DOSE_FMT_U16_SCALE: return launch_shape<DOSE_FMT_U16_SCALE, MODE>(A, p, smem, s);
        case DOSE_FMT_BF16: return launch_shape<DOSE_FMT_BF16, MODE>(A, p, smem, s);
        case DOSE_FMT_F16: return launch_shape<DOSE_FMT_F16, MODE>(A, p, smem, s);
        case DOSE_FMT_F32: return launch_shape<DOSE_FMT_F32, MODE>(A, p, smem, s);
        case DOSE_FMT_FP8E4M3_ROWSCALE: return launch_shape<DOSE_FMT_FP8E4M3_ROWSCALE, MODE>(A, p, smem, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// Gradient warps: as many as fit with their accumulators and rings.  The
// stored-row order fixes how many warps share a CTA's groups, as many as fitted
// beside whole stages and windows of it, and takes deeper rings of its smaller
// packets instead.
uint32_t rg_gradient_warps(const dose_matrix* A, const AdjTuning& t, bool quad, uint32_t* depth, size_t* smem) {
    const RowGroups& R = rg_of(A, quad ? RG_DEAL_FUSED : RG_DEAL_ADJOINT);
    if (!R.built || R.forward_only) return 0;
    uint32_t d = std::min<uint32_t>(t.rg_stages, kRgMaxDepth);
    const size_t fixed = kRgHeader + (quad ? kRgZeroBytes + round_up((R.wmax + 1) * 4, 128) : 0);
    const size_t base = kRgWarpBytes + (size_t)round_up(R.wmax, 32) * 4, per = base + (size_t)d * R.slot;
    if (fixed + per > kMaxSmemPerBlock) return 0;
    uint32_t most = t.rg_warps ? std::min<uint32_t>(t.rg_warps, kRgMaxWarps) : kRgMaxWarps;
    if (R.keep) most = std::min(most, R.keep_nw);
    // at most 195 KB, so that 60 instead of 28 KB of the SM's memory stay L1 for the
    // gathered vectors and the stream of the rows without entries: 77.0 -> 71.2 us on
    // the 200 x 200 x 120 beam with 12 instead of 14 warps (163 KB: 78.7 us)
    const size_t room = R.keep || fixed + per > kRgGradientSmem ? kMaxSmemPerBlock : kRgGradientSmem;
    const uint32_t nw = (uint32_t)std::min<size_t>(most, (room - fixed) / per);
    if (R.keep) d = (uint32_t)std::min<size_t>(kRgMaxDepth, (kMaxSmemPerBlock - fixed - nw * base) / ((size_t)nw * R.slot));
    if (depth) *depth = d;
    if (smem) *smem = fixed + nw * (base + (size_t)d * R.slot);
    return nw;
}

bool rg_active(const dose_matrix* A, bool quad) {
    return A->adj_tuning.layout != 1 && rg_gradient_warps(A, A->adj_tuning, quad, nullptr, nullptr) > 0;
}

// Bytes of one fused pass: the packets once, the non-empty bits, p and w of every
// row, d if written, x in, g out, and the CTA partials written and read once.
static uint64_t rg_parts(const RowGroups& R) { return 8ull * (R.wmax * (uint64_t)R.grid); }
uint64_t rg_fused_bytes(const dose_matrix* A, bool with_d) {
    const RowGroups& R = rg_of(A, RG_DEAL_FUSED);
    const uint64_t nr = A->nrows, nc = A->ncols, P = R.grid;
    return R.data_bytes + (nr + 7) / 8 + 8 * nr + (with_d ? 4 * nr : 0) + 8 * nc + rg_parts(R) + 8 * P + 8;
}

// Bytes of one dose_spmv on the layout: the packets once, x in (once), d out
// (every row).
uint64_t rg_spmv_bytes(const dose_matrix* A) { return A->rg.data_bytes + 4ull * A->ncols + 4ull * A->nrows; }

uint64_t rg_adjoint_bytes(const dose_matrix* A) {
    return A->rg.data_bytes + 4ull * A->nrows + 4ull * A->ncols + rg_parts(A->rg);
}

static cudaError_t launch_main(const dose_matrix* A, bool quad, const float* x, const float* p, const float* w,
                               const float* r, float* d, uint32_t chain, cudaStream_t s) {
    const int which = quad ? RG_DEAL_FUSED : RG_DEAL_ADJOINT;
    const RowGroups& R = rg_of(A, which);
    size_t smem = 0;
    RgParams prm;
    prm.nw = rg_gradient_warps(A, A->adj_tuning, quad, &prm.depth, &smem);
    if (!prm.nw || R.deal[which].nw != prm.nw) return cudaErrorInvalidConfiguration;
    if (A->nrows == 0) return cudaSuccess;
    prm.A = rg_view(A, which);
    prm.x = x;
    prm.v0 = quad ? p : r;
    prm.v1 = w;
    prm.d = d;
    prm.g_part = R.g_part;
    prm.f_part = A->f_part;
    prm.mask = R.mask;
    prm.wmax = R.wmax;
    prm.slot = R.slot;
    prm.chain = chain;
    prm.err = A->err;
    return quad ? launch_fmt<ADJ_MODE_QUADRATIC>(A, prm, smem, s) : launch_fmt<ADJ_MODE_ADJOINT>(A, prm, smem, s);
}

static RgFin finish_of(const dose_matrix* A, bool quad, double* f, float* g, float* x_update, float eta) {
    const RowGroups& R = rg_of(A, quad ? RG_DEAL_FUSED : RG_DEAL_ADJOINT);
    RgFin q;
    q.g_part = R.g_part;
    q.col_ptr = R.col_ptr;
    q.col_pos = R.col_pos;
    q.nparts = A->nrows > 0 ? R.grid : 0;
    q.ncols = A->ncols;
    q.scale = A->fmt == DOSE_FMT_U16_SCALE ? A->scale : 1.0f;
    q.g = g;
    q.x_update = x_update;
    q.eta = eta;
    q.f_part = A->f_part;
    q.f = quad ? f : nullptr;
    return q;
}

template <uint32_t N>
static cudaError_t launch_finish(const RgFins<N>& q, uint32_t n, bool early, cudaStream_t s) {
    const uint32_t nc = q.q[0].ncols;
    return rg_launch(rg_finalize<N>, q, dim3(nc ? (nc + 31) / 32 : 1, n), 256, 0, s, early);
}

cudaError_t launch_rg(const dose_matrix* A, int mode, const float* x, const float* p, const float* w, const float* r,
                      float* d, double* f, float* g, float* x_update, float eta, cudaStream_t s) {
    const bool quad = mode == ADJ_MODE_QUADRATIC;
    const cudaError_t e = launch_main(A, quad, x, p, w, r, d, 0, s);
    if (e != cudaSuccess) return e;
    RgFins<1> q;
    q.q[0] = finish_of(A, quad, f, g, x_update, eta);
    // early after the adjoint (18.7 -> 16.8 us on a plan of 780 spots); after the
    // fused pass, whose CTAs leave no registers for a block of this kernel, an
    // ordinary launch: waiting there early cost 14 us (27 -> 41 us, same plan)
    return launch_finish(q, 1, !quad, s);
}

// The fused passes of n matrices of one shape, overlapped where they may be
// (distinct matrices, all on this layout, none empty); false: not applicable.
bool rg_chain_applies(const dose_matrix* const* A, uint32_t n) {
    if (n < 2 || n > kRgMaxChain) return false;
    for (uint32_t k = 0; k < n; ++k) {
        if (!rg_active(A[k], true) || !A[k]->nrows) return false;
        for (uint32_t j = 0; j < k; ++j)
            if (A[j] == A[k]) return false;  // they would share one set of partials
    }
    return true;
}

cudaError_t launch_rg_chain(const dose_matrix* const* A, uint32_t n, const float* x, const float* p, const float* w,
                            double* f, float* g, cudaStream_t s) {
    RgFins<kRgMaxChain> q;
    for (uint32_t k = 0; k < n; ++k) {
        const cudaError_t e = launch_main(A[k], true, x, p, w, nullptr, nullptr,
                                          (k + 1 < n ? RG_CHAIN_NEXT : 0) | (k ? RG_CHAIN_PREV : 0), s);
        if (e != cudaSuccess) return e;
        q.q[k] = finish_of(A[k], true, f + k, g + (size_t)k * A[k]->ncols, nullptr, 0.f);
    }
    return launch_finish(q, n, false, s);
}

}  // namespace dose
