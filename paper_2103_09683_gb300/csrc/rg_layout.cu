// Host side of the row-group layout (the kernels are in rg_spmm.cu and
// rg_kernel.cu; the stored form is described at RowGroups in
// dose_internal.cuh).
//
// The gradient of the dose objective needs g = A^T r every iteration (Sec. I;
// Sec. II-A: A fixed, x changing).  Scattering a_ij r_i entry by entry costs a
// shared-memory read-modify-write per entry.  Neighbouring voxels of a dose
// matrix see almost the same spots, so rows that see the same spots are grouped
// and each group stores, for the union of its rows' columns, the rows' values
// side by side (stored zeros where a row has no entry).
//
// Order of the rows.  The rows of a group need not be consecutive: the groups
// carry their row numbers.  On a voxel grid the nearest spot sets belong to the
// neighbour along the beam (the same lateral position, one plane on), so the
// line and plane strides of the grid are looked for in the matrix itself (the
// row distances at which sampled rows overlap most) and the rows are taken
// plane by plane inside lateral tiles of 8 x 8 voxels, or, where several beams
// cross, in cubes of 2 x 2 x 2 voxels.  A CTA's share of that order is a
// compact region of the patient, so it sees few distinct spots.  Stored bytes
// per entry (u16, 16-bit columns) on the 200 x 200 x 120 pencil beam: 3.01 with
// four consecutive rows per group, 2.48 with eight rows along the beam; on a
// three-beam plan 2.91 and 2.67 (cubes).  Where no strides are found the rows
// keep their order, or, if that groups them better, go by their first and last
// column.
//
// Built once at create from the validated host CSR and the stored codes, by
// several threads (a CTA's share of the groups is one unit of work).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <exception>
#include <memory>
#include <new>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "dose_internal.cuh"

namespace dose {
namespace {

uint32_t round_up16(uint32_t v) { return (v + 15) / 16 * 16; }

constexpr uint32_t kMaxRowEntries = 4096;  // longest row of the gradient passes (and most columns of a packet)
constexpr uint32_t kMaxForwardRow = 32768; // ... of a layout for the forward passes alone
constexpr uint32_t kTile = 8;              // voxels per side of the tiles the rows are ordered by
// Dealing cost of a group, in steps of 32 columns: its reduction, outputs and its share
// of its packet.  By instructions it is 7 steps in dose_spmv (140 against 21 a step) and 6
// in the fused pass, less with FP64 or 16 vectors, whose steps are longer.  Measured with
// costs of 4 / 3 / 2: dose on 1.5e8 entries 66.7 / 66.3 / 66.5 us, fused pass on 6.3e7
// entries 71.2 / 71.7 / 72.9, FP64 dose 62.2 / 60.6 / 58.2, three matrices times 16 vectors
// 142.5 / 138.4 / 137.7.  3 gives the FP64 and batched forms most of their gain.
constexpr uint64_t kGroupCost = 3;

// rg_tile_union where the caller gave none: about 40 KB of union columns and values
// (a stage of the stored-row order, below), never less than the longest row, so that
// the reported value can be given back.
uint32_t default_tile_u(uint32_t max_row_len, uint32_t iw, uint32_t es) {
    const uint32_t def = std::max(512u, std::min(8192u, 40960 / (iw + 4 * es) / 32 * 32));
    return std::max(def, (max_row_len + 31) / 32 * 32);
}

cudaError_t rg_upload(void** dst, const void* src, size_t bytes, size_t alloc_bytes) {
    alloc_bytes = std::max<size_t>(alloc_bytes, 16);
    cudaError_t e = dev_malloc(dst, alloc_bytes);
    if (e != cudaSuccess) return e;
    if (alloc_bytes > bytes) {
        e = cudaMemset(static_cast<unsigned char*>(*dst) + bytes, 0, alloc_bytes - bytes);
        if (e != cudaSuccess) return e;
    }
    if (bytes) e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
    return e;
}

// fn(i, thread) for i < n on several threads (at most `most`); false if a thread could
// not get memory (no exception leaves a thread).
constexpr uint32_t kMaxThreads = 32;
template <class F>
bool parallel_for(uint32_t n, F fn, uint32_t most = kMaxThreads) {
    const uint32_t nt = std::max(1u, std::min({n, most, kMaxThreads, std::thread::hardware_concurrency()}));
    std::atomic<uint32_t> next{0};
    std::atomic<bool> ok{true};
    auto work = [&](uint32_t thread) {
        try {
            for (uint32_t i; ok && (i = next.fetch_add(1)) < n;) fn(i, thread);
        } catch (const std::exception&) {
            ok = false;
        }
    };
    std::vector<std::thread> th;
    th.reserve(nt);
    for (uint32_t t = 1; t < nt; ++t) {
        try {
            th.emplace_back(work, t);
        } catch (const std::exception&) {
            break;  // fewer threads
        }
    }
    work(0);
    for (std::thread& t : th) t.join();
    return ok;
}

struct Csr {
    const uint32_t* rp;
    const uint32_t* col;
    const unsigned char* vals;
    const float* scales;  // FP8
    uint32_t nrows, ncols, es;
    uint32_t max_union;   // union columns of a group
};

// Marks of the columns of the group being formed.
struct Marks {
    std::vector<uint32_t> stamp;
    uint32_t gen = 0;
    explicit Marks(uint32_t n) : stamp(std::max<uint32_t>(n, 1), 0u) {}
    void reset() { ++gen; }
    bool add(uint32_t c) {
        if (stamp[c] == gen) return false;
        stamp[c] = gen;
        return true;
    }
    bool has(uint32_t c) const { return stamp[c] == gen; }
};

// Greedy grouping of rows[0 .. n) in order: a row joins the open group of up to
// hr rows while it brings at most 0.7 of its columns (plus 8) as new ones and the
// union grows by at most half (plus 8) of the larger of the two.  A row that starts a new cube (cube != null) joins only a group of fewer than hr
// / 2 rows, so that groups stay aligned with the cubes.
// emit(first, count, union columns).
template <class E>
void form_groups(const Csr& A, const uint32_t* rows, const uint8_t* cube, size_t n, uint32_t hr, Marks& mk,
                 std::vector<uint32_t>& U, E emit) {
    const uint64_t max_union = A.max_union;
    size_t first = 0;
    uint32_t cnt = 0;
    U.clear();
    mk.reset();
    for (size_t i = 0; i < n; ++i) {
        const uint32_t r = rows[i], kb = A.rp[r], ke = A.rp[r + 1], len = ke - kb;
        if (cnt) {
            bool join = cnt < hr && !(cube && cube[i] && 2 * cnt >= hr);
            if (join) {
                uint32_t fresh = 0;
                for (uint32_t k = kb; k < ke; ++k) fresh += !mk.has(A.col[k]);
                const uint64_t nu = U.size() + fresh;
                join = 10 * (uint64_t)fresh <= 7 * (uint64_t)len + 80 &&
                       2 * nu <= 3 * std::max<uint64_t>(U.size(), len) + 16 && nu <= max_union;
            }
            if (!join) {
                emit(first, cnt, U);
                cnt = 0;
                U.clear();
                mk.reset();
            }
        }
        if (!cnt) first = i;
        for (uint32_t k = kb; k < ke; ++k)
            if (mk.add(A.col[k])) U.push_back(A.col[k]);
        ++cnt;
    }
    if (cnt) emit(first, cnt, U);
}

// Estimated time of groups of hr rows: the stored bytes and a group's fixed work
// in bytes.
constexpr uint64_t kGroupBytes = 512;
struct Estimate {
    uint64_t bytes = 0, entries = 0;
    double per_entry() const { return entries ? (double)bytes / (double)entries : 1e30; }
};
void estimate_add(const Csr& A, const std::vector<uint32_t>& rows, uint32_t hr, uint32_t iw, Marks& mk,
                  std::vector<uint32_t>& U, Estimate& e) {
    for (uint32_t r : rows) e.entries += A.rp[r + 1] - A.rp[r];
    form_groups(A, rows.data(), nullptr, rows.size(), hr, mk, U,
                [&](size_t, uint32_t, const std::vector<uint32_t>& u) { e.bytes += u.size() * (hr * A.es + iw) + kGroupBytes; });
}

// Strides of the voxel grid, looked for in the matrix: for sampled rows, the row
// distances at which other rows share most of their columns.
struct Strides {
    uint32_t line = 0, plane = 0;  // rows per voxel line and per plane (0: not found)
};

Strides find_strides(const Csr& A, const std::vector<uint32_t>& rows, const uint32_t* cmin, const uint32_t* cmax) {
    Strides S;
    const size_t n = rows.size();
    if (n < 64) return S;
    constexpr uint32_t kSamples = 24, kKeep = 256;
    struct Hit {
        uint32_t dist;
        double sim;
    };
    std::vector<std::vector<Hit>> hits(kSamples);
    // samples of typical length in the first half of the rows (their neighbours a
    // plane on must exist)
    const bool ok = parallel_for(kSamples, [&](uint32_t s, uint32_t) {
        size_t i = n / 8 + (size_t)((uint64_t)n * s / (2 * kSamples));
        uint32_t best = rows[i];
        for (size_t k = i; k < std::min(n, i + 64); ++k)  // the longest row nearby: inside the beam
            if (A.rp[rows[k] + 1] - A.rp[rows[k]] > A.rp[best + 1] - A.rp[best]) best = rows[k];
        const uint32_t r = best, len = A.rp[r + 1] - A.rp[r];
        if (len < 4) return;
        Marks mk(A.ncols);
        mk.reset();
        for (uint32_t k = A.rp[r]; k < A.rp[r + 1]; ++k) mk.add(A.col[k]);
        const uint32_t slack = (cmax[r] - cmin[r]) / 2 + 2;
        std::vector<Hit> h;
        uint64_t budget = std::max<uint64_t>(4000000, 12000ull * len);  // entries looked at per sample
        for (size_t k = std::upper_bound(rows.begin(), rows.end(), r) - rows.begin(); k < n; ++k) {
            const uint32_t q = rows[k], lq = A.rp[q + 1] - A.rp[q];
            if (q - r < 2 || 4 * lq < 3 * len || 4 * len < 3 * lq) continue;
            const uint32_t dl = cmin[q] > cmin[r] ? cmin[q] - cmin[r] : cmin[r] - cmin[q];
            const uint32_t dh = cmax[q] > cmax[r] ? cmax[q] - cmax[r] : cmax[r] - cmax[q];
            if (dl > slack || dh > slack) continue;
            if (budget < lq) break;
            budget -= lq;
            uint32_t common = 0;
            for (uint32_t e = A.rp[q]; e < A.rp[q + 1]; ++e) common += mk.has(A.col[e]);
            const double sim = (double)common / (double)(len + lq - common);
            if (sim >= 0.3) h.push_back({q - r, sim});
        }
        std::stable_sort(h.begin(), h.end(), [](const Hit& a, const Hit& b) { return a.sim > b.sim; });
        if (h.size() > kKeep) h.resize(kKeep);
        hits[s] = std::move(h);
    });
    if (!ok) return S;
    std::unordered_map<uint32_t, double> sum;  // summed similarity of each distance
    for (const std::vector<Hit>& h : hits)
        for (const Hit& x : h) sum[x.dist] += x.sim;
    auto of = [&](uint64_t d) {
        const auto it = d <= 0xFFFFFFFFull ? sum.find((uint32_t)d) : sum.end();
        return it == sum.end() ? 0.0 : it->second;
    };
    // the distance with the most similar rows: a plane (one beam: the next voxel
    // along it) or a line.  Ties go to the smaller distance.
    auto best_of = [&](auto take) {
        Hit m{0, 0.0};
        for (const auto& [d, v] : sum)
            if (take(d, v) && (v > m.sim || (v == m.sim && d < m.dist))) m = {d, v};
        return m;
    };
    const Hit top = best_of([&](uint32_t d, double) { return d >= 3; });
    if (top.sim < 3.0) return S;  // no distance that several samples agree on
    // it is a line if a multiple of it comes back stronger than its double
    const Hit pl = best_of([&](uint32_t d, double v) {
        return d % top.dist == 0 && d >= 3 * (uint64_t)top.dist && v >= 0.6 * top.sim && v > of(2ull * top.dist);
    });
    if (pl.dist) {
        S.line = top.dist;
        S.plane = pl.dist;
        return S;
    }
    S.plane = top.dist;
    S.line = best_of([&](uint32_t d, double v) {
                 return d >= 3 && top.dist % d == 0 && top.dist >= 3 * (uint64_t)d && v >= 0.2 * top.sim;
             }).dist;
    return S;
}

// Row orders the groups may be formed in.
enum Order { ORDER_MATRIX, ORDER_PLANES, ORDER_CUBES, ORDER_COLUMNS };

// rows in the given order.  Counting sorts by a key; the rows of one key keep
// their order.  cube: marks the rows that start a new cube (ORDER_CUBES).
bool order_rows(const Csr& A, std::vector<uint32_t>& rows, Order o, const Strides& S, const uint32_t* cmin,
                const uint32_t* cmax, std::vector<uint8_t>* cube) {
    if (o == ORDER_MATRIX) return true;
    if (o == ORDER_COLUMNS) {
        std::stable_sort(rows.begin(), rows.end(), [&](uint32_t a, uint32_t b) {
            return cmin[a] != cmin[b] ? cmin[a] < cmin[b] : cmax[a] < cmax[b];
        });
        return true;
    }
    const uint64_t L = S.line ? S.line : S.plane, P = S.plane;
    const uint64_t ny = S.line ? P / L : 1, nz = (A.nrows + P - 1) / P;
    const uint64_t tx = (L + kTile - 1) / kTile, ty = (ny + kTile - 1) / kTile, tz = (nz + kTile - 1) / kTile;
    // neighbours in the order are neighbours in the grid (every other line of
    // cubes runs backwards), so a group that reaches past its cube stays alike
    auto key = [&](uint32_t r) -> uint64_t {
        const uint64_t z = r / P, q = r % P, y = q / L, x = q % L;
        if (o == ORDER_PLANES) {
            if (!S.line) return q;
            const uint64_t v = y % kTile, u = x % kTile;
            return ((y / kTile) * tx + x / kTile) * (kTile * kTile) + v * kTile + ((v & 1) ? kTile - 1 - u : u);
        }
        // cubes of 2 x 2 x 2 voxels inside tiles of 8 x 8 x 8
        const uint64_t tile = ((z / kTile) * ty + y / kTile) * tx + x / kTile, c = kTile / 2;
        const uint64_t w = (z % kTile) / 2, v0 = (y % kTile) / 2, v = (w & 1) ? c - 1 - v0 : v0, u = (x % kTile) / 2;
        return tile * (c * c * c) + (w * c + v) * c + ((w * c + v) & 1 ? c - 1 - u : u);
    };
    const uint64_t nkeys = o == ORDER_PLANES ? (S.line ? tx * ty * kTile * kTile : P) : tx * ty * tz * 64;
    if (nkeys > 4ull * A.nrows + (1u << 20)) return false;
    std::vector<uint32_t> start(nkeys + 1, 0), out(rows.size());
    for (uint32_t r : rows) ++start[key(r) + 1];
    for (uint64_t k = 0; k < nkeys; ++k) start[k + 1] += start[k];
    for (uint32_t r : rows) out[start[key(r)]++] = r;
    if (o == ORDER_PLANES)  // down one lateral position, up the next
        for (uint64_t k = 1; k < nkeys; k += 2) std::reverse(out.begin() + start[k - 1], out.begin() + start[k]);
    rows.swap(out);
    if (o == ORDER_CUBES && cube) {
        cube->assign(rows.size(), 0);
        for (size_t i = 1; i < rows.size(); ++i) (*cube)[i] = key(rows[i]) != key(rows[i - 1]);
    }
    return true;
}

// The order and group height with the fewest estimated bytes on samples: around
// 48 rows each, the rows that the order would put there.
void choose_order(const Csr& A, const std::vector<uint32_t>& rows, const Strides& S, const uint32_t* cmin,
                  const uint32_t* cmax, uint32_t iw, uint32_t hr_hi, Order& order, uint32_t& hr) {
    constexpr uint32_t kSamples = 48;
    const size_t n = rows.size();
    std::vector<Order> orders{ORDER_MATRIX};
    if (S.plane) orders.push_back(ORDER_PLANES);
    if (S.line) orders.push_back(ORDER_CUBES);
    std::vector<uint32_t> by_col;
    if (!S.plane) {  // (else the grid orders know more)
        orders.push_back(ORDER_COLUMNS);
        by_col = rows;
        order_rows(A, by_col, ORDER_COLUMNS, S, cmin, cmax, nullptr);
    }
    // on several threads where rows have thousands of entries (1.05e8 entries in 1.35e5
    // rows: 48 -> 8 ms on eight); a millisecond of work otherwise, less than the threads
    const bool threads = A.rp[A.nrows] / std::max<size_t>(n, 1) >= 512;
    std::vector<Estimate> est(orders.size() * kSamples * 2);  // of 4 and of 8 rows
    std::vector<std::unique_ptr<Marks>> marks(kMaxThreads);
    const bool ok = parallel_for((uint32_t)orders.size() * kSamples, [&](uint32_t task, uint32_t thread) {
        if (!marks[thread]) marks[thread].reset(new Marks(A.ncols));
        Marks& mk = *marks[thread];
        const Order o = orders[task / kSamples];
        const size_t i = (size_t)((uint64_t)n * (2 * (task % kSamples) + 1) / (2 * kSamples));
        std::vector<uint32_t> U, set;
        if (o == ORDER_MATRIX || o == ORDER_COLUMNS) {
            const std::vector<uint32_t>& src = o == ORDER_MATRIX ? rows : by_col;
            for (size_t k = i; k < std::min(n, i + 64); ++k) set.push_back(src[k]);
        } else if (o == ORDER_PLANES) {
            const uint64_t z0 = rows[i] / S.plane, zb = z0 > 128 ? z0 - 128 : 0;
            for (uint64_t z = zb; z < zb + 256; ++z) {
                const uint64_t r = z * S.plane + rows[i] % S.plane;
                if (r >= A.nrows) break;
                if (A.rp[r + 1] > A.rp[r]) set.push_back((uint32_t)r);
            }
        } else {
            const uint64_t z = rows[i] / S.plane / 2 * 2, q = rows[i] % S.plane, y = q / S.line / 2 * 2, x = q % S.line / 8 * 8,
                           ny = S.plane / S.line;
            for (uint64_t c = 0; c < 4; ++c)
                for (uint64_t k = 0; k < 8; ++k) {
                    const uint64_t zz = z + (k >> 2), yy = y + ((k >> 1) & 1), xx = x + 2 * c + (k & 1);
                    const uint64_t r = zz * S.plane + yy * S.line + xx;
                    if (yy < ny && xx < S.line && r < A.nrows && A.rp[r + 1] > A.rp[r]) set.push_back((uint32_t)r);
                }
        }
        for (uint32_t h : {4u, 8u})
            if (h <= hr_hi) estimate_add(A, set, h, iw, mk, U, est[2 * task + h / 8]);
    }, threads ? kMaxThreads : 1);
    if (!ok) throw std::bad_alloc();
    double best = 1e30;
    order = ORDER_MATRIX;
    hr = hr_hi;
    for (size_t j = 0; j < orders.size(); ++j)
        for (uint32_t h : {4u, 8u}) {
            Estimate e;
            for (uint32_t s = 0; s < kSamples; ++s) {
                e.bytes += est[2 * (j * kSamples + s) + h / 8].bytes;
                e.entries += est[2 * (j * kSamples + s) + h / 8].entries;
            }
            if (h <= hr_hi && e.per_entry() < 0.98 * best) {
                best = e.per_entry();
                order = orders[j];
                hr = h;
            }
        }
}

struct Grp {
    uint32_t first, cnt;  // rows[first .. first + cnt)
    uint32_t nu;
    uint64_t uoff;        // its union in the segment's column list
    // in steps of 32 columns; all but the last piece of a long group come twice
    uint64_t cost(uint32_t max_u, bool again) const {
        const uint64_t steps = (nu + 31) / 32, np = (nu + max_u - 1) / max_u;
        return kGroupCost * np + steps + (again ? kGroupCost * (np - 1) + steps * (np - 1) / (2 * np) : 0);
    }
};

// ---- the stored-row order (RowGroups::keep).
//
// The objective is an FP64 number whose digits below FP32 rounding follow the
// order in which each row's products, and each column's contributions, are
// added; a projected-gradient loop carries them on from step to step.  Over many
// rows such differences average out (2e-10 of f over 2.5e5 rows), over few they
// do not (up to 3e-9 on small plans, 1e-8 after 100 steps).  So the fused pass of
// small matrices (kRgKeepRows, kRgKeepPlanRows) keeps one fixed order, whatever order
// the other passes' groups take: groups of up to four consecutive non-empty rows,
// each group's columns in one order.  These alone set the doses, and with them f (its
// terms are added in double-float and FP64).
// The gradient's rounding, which a projected-gradient loop feeds back, follows the
// deal of the groups as well.  Small matrices keep that too: stages of consecutive
// groups, dealt to CTAs by column windows, and the groups of a stage round-robin to
// the warps, a step further at each stage.  From kRgKeepDealRows rows on, where its
// uneven shares and small packets (a shared-memory slot for each of fifteen warps, so
// unions cut in pieces that are read twice) made the fused pass slower than the
// stage-ring kernels, the kept groups are dealt like the other layout's.
// Objective on F32 beams and three-beam plans, stage rings / kept deal / this: 1.7e5 rows
// F32 38.6 / 39.2 / 32.6 us; plans of 1.5e5 rows u16 39.1 / 39.1 / 36.9, F32 49.4 / 51.3 /
// 41.6; of 2.2e5 rows u16 59.6 / 65.8 / 57.9, F32 79.6 / 93.0 / 67.7.  Same d, f to 6e-16.
// FP8, whose unions fit the packets, is faster on the kept deal (1.7e5 rows: 33.0 /
// 28.9 / 30.9) and stays on it.

// Groups of up to four consecutive non-empty rows within 255 rows whose union
// stays within 320 columns and grows by at most half.
constexpr uint32_t kKeepUnion = 320, kKeepSpan = 255, kKeepStageGroups = 64;
template <class E>
void form_kept_groups(const Csr& A, const std::vector<uint32_t>& rows, E emit) {
    Marks mk(A.ncols);
    std::vector<uint32_t> U;
    size_t first = 0;
    uint32_t cnt = 0;
    for (size_t i = 0; i < rows.size(); ++i) {
        const uint32_t r = rows[i], kb = A.rp[r], ke = A.rp[r + 1], len = ke - kb;
        bool join = cnt && cnt < 4 && r - rows[first] <= kKeepSpan;
        if (join) {
            uint64_t nu = U.size();
            for (uint32_t k = kb; k < ke; ++k) nu += !mk.has(A.col[k]);
            join = nu <= kKeepUnion && 2 * nu <= 3 * std::max<uint64_t>(U.size(), len);
        }
        if (!join) {
            if (cnt) emit(first, cnt, U);
            first = i;
            cnt = 0;
            U.clear();
            mk.reset();
        }
        for (uint32_t k = kb; k < ke; ++k)
            if (mk.add(A.col[k])) U.push_back(A.col[k]);
        ++cnt;
    }
    if (cnt) emit(first, cnt, U);
}

// Stages of kept groups and their deal to CTAs.  A stage ends at tile_u union
// columns, tile_rows rows or 64 groups, and where its column range would more
// than double (the voxel order wrapping across the beam); the tighter of two such
// cuts is taken where its windows are narrower.
Schedule kept_schedule(const Csr& A, const std::vector<uint32_t>& rows, const std::vector<Grp>& G,
                       const std::vector<uint32_t>& U, uint32_t iw, uint32_t grid, uint32_t tile_u, uint32_t tile_rows,
                       bool fp8) {
    const uint32_t ng = (uint32_t)G.size();
    std::vector<uint32_t> lo(ng, 0xFFFFFFFFu), hi(ng, 0);
    uint32_t span_max = 0;
    for (uint32_t g = 0; g < ng; ++g) {
        for (uint32_t k = 0; k < G[g].nu; ++k) {
            lo[g] = std::min(lo[g], U[G[g].uoff + k]);
            hi[g] = std::max(hi[g], U[G[g].uoff + k]);
        }
        span_max = std::max(span_max, hi[g] - lo[g]);
    }
    const uint64_t span_cap = (uint64_t)span_max * 3 / 2;
    const uint32_t row_bytes = 8 + (fp8 ? 4 : 0);
    auto cut = [&](bool tight, Schedule& S, std::vector<DealItem>& items) {
        for (uint32_t g = 0; g < ng;) {
            StageDesc D{};
            D.row0 = rows[G[g].first];
            D.ne0 = g;
            uint32_t u = 0, l = 0xFFFFFFFFu, h = 0;
            for (; g < ng; ++g) {
                const uint32_t last = rows[G[g].first + G[g].cnt - 1];
                if (g > D.ne0) {
                    if (last >= D.row0 + tile_rows || u + G[g].nu > tile_u || g - D.ne0 >= kKeepStageGroups) break;
                    const uint32_t nl = std::min(l, lo[g]), nh = std::max(h, hi[g]);
                    if (nh - nl > 2 * std::max(h - l, hi[g] - lo[g]) + 64 && (tight || nh - nl > span_cap)) break;
                }
                l = std::min(l, lo[g]);
                h = std::max(h, hi[g]);
                u += G[g].nu;
                D.row1 = last + 1;
            }
            D.ne1 = g;
            items.push_back({(uint32_t)S.desc.size(), (uint32_t)S.desc.size() + 1, l, h,
                             (uint64_t)u * (iw + 4 * A.es) + 16ull * (D.ne1 - D.ne0) +
                                 (uint64_t)(D.row1 - D.row0) * row_bytes + 256ull * (D.ne1 - D.ne0)});
            S.desc.push_back(D);
        }
    };
    Schedule S1, S2;
    std::vector<DealItem> i1, i2;
    cut(false, S1, i1);
    cut(true, S2, i2);
    deal_items(S1, i1, grid, A.ncols, true, true);
    deal_items(S2, i2, grid, A.ncols, true, true);
    return S2.wwidth < S1.wwidth ? S2 : S1;
}

// Order the local columns loc[0 .. n) of one packet's group for the kernels:
// position 32 it + l is read by lane l in step it, and its gather of x and its
// update of the gradient accumulator touch shared-memory bank loc mod 32, so
// the columns of one step should differ mod 32.  Greedy: residues with the most
// columns first, each column to the step with the most free positions among
// those that do not hold its residue yet.  perm: the chosen order as indices
// into loc.
struct BankOrder {
    std::vector<uint32_t> cap, has, at;
    uint16_t step_of[kMaxRowEntries];
    // blocks: also arrange each step for the batched SpMM's gathers
    void operator()(const uint32_t* loc, uint32_t n, uint32_t* perm, bool blocks) {
        const uint32_t steps = (n + 31) / 32;
        if (n <= 1) {
            if (n) perm[0] = 0;
            return;
        }
        uint32_t cnt[33] = {0}, bank[32], item[kMaxRowEntries];
        for (uint32_t i = 0; i < n; ++i) ++cnt[(loc[i] & 31u) + 1];
        for (uint32_t b = 0; b < 32; ++b) bank[b] = b;
        std::stable_sort(bank, bank + 32, [&](uint32_t a, uint32_t b) { return cnt[a + 1] > cnt[b + 1]; });
        uint32_t start[33];
        start[0] = 0;
        for (uint32_t b = 0; b < 32; ++b) start[b + 1] = start[b] + cnt[b + 1];
        uint32_t fill[32];
        std::copy(start, start + 32, fill);
        for (uint32_t i = 0; i < n; ++i) item[fill[loc[i] & 31u]++] = i;  // loc ascends, so do the buckets
        cap.assign(steps, 32u);
        has.assign(steps, 0u);
        at.assign(steps, 0u);
        cap[steps - 1] = n - 32 * (steps - 1);
        for (uint32_t bi = 0; bi < 32; ++bi) {
            const uint32_t b = bank[bi];
            for (uint32_t k = start[b]; k < start[b + 1]; ++k) {
                int best = -1;
                for (uint32_t s = 0; s < steps; ++s)
                    if (cap[s] && !((has[s] >> b) & 1u) && (best < 0 || cap[s] > cap[best])) best = (int)s;
                if (best < 0)
                    for (uint32_t s = 0; s < steps; ++s)
                        if (cap[s] && (best < 0 || cap[s] > cap[best])) best = (int)s;
                step_of[item[k]] = (uint16_t)best;
                --cap[best];
                has[best] |= 1u << b;
            }
        }
        for (uint32_t i = 0; i < n; ++i) perm[32 * step_of[i] + at[step_of[i]]++] = i;  // ascending inside a step
        if (!blocks) return;
        // inside a step: eight consecutive positions with columns that differ mod 8
        // where that is possible (the batched SpMM's 16-byte X gathers: without it 37 %
        // of its shared-memory wavefronts were bank conflicts): the first column left of
        // each residue, then (no other residues left) the first columns left
        for (uint32_t s = 0; s < steps; ++s) {
            uint32_t* p = perm + 32 * s;
            uint32_t of[8] = {0}, tmp[32], left = 0, k = 0;  // positions left, by residue and in all
            for (uint32_t i = 0; i < at[s]; ++i) of[loc[p[i]] & 7u] |= 1u << i;
            for (uint32_t q = 0; q < 8; ++q) left |= of[q];
            while (left) {
                uint32_t pick = 0, in_block = 0;
                for (uint32_t q = 0; q < 8; ++q) pick |= of[q] & (0u - of[q]);
                while (in_block < 8 && left) {
                    const uint32_t from = pick ? pick : left, bit = from & (0u - from), i = (uint32_t)__builtin_ctz(bit);
                    of[loc[p[i]] & 7u] &= ~bit;
                    left &= ~bit;
                    pick &= ~bit;
                    tmp[k++] = p[i];
                    ++in_block;
                }
            }
            std::copy(tmp, tmp + at[s], p);
        }
    }
};

// One CTA's share, written by one thread.
struct CtaOut {
    std::vector<unsigned char> data;
    std::vector<uint4> pk;        // offset (16-byte units) inside this CTA's data, size | flags, row_list, rows
    std::vector<uint32_t> rows;   // the packets' rows
    std::vector<uint32_t> cost;   // dealing cost of each packet
    std::vector<uint32_t> dict;   // global columns, ascending
    std::vector<uint32_t> tag;    // (stored-row order) each packet's warp
    uint32_t slot = 0;            // largest packet
};


// cap: union columns a packet of several groups may hold; max_u: ... a packet of
// one.  kept: a group's columns in the order of the stored-row layout; tags (each
// group's warp): packets hold groups of one warp.
void write_cta(const Csr& A, uint32_t hr, uint32_t iw, uint32_t cap, uint32_t max_u, const uint32_t* rows,
               const std::vector<std::pair<const Grp*, const uint32_t*>>& groups, bool kept, const std::vector<uint32_t>* tags, bool again,
               std::vector<uint32_t>& pos, std::vector<uint32_t>& seen, uint32_t gen, CtaOut& out) {
    const bool fp8 = A.scales != nullptr;
    // distinct columns
    for (const auto& g : groups)
        for (uint32_t k = 0; k < g.first->nu; ++k) {
            const uint32_t c = g.second[k];
            if (seen[c] != gen) {
                seen[c] = gen;
                out.dict.push_back(c);
            }
        }
    std::sort(out.dict.begin(), out.dict.end());
    for (uint32_t i = 0; i < out.dict.size(); ++i) pos[out.dict[i]] = i;  // global column -> local
    std::vector<uint32_t> loc, perm;
    std::vector<size_t> where(out.dict.size());  // where a column's values lie in out.data
    BankOrder order;
    struct Piece {
        const Grp* g;
        uint32_t lo, n;  // its columns: loc[lo .. lo + n) in the order of loc
    };
    std::vector<Piece> open;
    std::vector<std::vector<uint32_t>> open_loc;  // each piece's local columns in stored order
    uint32_t open_u = 0;
    auto put_values = [&](const Grp& g) {
        for (uint32_t s = 0; s < g.cnt; ++s) {
            const uint32_t r = rows[g.first + s];
            for (uint32_t k = A.rp[r]; k < A.rp[r + 1]; ++k) {
                unsigned char* o = out.data.data() + where[pos[A.col[k]]] + (size_t)s * A.es;
                if (A.es == 2)
                    std::memcpy(o, A.vals + 2 * (size_t)k, 2);
                else if (A.es == 1)
                    *o = A.vals[k];
                else
                    std::memcpy(o, A.vals + 4 * (size_t)k, 4);
            }
        }
    };
    // values: write the groups' values (else, for a piece, only note where they go)
    auto flush = [&](uint32_t flags, bool values) -> size_t {
        const uint32_t ng = (uint32_t)open.size();
        const RgPacket L = rg_packet(ng, open_u, hr, iw, A.es, fp8);
        const size_t base = out.data.size();
        out.data.resize(base + L.bytes, 0);
        unsigned char* p = out.data.data() + base;
        uint32_t* h = reinterpret_cast<uint32_t*>(p);
        h[0] = ng;
        h[1] = open_u;
        uint32_t u = 0;
        uint64_t cost = 1;
        for (uint32_t gi = 0; gi < ng; ++gi) {
            const Grp& g = *open[gi].g;
            const std::vector<uint32_t>& lc = open_loc[gi];
            const uint32_t n = (uint32_t)lc.size();
            h[4 + gi] = n;
            cost += kGroupCost + (n + 31) / 32;
            uint32_t* ro = reinterpret_cast<uint32_t*>(p + L.rows) + gi * hr;
            float* so = reinterpret_cast<float*>(p + L.scales) + gi * hr;
            for (uint32_t s = 0; s < hr; ++s) {
                ro[s] = s < g.cnt ? rows[g.first + s] : 0xFFFFFFFFu;
                if (fp8) so[s] = s < g.cnt ? A.scales[ro[s]] : 0.f;
            }
            for (uint32_t k = 0; k < n; ++k) {
                if (iw == 2)
                    reinterpret_cast<uint16_t*>(p + L.cols)[u + k] = (uint16_t)lc[k];
                else
                    reinterpret_cast<uint32_t*>(p + L.cols)[u + k] = lc[k];
                where[lc[k]] = base + L.vals + ((size_t)u + k) * hr * A.es;
            }
            if (values) put_values(g);
            u += n;
        }
        const uint32_t* ro = reinterpret_cast<const uint32_t*>(p + L.rows);
        out.pk.push_back(make_uint4((uint32_t)(base / 16), (L.bytes / 16) | flags, (uint32_t)out.rows.size(), ng * hr));
        out.rows.insert(out.rows.end(), ro, ro + ng * hr);
        out.cost.push_back((uint32_t)cost);
        out.slot = std::max(out.slot, L.bytes);
        open.clear();
        open_loc.clear();
        open_u = 0;
        return out.pk.size() - 1;
    };
    const uint32_t max_g = kRgMaxRows / hr;
    std::vector<uint32_t> res;
    for (size_t gi = 0; gi < groups.size(); ++gi) {
        const auto& gp = groups[gi];
        const Grp& g = *gp.first;
        loc.resize(g.nu);
        for (uint32_t k = 0; k < g.nu; ++k) loc[k] = pos[gp.second[k]];
        std::sort(loc.begin(), loc.end());
        perm.resize(g.nu);
        if (kept) {  // banks by global column, over the whole union
            res.resize(g.nu);
            for (uint32_t k = 0; k < g.nu; ++k) res[k] = out.dict[loc[k]];
            order(res.data(), g.nu, perm.data(), false);
        }
        const uint32_t np = (g.nu + max_u - 1) / max_u;
        if (!open.empty() && (np > 1 || open_u + g.nu > cap || open.size() >= max_g || (tags && (*tags)[gi] != (*tags)[gi - 1]))) {
            flush(RG_FORWARD | RG_SCATTER, true);
            if (tags) out.tag.resize(out.pk.size(), (*tags)[gi - 1]);
        }
        std::vector<size_t> piece_pk;
        for (uint32_t i = 0; i < np; ++i) {
            // pieces of whole 32-column steps, as equal as they can be
            const uint32_t steps = (g.nu + 31) / 32;
            const uint32_t lo = 32 * (uint32_t)((uint64_t)steps * i / np);
            const uint32_t hi = i + 1 == np ? g.nu : 32 * (uint32_t)((uint64_t)steps * (i + 1) / np);
            std::vector<uint32_t> lc(hi - lo);
            if (!kept) {
                order(loc.data() + lo, hi - lo, perm.data() + lo, true);
                for (uint32_t k = lo; k < hi; ++k) perm[k] += lo;
            }
            for (uint32_t k = 0; k < hi - lo; ++k) lc[k] = loc[perm[lo + k]];
            open.push_back({&g, lo, hi - lo});
            open_loc.push_back(std::move(lc));
            open_u += hi - lo;
            if (np > 1)
                piece_pk.push_back(flush(RG_FORWARD | (i ? RG_CARRY_IN : 0u) | (i + 1 < np ? RG_CARRY_OUT : RG_SCATTER), false));
        }
        // the values of a group of several pieces, once over its rows (piece by piece, each
        // over all entries, the layout of the beam shaped like the paper's liver beam 1
        // took 3.5 times as long to write)
        if (np > 1) put_values(g);
        // a group of several pieces: its residuals are known after the last one, so
        // the earlier pieces come once more for the scatter
        for (uint32_t i = 0; again && i + 1 < np; ++i) {
            const uint4 q = out.pk[piece_pk[i]];
            out.pk.push_back(make_uint4(q.x, (q.y & RG_SIZE_MASK) | RG_SCATTER | RG_AGAIN, q.z, q.w));
            out.cost.push_back(out.cost[piece_pk[i]]);
        }
        if (tags) out.tag.resize(out.pk.size(), (*tags)[gi]);
    }
    if (!open.empty()) flush(RG_FORWARD | RG_SCATTER, true);
    if (tags && !tags->empty()) out.tag.resize(out.pk.size(), tags->back());
}

}  // namespace

// Byte offsets of the parts of a packet.
RgPacket rg_packet(uint32_t ng, uint32_t nu, uint32_t hr, uint32_t iw, uint32_t es, bool scales) {
    RgPacket L;
    L.rows = 16 + round_up16(4 * ng);
    L.scales = L.rows + 4 * hr * ng;
    L.cols = L.scales + (scales ? 4 * hr * ng : 0);
    L.vals = L.cols + round_up16(nu * iw);
    L.bytes = L.vals + round_up16(nu * hr * es);
    return L;
}

void free_row_groups(RowGroups& R) {
    cudaFree(R.data);
    cudaFree(R.row_list);
    cudaFree(R.dict);
    cudaFree(R.dict_begin);
    cudaFree(R.col_ptr);
    cudaFree(R.col_pos);
    cudaFree(R.zero_runs);
    cudaFree(R.mask);
    cudaFree(R.g_part);
    for (RgDeal& d : R.deal) {
        cudaFree(d.begin);
        cudaFree(d.pk);
        d = RgDeal();
    }
    const uint32_t grid = R.grid;
    R = RowGroups();
    R.grid = grid;
}

// Deal the packets of every CTA to nw warps (kept order: as its stages say, see
// above): the costliest first, each to the
// warp with the least so far (a matrix of 2e7 entries has about eight packets
// per warp: contiguous runs of equal cost left the busiest warp 25-45 % above
// the mean, this 3-8 %).  The pieces of one group stay together; a warp takes
// its packets in their order in memory.
cudaError_t rg_deal(const RowGroups& R, uint32_t nw, RgDeal& D) {
    const uint32_t np = (uint32_t)R.host_pk.size();
    std::vector<uint32_t> b((size_t)R.grid * nw + 1, 0);
    std::vector<uint4> pk;
    pk.reserve(np);
    struct Unit {
        uint32_t p, n;
        uint64_t cost;
    };
    std::vector<Unit> units;
    std::vector<std::vector<uint32_t>> mine(nw);
    std::vector<uint64_t> load(nw);
    for (uint32_t c = 0; c < R.grid; ++c) {
        units.clear();
        for (uint32_t p = R.cta_pk[c]; p < R.cta_pk[c + 1];) {
            Unit u{p, 1, R.pk_cost[p]};
            while (p + u.n < R.cta_pk[c + 1] && R.pk_chain[p + u.n]) u.cost += R.pk_cost[p + u.n++];
            units.push_back(u);
            p += u.n;
        }
        std::vector<uint32_t> by(units.size());
        for (uint32_t i = 0; i < by.size(); ++i) by[i] = i;
        std::stable_sort(by.begin(), by.end(), [&](uint32_t x, uint32_t y) { return units[x].cost > units[y].cost; });
        std::fill(load.begin(), load.end(), 0);
        for (auto& v : mine) v.clear();
        if (R.keep)
            for (uint32_t i = 0; i < by.size(); ++i) by[i] = i;
        for (uint32_t i : by) {
            const uint32_t w = R.keep ? R.keep_tag[units[i].p] % nw
                                      : (uint32_t)(std::min_element(load.begin(), load.end()) - load.begin());
            load[w] += units[i].cost;
            mine[w].push_back(i);
        }
        for (uint32_t w = 0; w < nw; ++w) {
            std::sort(mine[w].begin(), mine[w].end());
            for (uint32_t i : mine[w])
                for (uint32_t k = 0; k < units[i].n; ++k) pk.push_back(R.host_pk[units[i].p + k]);
            b[(size_t)c * nw + w + 1] = (uint32_t)pk.size();
        }
    }
    uint32_t* dev_b = nullptr;
    uint4* dev_p = nullptr;
    cudaError_t e = rg_upload(reinterpret_cast<void**>(&dev_b), b.data(), b.size() * 4, b.size() * 4);
    if (e == cudaSuccess) e = rg_upload(reinterpret_cast<void**>(&dev_p), pk.data(), pk.size() * 16, pk.size() * 16 + 16);
    if (e != cudaSuccess) {
        cudaFree(dev_b);
        cudaFree(dev_p);
        return e;
    }
    D.begin = dev_b;
    D.pk = dev_p;
    D.nw = nw;
    return cudaSuccess;
}

bool build_row_groups(dose_matrix* A, RowGroups& R, bool keep, const uint32_t* rp, const uint32_t* col,
                      const unsigned char* vals, const float* scales, std::string* why, cudaError_t* err) {
    *err = cudaSuccess;
    const uint32_t nrows = A->nrows, ncols = A->ncols;
    const uint32_t es = value_bytes(A->fmt);
    const Csr M{rp, col, vals, A->fmt == DOSE_FMT_FP8E4M3_ROWSCALE ? scales : nullptr, nrows, ncols, es,
                A->max_row_len > kMaxRowEntries ? 2 * kMaxForwardRow : kMaxRowEntries};
    // Rows past the gradient passes' limit: a layout for the forward passes alone,
    // if it stores less than the CSR arrays (below).  The beam shaped like the
    // paper's liver beam 1 has rows of 5000 of its 68,000 spots: dose 206 us on CSR.
    const bool forward_only = A->max_row_len > kMaxRowEntries;
    // (the indices are positions in a CTA's list, which fits shared memory and so
    // 16 bits wherever the forward passes run; the wide form is kept where a
    // handle's gradient passes have reported it)
    R.iw = ncols <= 65536u || forward_only ? 2u : 4u;
    const std::string too_long = "a row has " + std::to_string(A->max_row_len) + " entries; row groups hold at most " +
                                 std::to_string(kMaxRowEntries) + " columns";
    if (forward_only && (keep || A->max_row_len > kMaxForwardRow || A->adj_tuning.layout == 2)) {
        *why = too_long;
        return false;
    }
    const uint32_t tile_u =
        A->adj_tuning.rg_tile_u ? A->adj_tuning.rg_tile_u : forward_only ? 0u : default_tile_u(A->max_row_len, R.iw, es);
    if (A->max_row_len > tile_u && A->adj_tuning.rg_tile_u && !forward_only) {
        *err = cudaErrorInvalidValue;
        return false;
    }
    const uint32_t grid = R.grid;
    try {
        std::vector<uint32_t> rows;
        rows.reserve(nrows / 4 + 64);
        for (uint32_t r = 0; r < nrows; ++r)
            if (rp[r + 1] > rp[r]) rows.push_back(r);
        const uint32_t* cmin = A->host_row_cmin.data();
        const uint32_t* cmax = A->host_row_cmax.data();
        // columns a packet may hold: the slot of a warp is a few KB
        const uint32_t cap = tile_u ? std::min(tile_u, kRgDefaultUnion) : kRgDefaultUnion;
        uint32_t max_u = cap;
        std::vector<std::vector<Grp>> sg;
        std::vector<std::vector<uint32_t>> su;
        Order order = ORDER_MATRIX;
        bool ok = true;
        Schedule KS;
        const bool kept_deal = keep && (rows.size() < kRgKeepDealRows || es == 1);
        if (keep) {
            R.hr = 4;
            sg.resize(1);
            su.resize(1);
            form_kept_groups(M, rows, [&](size_t first, uint32_t cnt, const std::vector<uint32_t>& u) {
                sg[0].push_back({(uint32_t)first, cnt, (uint32_t)u.size(), su[0].size()});
                su[0].insert(su[0].end(), u.begin(), u.end());
            });
            if (kept_deal) {
                const AdjTuning& t = A->adj_tuning;
                KS = kept_schedule(M, rows, sg[0], su[0], R.iw, grid, tile_u, t.rg_tile_rows, M.scales != nullptr);
                // the warps that fitted beside this order's stages and windows; packets as
                // large as two slots each leave room for
                auto r128 = [](uint64_t v) { return (v + 127) / 128 * 128; };
                const uint64_t own = r128(4ull * KS.wwidth), most = t.rg_warps ? std::min<uint32_t>(t.rg_warps, kRgMaxWarps) : kRgMaxWarps;
                const uint64_t stage = 128 + r128(kKeepStageGroups * 16) + r128((tile_u + 16) * R.iw) + r128((tile_u + 8ull) * 4 * es) +
                                       (M.scales ? 3 : 2) * r128((t.rg_tile_rows + 8) * 4);
                const uint64_t rest = 3072 + r128(4ull * KS.wwidth + 4) + t.rg_stages * stage;
                R.keep_nw = (uint32_t)(rest + own <= kMaxSmemPerBlock ? std::min<uint64_t>(most, (kMaxSmemPerBlock - rest) / own) : most);
                const uint64_t room = (kMaxSmemPerBlock - std::min<uint64_t>(kMaxSmemPerBlock, 8192 + own)) / R.keep_nw;
                max_u = (uint32_t)std::min<uint64_t>(kMaxRowEntries, room > own + 2560 ? (room - own - 2048) / 2 / (4 * es + R.iw) / 32 * 32 : 0);
                max_u = std::max(max_u, 128u);
            } else {
                // shares of the other calls' order: a CTA then sees a compact region
                std::vector<uint32_t> sorted = rows, rank(nrows, 0);
                Strides S;
                S.line = A->rg.line;
                S.plane = A->rg.plane;
                order_rows(M, sorted, (Order)A->rg.order, S, cmin, cmax, nullptr);
                for (uint32_t i = 0; i < sorted.size(); ++i) rank[sorted[i]] = i;
                std::sort(sg[0].begin(), sg[0].end(),
                          [&](const Grp& a, const Grp& b) { return rank[rows[a.first]] < rank[rows[b.first]]; });
            }
        } else {
            const Strides S = find_strides(M, rows, cmin, cmax);
            R.line = S.line;
            R.plane = S.plane;
            choose_order(M, rows, S, cmin, cmax, R.iw, es <= 2 ? 8 : 4, order, R.hr);
            std::vector<uint8_t> cube;
            if (!order_rows(M, rows, order, S, cmin, cmax, &cube)) order = ORDER_MATRIX;
            const uint32_t hr = R.hr;

            // groups, formed segment by segment (four segments per CTA, about equal entries)
            const uint32_t nseg = std::max<uint32_t>(1, std::min<uint32_t>(4 * grid, (uint32_t)(rows.size() / 256)));
            std::vector<size_t> seg(nseg + 1, rows.size());
            {
                uint64_t run = 0;
                uint32_t s = 0;
                for (size_t i = 0; i < rows.size(); ++i) {
                    while (s < nseg && run * nseg >= (uint64_t)s * A->nnz) seg[s++] = i;
                    run += rp[rows[i] + 1] - rp[rows[i]];
                }
                while (s < nseg) seg[s++] = rows.size();
                seg[0] = 0;
            }
            sg.resize(nseg);
            su.resize(nseg);
            ok = parallel_for(nseg, [&](uint32_t s, uint32_t) {
                Marks mk(ncols);
                std::vector<uint32_t> U;
                form_groups(M, rows.data() + seg[s], cube.empty() ? nullptr : cube.data() + seg[s], seg[s + 1] - seg[s], hr, mk, U,
                            [&](size_t first, uint32_t cnt, const std::vector<uint32_t>& u) {
                                sg[s].push_back({(uint32_t)(seg[s] + first), cnt, (uint32_t)u.size(), su[s].size()});
                                su[s].insert(su[s].end(), u.begin(), u.end());
                            });
            });
            if (!ok) throw std::bad_alloc();
        }
        const uint32_t hr = R.hr;
        // contiguous runs of groups of equal cost, one per CTA
        uint64_t total = 0, n_groups = 0, n_union = 0;
        for (const auto& v : sg)
            for (const Grp& g : v) {
                total += g.cost(cap, !forward_only);
                n_union += g.nu;
                ++n_groups;
            }
        const uint64_t per_entry = es + ((A->flags & DOSE_CREATE_U16_INDEX) ? 2u : 4u);
        if (forward_only && n_union * (hr * es + R.iw) >= (uint64_t)A->nnz * per_entry) {
            *why = too_long;
            return false;
        }
        std::vector<std::vector<std::pair<const Grp*, const uint32_t*>>> cta(grid);
        std::vector<std::vector<uint32_t>> tag(kept_deal ? grid : 0);
        if (kept_deal) {
            for (uint32_t c = 0; c < grid; ++c)
                for (uint32_t w = 0; w < R.keep_nw; ++w)
                    for (uint32_t d = KS.cta_begin[c]; d < KS.cta_begin[c + 1]; ++d) {
                        // the stage's groups go round-robin, a warp further at each stage
                        const uint32_t rot = (d - KS.cta_begin[c]) % R.keep_nw, first = (w + R.keep_nw - rot) % R.keep_nw;
                        for (uint32_t g = KS.desc[d].ne0 + first; g < KS.desc[d].ne1; g += R.keep_nw) {
                            cta[c].push_back({&sg[0][g], su[0].data() + sg[0][g].uoff});
                            tag[c].push_back(w);
                        }
                    }
        } else {
            uint64_t run = 0;
            for (uint32_t s = 0; s < sg.size(); ++s)
                for (const Grp& g : sg[s]) {
                    const uint64_t c = g.cost(cap, !forward_only);
                    cta[std::min<uint64_t>(grid - 1, (2 * run + c) * grid / (2 * total))].push_back({&g, su[s].data() + g.uoff});
                    run += c;
                }
        }
        // small matrices: packets small enough that a warp gets several
        const uint32_t pack = kept_deal ? max_u : (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(cap, n_union / ((uint64_t)grid * 96)));
        std::vector<CtaOut> out(grid);
        struct Work {
            std::vector<uint32_t> pos, seen;
            uint32_t gen = 0;
        };
        std::vector<Work> work(kMaxThreads);
        ok = parallel_for(grid, [&](uint32_t c, uint32_t thread) {
            Work& w = work[thread];
            if (w.seen.empty()) {
                w.pos.assign(std::max(ncols, 1u), 0);
                w.seen.assign(std::max(ncols, 1u), 0);
            }
            write_cta(M, hr, R.iw, pack, max_u, rows.data(), cta[c], keep, kept_deal ? &tag[c] : nullptr,
                      !forward_only, w.pos, w.seen, ++w.gen, out[c]);
        });
        if (!ok) throw std::bad_alloc();

        R.cta_pk.assign(grid + 1, 0);
        std::vector<uint32_t> dict, dict_begin(grid + 1, 0);
        std::vector<uint4> pk;
        std::vector<uint32_t> row_list;
        uint64_t bytes = 0;
        R.wmax = 0;
        R.slot = 0;
        R.pk_cost.clear();
        R.pk_chain.clear();
        R.keep_tag.clear();
        std::vector<uint64_t> base(grid);
        for (uint32_t c = 0; c < grid; ++c) {
            base[c] = bytes;
            for (size_t i = 0; i < out[c].pk.size(); ++i) {
                const uint4 q = out[c].pk[i];
                pk.push_back(make_uint4((uint32_t)(bytes / 16 + q.x), q.y, (uint32_t)(row_list.size() + q.z), q.w));
                R.pk_chain.push_back((q.y & (RG_CARRY_IN | RG_AGAIN)) != 0);
            }
            R.keep_tag.insert(R.keep_tag.end(), out[c].tag.begin(), out[c].tag.end());
            row_list.insert(row_list.end(), out[c].rows.begin(), out[c].rows.end());
            R.pk_cost.insert(R.pk_cost.end(), out[c].cost.begin(), out[c].cost.end());
            bytes += out[c].data.size();
            dict.insert(dict.end(), out[c].dict.begin(), out[c].dict.end());
            dict_begin[c + 1] = (uint32_t)dict.size();
            R.cta_pk[c + 1] = (uint32_t)pk.size();
            R.wmax = std::max(R.wmax, (uint32_t)out[c].dict.size());
            if (R.iw == 2 && out[c].dict.size() > 65536) {
                *why = "a CTA's rows see more than 65536 columns";
                return false;
            }
            R.slot = std::max(R.slot, out[c].slot);
        }
        R.slot = (std::max(R.slot, 128u) + 127) / 128 * 128;
        if (bytes / 16 >= 0xFFFFFFFFull) {
            *why = "the layout takes more than 64 GB";
            return false;
        }
        // where each column's partial sums lie among the CTAs': eight lists per
        // column, list k of CTAs k, k + 8, ... in order
        std::vector<uint32_t> col_ptr(8 * (size_t)ncols + 1, 0), col_pos(dict.size());
        for (uint32_t c = 0; c < grid; ++c)
            for (uint32_t i = dict_begin[c]; i < dict_begin[c + 1]; ++i) ++col_ptr[8 * (size_t)dict[i] + c % 8 + 1];
        for (size_t j = 0; j < 8 * (size_t)ncols; ++j) col_ptr[j + 1] += col_ptr[j];
        {
            std::vector<uint32_t> at(col_ptr.begin(), col_ptr.end() - 1);
            for (uint32_t c = 0; c < grid; ++c)
                for (uint32_t i = dict_begin[c]; i < dict_begin[c + 1]; ++i) col_pos[at[8 * (size_t)dict[i] + c % 8]++] = i;
        }
        // runs of rows without entries, at most kRgZeroRun rows each
        std::vector<uint2> zr;
        for (uint32_t r = 0; r < nrows;) {
            if (rp[r + 1] > rp[r]) {
                ++r;
                continue;
            }
            uint32_t e = r + 1;
            while (e < nrows && rp[e + 1] == rp[e] && e - r < kRgZeroRun) ++e;
            zr.push_back(make_uint2(r, e - r));
            r = e;
        }
        const size_t nwords = ((size_t)nrows + 31) / 32;
        std::vector<uint32_t> mask((nwords + 3) / 4 * 4 + 4, 0);
        for (uint32_t r : rows) mask[r >> 5] |= 1u << (r & 31);

        cudaError_t e = dev_malloc(&R.data, std::max<uint64_t>(bytes, 16));
        for (uint32_t c = 0; c < grid && e == cudaSuccess; ++c)
            if (!out[c].data.empty())
                e = cudaMemcpy(R.data + base[c], out[c].data.data(), out[c].data.size(), cudaMemcpyHostToDevice);
        auto up = [&](auto** dst, const auto& v) {
            using T = typename std::decay_t<decltype(v)>::value_type;
            if (e == cudaSuccess)
                e = rg_upload(reinterpret_cast<void**>(dst), v.data(), v.size() * sizeof(T), v.size() * sizeof(T) + 16);
        };
        up(&R.row_list, row_list);
        up(&R.dict, dict);
        up(&R.dict_begin, dict_begin);
        up(&R.col_ptr, col_ptr);
        up(&R.col_pos, col_pos);
        up(&R.zero_runs, zr);
        up(&R.mask, mask);
        if (e == cudaSuccess) e = dev_malloc(&R.g_part, std::max<size_t>(dict.size(), 4) * 4);
        if (e != cudaSuccess) {
            *err = e;
            free_row_groups(R);
            return false;
        }
        R.host_pk = std::move(pk);
        R.n_zero_runs = (uint32_t)zr.size();
        R.n_groups = n_groups;
        R.n_union = n_union;
        R.tile_u = tile_u;
        R.order = (uint32_t)order;
        R.keep = kept_deal;
        R.forward_only = forward_only;
        R.data_bytes = bytes;
        R.bytes = bytes + row_list.size() * 4 + dict.size() * 12 + (size_t)ncols * 32 + zr.size() * 8 + mask.size() * 4;
        R.built = true;
    } catch (const std::exception&) {  // host memory for the lists
        free_row_groups(R);
        *why = "not enough host memory to build it";
        *err = cudaErrorMemoryAllocation;
        return false;
    }
    return true;
}

const RowGroups& rg_of(const dose_matrix* A, int which) {
    return which == RG_DEAL_FUSED && A->rgf.built ? A->rgf : A->rg;
}

uint32_t rg_warps(const dose_matrix* A, int which, uint32_t* depth, size_t* smem) {
    return which == RG_DEAL_FUSED || which == RG_DEAL_ADJOINT
               ? rg_gradient_warps(A, A->adj_tuning, which == RG_DEAL_FUSED, depth, smem)
               : rg_forward_warps(A, which, depth, smem);
}

// Warps of each call under the knobs t and the deals of packets to them.  The knobs
// and deals in effect are replaced when all the new ones are there: after a failure
// every call runs as before.
cudaError_t rg_schedule(dose_matrix* A, const AdjTuning& t) {
    const AdjTuning old = A->adj_tuning;
    A->adj_tuning = t;
    RgDeal fresh[RG_DEALS];
    uint32_t depth = 0;
    size_t smem = 0;
    cudaError_t e = cudaSuccess;
    auto layout = [&](int which) -> RowGroups& { return which == RG_DEAL_FUSED && A->rgf.built ? A->rgf : A->rg; };
    for (int which = 0; which < RG_DEALS && e == cudaSuccess; ++which) {
        const RowGroups& R = layout(which);
        const uint32_t nw = R.built ? rg_warps(A, which, &depth, &smem) : 0;
        try {
            if (nw && nw != R.deal[which].nw) e = rg_deal(R, nw, fresh[which]);
        } catch (const std::exception&) {  // host memory for the lists
            e = cudaErrorMemoryAllocation;
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);  // the copies have reached the device
    for (int which = 0; which < RG_DEALS; ++which) {
        RowGroups& R = layout(which);
        RgDeal& D = R.deal[which];
        const RgDeal n = fresh[which];
        if (!n.begin) continue;
        if (e == cudaSuccess) {
            auto bytes = [&](const RgDeal& d) { return d.begin ? ((size_t)R.grid * d.nw + 1) * 4 + R.host_pk.size() * 16 : 0; };
            R.bytes = R.bytes - bytes(D) + bytes(n);
            cudaFree(D.begin);
            cudaFree(D.pk);
            D = n;
        } else {
            cudaFree(n.begin);
            cudaFree(n.pk);
        }
    }
    if (e != cudaSuccess) A->adj_tuning = old;
    return e;
}

}  // namespace dose
