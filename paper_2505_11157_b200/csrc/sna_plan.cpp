// Host planner.  Grids and quadrature: App. A.1 and Eq. (quadrature); neighborhood indicator: App. B.3,
// disc of Eq. (s2_neighborhood_attention).
//
// Construction (deliberately not a brute-force scan): on a fixed input ring the geodesic distance to the
// output point grows monotonically with the longitude difference, so each ring contributes one window
// symmetric about offset 0.  The half width follows from the spherical law of cosines,
//     cos(dphi_max) = (cos(theta_c) - cos(t_o) cos(t_i)) / (sin(t_o) sin(t_i)),
// and the columns around that estimate are then tested exactly with a cross/dot (atan2) distance, which is
// accurate for small and large angles alike.  Boundary ties are members (d <= theta_c + 1e-10); a candidate in
// the band 1e-12 < |d - theta_c| < 1e-8 aborts the build as ambiguous.
#include "sna_plan.hpp"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

namespace sna {
namespace {

const long double PI_L = 3.14159265358979323846264338327950288L;
const double TIE_SLACK = 1e-10, BAND_LO = 1e-12, BAND_HI = 1e-8;

// Gauss-Legendre nodes (descending) and weights by Newton iteration in extended precision, started from
// Tricomi's asymptotic estimate of the roots.
void legendre_gauss(int n, std::vector<double>& x, std::vector<double>& w) {
    x.resize(n);
    w.resize(n);
    for (int i = 1; i <= (n + 1) / 2; ++i) {
        long double z = (1.0L - (n - 1.0L) / (8.0L * n * n * n)) * cosl(PI_L * (4.0L * i - 1.0L) / (4.0L * n + 2.0L));
        long double pn = 0, pn1 = 0;
        for (int it = 0; it < 64; ++it) {
            long double a = 1.0L, b = z;   // P_0, P_1
            for (int l = 1; l < n; ++l) {
                long double c = ((2 * l + 1) * z * b - l * a) / (l + 1);
                a = b;
                b = c;
            }
            pn = b;
            pn1 = a;
            long double deriv = n * (pn1 - z * pn) / (1.0L - z * z);
            long double step = pn / deriv;
            z -= step;
            if (fabsl(step) < 1e-19L) break;
        }
        // re-evaluate at the converged node for the weight
        long double a = 1.0L, b = z;
        for (int l = 1; l < n; ++l) {
            long double c = ((2 * l + 1) * z * b - l * a) / (l + 1);
            a = b;
            b = c;
        }
        long double deriv = n * (a - z * b) / (1.0L - z * z);
        long double wt = 2.0L / ((1.0L - z * z) * deriv * deriv);
        x[i - 1] = (double)z;
        w[i - 1] = (double)wt;
        x[n - i] = (double)(-z);
        w[n - i] = (double)wt;
    }
    if (n % 2 == 1) x[n / 2] = 0.0;
}

// Clenshaw-Curtis weights on nlat equally spaced colatitudes including both poles.
void clenshaw_curtis(int nlat, std::vector<double>& w) {
    const int n = nlat - 1;
    w.resize(nlat);
    std::vector<long double> cosine(2 * n);              // of i pi / n: all that the sums need
    for (int i = 0; i < 2 * n; ++i) cosine[i] = cosl(PI_L * (long double)i / (long double)n);
    for (int h = 0; h <= n; ++h) {
        long double acc = 1.0L;
        for (int k = 1; k <= n / 2; ++k) {
            long long arg = (2LL * k * h) % (2LL * n);           // cos(2 k pi h / n) with an exactly reduced argument
            long double bk = (2 * k == n) ? 1.0L : 2.0L;
            acc -= bk * cosine[arg] / (4.0L * k * k - 1.0L);
        }
        long double ch = (h == 0 || h == n) ? 1.0L : 2.0L;
        w[h] = (double)(ch * acc / n);
    }
}

bool make_grid(int grid, int nlat, std::vector<double>& theta, std::vector<double>& wlat) {
    if (grid == 0) {
        theta.resize(nlat);
        for (int h = 0; h < nlat; ++h) theta[h] = (double)(PI_L * h / (nlat - 1));
        clenshaw_curtis(nlat, wlat);
        return true;
    }
    if (grid == 1) {
        std::vector<double> x;
        legendre_gauss(nlat, x, wlat);
        theta.resize(nlat);
        for (int h = 0; h < nlat; ++h) theta[h] = std::acos(x[h]);
        return true;
    }
    if (grid == 2) {
        // the grid as App. A.1 prints it (Eq. latlon_grid, Eq. latlon_quad_weights): north pole in, south pole out,
        // trapezoid weights (pi/nlat) sin(theta) in latitude; the pole ring's weight is exactly zero
        theta.resize(nlat);
        wlat.resize(nlat);
        for (int h = 0; h < nlat; ++h) {
            theta[h] = (double)(PI_L * h / nlat);
            wlat[h] = h == 0 ? 0.0 : (double)(PI_L / nlat * sinl(PI_L * h / nlat));
        }
        return true;
    }
    return false;
}

// Geodesic distance between (t_o, 0) and (t_i, phi) from cross and dot products of the unit vectors.
double geodesic(double so, double co, double si, double ci, double phi) {
    const double cp = std::cos(phi), sp = std::sin(phi);
    const double ox = so, oz = co;
    const double ix = si * cp, iy = si * sp, iz = ci;
    const double cx = -oz * iy, cy = oz * ix - ox * iz, cz = ox * iy;
    return std::atan2(std::sqrt(cx * cx + cy * cy + cz * cz), ox * ix + oz * iz);
}

}  // namespace

PlanStatus build_plan(int nlat_in, int nlon_in, int nlat_out, int nlon_out, int grid_in, int grid_out,
                      double theta_cutoff, HostPlan& P, std::string& why) {
    if (nlat_in < 2 || nlat_out < 2 || nlon_in < 1 || nlon_out < 1) { why = "nlat must be >= 2 and nlon >= 1"; return PLAN_INVALID; }
    if (!(theta_cutoff > 0.0) || std::isnan(theta_cutoff)) { why = "theta_cutoff must be positive"; return PLAN_INVALID; }
    if (nlon_in % nlon_out != 0) { why = "nlon_in must be a multiple of nlon_out"; return PLAN_UNSUPPORTED; }
    P = HostPlan();
    P.nlat_in = nlat_in; P.nlon_in = nlon_in; P.nlat_out = nlat_out; P.nlon_out = nlon_out;
    P.ps = nlon_in / nlon_out; P.grid_in = grid_in; P.grid_out = grid_out; P.theta_cutoff = theta_cutoff;
    std::vector<double> wlat_in, wlat_out;
    if (!make_grid(grid_in, nlat_in, P.theta_in, wlat_in) || !make_grid(grid_out, nlat_out, P.theta_out, wlat_out)) {
        why = "unknown grid type";
        return PLAN_UNSUPPORTED;
    }
    P.omega.resize(nlat_in);
    for (int h = 0; h < nlat_in; ++h) P.omega[h] = wlat_in[h] * (double)(2.0L * PI_L / nlon_in);

    const bool everything = theta_cutoff >= (double)PI_L;
    const int half = nlon_in / 2;                        // largest |column offset| on a ring
    const double dphi = (double)(2.0L * PI_L / nlon_in);
    const double cos_tc = std::cos(theta_cutoff);
    bool ambiguous = false;
    auto member = [&](double d) {
        const double gap = std::fabs(d - theta_cutoff);
        if (gap > BAND_LO && gap < BAND_HI) ambiguous = true;
        return d <= theta_cutoff + TIE_SLACK;
    };

    P.row_ptr.assign(nlat_out + 1, 0);
    P.row_nnz.assign(nlat_out, 0);
    std::vector<std::vector<RingWindow>> by_input(nlat_in);
    std::vector<double> sin_in(nlat_in), cos_in(nlat_in);
    for (int hp = 0; hp < nlat_in; ++hp) { sin_in[hp] = std::sin(P.theta_in[hp]); cos_in[hp] = std::cos(P.theta_in[hp]); }
    for (int h = 0; h < nlat_out; ++h) {
        const double so = std::sin(P.theta_out[h]), co = std::cos(P.theta_out[h]);
        for (int hp = 0; hp < nlat_in; ++hp) {
            int m = -2;   // -2: ring not in the disc, -1: whole ring, >= 0: half width
            if (everything) {
                m = -1;
            } else {
                // the nearest point is as far as the colatitudes differ: no need to evaluate rings that are clearly outside
                if (std::fabs(P.theta_out[h] - P.theta_in[hp]) > theta_cutoff + 1e-3) continue;
                const double si = sin_in[hp], ci = cos_in[hp];
                if (!member(geodesic(so, co, si, ci, 0.0))) continue;   // nearest point of the ring is outside
                const double denom = so * si;
                int guess;
                if (denom < 1e-300) {
                    guess = half;   // a pole is involved: every column is equally far
                } else {
                    const double r = (cos_tc - co * ci) / denom;
                    guess = r <= -1.0 ? half : (r >= 1.0 ? 0 : (int)std::floor(std::acos(r) / dphi));
                }
                // exact test around the estimate; membership is monotone in the offset
                int lo = std::max(0, guess - 2), hi = std::min(half, guess + 2);
                while (lo > 0 && !member(geodesic(so, co, si, ci, lo * dphi))) lo = std::max(0, lo - 4);
                m = lo;
                for (int j = lo + 1; j <= hi; ++j) {
                    if (member(geodesic(so, co, si, ci, j * dphi))) m = j; else break;
                }
                if (m == hi && hi < half) {   // estimate was too small (never seen, but stay correct)
                    int j = hi + 1;
                    while (j <= half && member(geodesic(so, co, si, ci, j * dphi))) m = j++;
                }
                if (2 * m + 1 >= nlon_in) m = -1;
            }
            RingWindow w{hp, m};
            P.windows.push_back(w);
            P.row_nnz[h] += P.window_count(w);
            by_input[hp].push_back(RingWindow{h, m});
        }
        P.row_ptr[h + 1] = (int32_t)P.windows.size();
        if (P.row_ptr[h + 1] == P.row_ptr[h] && !ambiguous) { why = "an output latitude has no input point within theta_cutoff"; return PLAN_EMPTY; }
        bool weighted = false;
        for (int i = P.row_ptr[h]; i < P.row_ptr[h + 1]; ++i) weighted = weighted || P.omega[P.windows[i].lat] > 0.0;
        if (!weighted && !ambiguous) { why = "every input point within theta_cutoff of an output latitude has quadrature weight zero"; return PLAN_EMPTY; }
        P.nnz += P.row_nnz[h];
    }
    if (ambiguous) { why = "a grid point lies within 1e-8 rad of the disc boundary without being on it"; return PLAN_AMBIGUOUS; }

    P.t_row_ptr.assign(nlat_in + 1, 0);
    P.t_row_nnz.assign(nlat_in, 0);
    for (int hp = 0; hp < nlat_in; ++hp) {
        for (const RingWindow& w : by_input[hp]) {
            P.t_windows.push_back(w);
            P.t_row_nnz[hp] += P.window_count(w);
        }
        P.t_row_ptr[hp + 1] = (int32_t)P.t_windows.size();
    }
    return PLAN_OK;
}

bool drop_zero_weight_rings(const HostPlan& full, HostPlan& out) {
    bool any = false;
    for (double w : full.omega) any = any || !(w > 0.0);
    if (!any) return false;
    out = full;
    out.windows.clear();
    out.t_windows.clear();
    out.nnz = 0;
    for (int h = 0; h < full.nlat_out; ++h) {
        out.row_ptr[h] = (int32_t)out.windows.size();
        out.row_nnz[h] = 0;
        for (int i = full.row_ptr[h]; i < full.row_ptr[h + 1]; ++i) {
            const RingWindow& w = full.windows[i];
            if (!(full.omega[w.lat] > 0.0)) continue;
            out.windows.push_back(w);
            out.row_nnz[h] += full.window_count(w);
        }
        out.nnz += out.row_nnz[h];
    }
    out.row_ptr[full.nlat_out] = (int32_t)out.windows.size();
    for (int hp = 0; hp < full.nlat_in; ++hp) {
        out.t_row_ptr[hp] = (int32_t)out.t_windows.size();
        out.t_row_nnz[hp] = 0;
        if (!(full.omega[hp] > 0.0)) continue;
        for (int i = full.t_row_ptr[hp]; i < full.t_row_ptr[hp + 1]; ++i) {
            out.t_windows.push_back(full.t_windows[i]);
            out.t_row_nnz[hp] += full.window_count(full.t_windows[i]);
        }
    }
    out.t_row_ptr[full.nlat_in] = (int32_t)out.t_windows.size();
    return true;
}

namespace {

inline int floor_div(int a, int b) { int q = a / b; return ((a % b != 0) && ((a < 0) != (b < 0))) ? q - 1 : q; }
inline int ceil_div(int a, int b) { return -floor_div(-a, b); }

// Merges the window lists of the rings of a group (each sorted by partner ring) and calls
// emit(partner_ring, m[TILE_LAT]) with m = -2 for "not in this ring's list".
template <typename Emit>
void merge_group(const std::vector<int32_t>& ptr, const std::vector<RingWindow>& win, int first_ring, int nrings, int dense_min_width, Emit&& emit) {
    int pos[TILE_LAT], end[TILE_LAT];
    for (int k = 0; k < TILE_LAT; ++k) {
        const int ring = first_ring + k;
        pos[k] = ring < nrings ? ptr[ring] : 0;
        end[k] = ring < nrings ? ptr[ring + 1] : 0;
    }
    for (;;) {
        int lat = INT32_MAX;
        for (int k = 0; k < TILE_LAT; ++k)
            if (pos[k] < end[k]) lat = std::min(lat, win[pos[k]].lat);
        if (lat == INT32_MAX) break;
        int m[TILE_LAT];
        for (int k = 0; k < TILE_LAT; ++k) {
            m[k] = (pos[k] < end[k] && win[pos[k]].lat == lat) ? win[pos[k]++].m : -2;
            if (m[k] != -2 && served_by_dense(RingWindow{lat, m[k]}, dense_min_width)) m[k] = -2;
        }
        emit(lat, m);
    }
}

// Collects the columns of one stream row and packs them into chunks.
class BandBuilder {
public:
    // All `count` points of a partner ring, for the group rings that take it whole (m = -1).
    void add_whole(int32_t base, float bias, const int (&m)[TILE_LAT], int count) {
        uint32_t mask = 0;
        for (int k = 0; k < TILE_LAT; ++k)
            if (m[k] == -1) mask |= ((1u << TILE_LON) - 1u) << (k * TILE_LON);
        if (mask) for (int u = 0; u < count; ++u) add((int32_t)(base | (int32_t)0x80000000), u, bias, mask);
    }
    // A partner ring for the group rings with a band (m >= 0): band_range(m, i, lo, hi) gives the partner offsets [lo, hi] that
    // tile longitude i uses.
    template <typename Range>
    void add_band(int32_t base, float bias, const int (&m)[TILE_LAT], Range&& band_range) {
        int rlo[TILE_LAT * TILE_LON], rhi[TILE_LAT * TILE_LON], lo = INT32_MAX, hi = INT32_MIN;
        for (int row = 0; row < TILE_LAT * TILE_LON; ++row) {
            rlo[row] = 0; rhi[row] = -1;          // empty
            if (m[row / TILE_LON] < 0) continue;
            band_range(m[row / TILE_LON], row % TILE_LON, rlo[row], rhi[row]);
            if (rhi[row] >= rlo[row]) { lo = std::min(lo, rlo[row]); hi = std::max(hi, rhi[row]); }
        }
        if (hi < lo) return;
        // where each row's range begins and ends; the running exclusive-or is the mask
        toggle_.assign((size_t)(hi - lo) + 2, 0u);
        for (int row = 0; row < TILE_LAT * TILE_LON; ++row)
            if (rhi[row] >= rlo[row]) { toggle_[rlo[row] - lo] ^= 1u << row; toggle_[rhi[row] + 1 - lo] ^= 1u << row; }
        uint32_t mask = 0;
        for (int e = lo; e <= hi; ++e) {
            mask ^= toggle_[e - lo];
            if (mask) add(base, e, bias, mask);
        }
    }
    // Appends the columns to the stream as a row, and starts anew.
    void finish(BandStream& S) {
        if (S.chunk_ptr.empty()) S.chunk_ptr.push_back(0);
        // padding repeats the last column with an empty mask
        while (cols_.size() % BAND_CHUNK != 0) { cols_.push_back(BandColumn(cols_.back())); masks_.push_back(0u); }
        S.columns.insert(S.columns.end(), cols_.begin(), cols_.end());
        for (size_t c = 0; c < masks_.size(); c += BAND_CHUNK) {
            const uint32_t* mask = masks_.data() + c;
            uint32_t all = 0xffffu;
            for (size_t j = 0; j < BAND_CHUNK; ++j) all &= mask[j];
            uint32_t lanes[32];
            for (int t = 0; t < 4; ++t) {
                // the four columns of lanes 4 g + t, each as two bytes of rows: an 8 x 8 bit matrix whose columns are the lanes' masks
                const uint64_t rows = (mask[2 * t] & 0xffu) | (uint64_t)(mask[2 * t + 1] & 0xffu) << 8 | (uint64_t)(mask[2 * t] >> 8) << 16 |
                                      (uint64_t)(mask[2 * t + 1] >> 8) << 24 | (uint64_t)(mask[8 + 2 * t] & 0xffu) << 32 |
                                      (uint64_t)(mask[9 + 2 * t] & 0xffu) << 40 | (uint64_t)(mask[8 + 2 * t] >> 8) << 48 |
                                      (uint64_t)(mask[9 + 2 * t] >> 8) << 56;
                const uint64_t bytes = transpose_bits(rows);
                for (int g = 0; g < 8; ++g) lanes[4 * g + t] = (uint32_t)(bytes >> 8 * g & 0xffu) | (all == 0xffffu ? BAND_ALL : 0u);
            }
            S.masks.insert(S.masks.end(), lanes, lanes + 32);
        }
        S.chunk_ptr.push_back((int32_t)(S.columns.size() / BAND_CHUNK));
        cols_.clear();
        masks_.clear();
    }

private:
    void add(int32_t base, int32_t e, float bias, uint32_t mask) {
        cols_.push_back(BandColumn{base, e, bias, 0});
        masks_.push_back(mask);
    }
    // byte i, bit j -> byte j, bit i (three rounds of swapping blocks, as one does by hand)
    static uint64_t transpose_bits(uint64_t x) {
        auto swap = [&](uint64_t where, int by) { const uint64_t d = (x ^ (x >> by)) & where; x ^= d ^ (d << by); };
        swap(0x00aa00aa00aa00aaull, 7);
        swap(0x0000cccc0000ccccull, 14);
        swap(0x00000000f0f0f0f0ull, 28);
        return x;
    }
    std::vector<BandColumn> cols_;
    std::vector<uint32_t> masks_;
    std::vector<uint32_t> toggle_;
};

// the kernels read three chunks ahead
void pad(BandStream& S) {
    const BandColumn last = S.columns.empty() ? BandColumn{0, 0, 0.f, 0} : S.columns.back();
    S.columns.insert(S.columns.end(), 3 * BAND_CHUNK, last);
    S.masks.insert(S.masks.end(), 3 * 32, 0u);
}

// ptr, win, dense_min_width: as given to merge_group
void complete(BandStream& S, int rows_per_group, const std::vector<int32_t>& ptr, const std::vector<RingWindow>& win, int dense_min_width) {
    pad(S);
    S.order.resize((S.chunk_ptr.size() - 1) / rows_per_group);
    for (size_t i = 0; i < S.order.size(); ++i) S.order[i] = (int32_t)i;
    auto length = [&](int g) { return S.chunk_ptr[(size_t)(g + 1) * rows_per_group] - S.chunk_ptr[(size_t)g * rows_per_group]; };
    std::stable_sort(S.order.begin(), S.order.end(), [&](int a, int b) { return length(a) > length(b); });
    // Groups with windows on the dense kernels depend on their results: not among the first, which may start before those are there.
    std::vector<int32_t> independent, dependent;
    for (int g : S.order) {
        bool dense = false;
        const size_t end = std::min<size_t>((size_t)(g + 1) * TILE_LAT, ptr.size() - 1);
        for (int i = ptr[(size_t)g * TILE_LAT]; i < ptr[end]; ++i) dense = dense || served_by_dense(win[i], dense_min_width);
        (dense ? dependent : independent).push_back(g);
    }
    S.order = independent;
    S.order.insert(S.order.begin() + independent.size() / 4, dependent.begin(), dependent.end());
    for (int g : S.order) S.lengths.push_back(length(g) / rows_per_group);
}

}  // namespace

void build_dense_lists(const HostPlan& P, DenseLists& D, int dense_min_width) {
    D = DenseLists();
    D.ptr.assign(P.nlat_out + 1, 0);
    for (int h = 0; h < P.nlat_out; ++h) {
        int64_t blocks = 0;
        for (int e = P.row_ptr[h]; e < P.row_ptr[h + 1]; ++e) {
            if (!served_by_dense(P.windows[e], dense_min_width)) continue;
            D.lat.push_back(P.windows[e].lat);
            D.m.push_back(P.windows[e].m);
            D.pairs += P.window_count(P.windows[e]);
            // the columns between the first row's window and the last row's
            const int64_t span = P.windows[e].m < 0 ? P.nlon_in : std::min<int64_t>(2 * P.windows[e].m + 1 + 127LL * P.ps, P.nlon_in);
            blocks += (span + 127) / 128;
        }
        D.ptr[h + 1] = (int32_t)D.lat.size();
        if (D.ptr[h + 1] > D.ptr[h]) D.rows.push_back(h);
        D.blocks += blocks;
        D.longest = std::max(D.longest, blocks);
    }
}

void build_transposed_dense_lists(const HostPlan& P, DenseLists& D, int dense_min_width) {
    D = DenseLists();
    D.ptr.assign(P.nlat_in + 1, 0);
    for (int hp = 0; hp < P.nlat_in; ++hp) {
        for (int e = P.t_row_ptr[hp]; e < P.t_row_ptr[hp + 1]; ++e) {
            if (!served_by_dense(P.t_windows[e], dense_min_width)) continue;
            D.lat.push_back(P.t_windows[e].lat);
            D.m.push_back(P.t_windows[e].m);
            D.pairs += P.window_count(P.t_windows[e]);
        }
        D.ptr[hp + 1] = (int32_t)D.lat.size();
        if (D.ptr[hp + 1] > D.ptr[hp]) D.rows.push_back(hp);
    }
}

void build_global_bands(const HostPlan& P, BandStream& forward, BandStream& transposed) {
    const int whole[TILE_LAT] = {-1, -1};
    auto one_row = [](BandBuilder& b, BandStream& S, int rings) {
        S = BandStream();
        b.finish(S);
        pad(S);
        S.one_row = true;
        S.order.assign(ceil_div(rings, TILE_LAT), 0);
        for (size_t i = 0; i < S.order.size(); ++i) S.order[i] = (int32_t)i;
        S.lengths.assign(S.order.size(), S.chunk_ptr[1]);
    };
    BandBuilder f, t;
    for (int lat = 0; lat < P.nlat_in; ++lat)
        for (int r = 0; r < P.ps && P.omega[lat] > 0.0; ++r) f.add_whole(lat * P.nlon_in + r, (float)std::log2(P.omega[lat]), whole, P.nlon_out);
    for (int lat = 0; lat < P.nlat_out; ++lat) t.add_whole(lat * P.nlon_out, 0.f, whole, P.nlon_out);
    one_row(f, forward, P.nlat_out);
    one_row(t, transposed, P.nlat_in);
}

void build_forward_band(const HostPlan& P, BandStream& S, int dense_min_width) {
    S = BandStream();
    BandBuilder b;
    for (int first = 0; first < P.nlat_out; first += TILE_LAT) {
        merge_group(P.row_ptr, P.windows, first, P.nlat_out, dense_min_width, [&](int lat, const int (&m)[TILE_LAT]) {
            const float bias = (float)std::log2(P.omega[lat]);
            for (int r = 0; r < P.ps; ++r) {
                b.add_whole(lat * P.nlon_in + r, bias, m, P.nlon_out);
                b.add_band(lat * P.nlon_in + r, bias, m, [&](int mk, int i, int& lo, int& hi) {
                    lo = i + ceil_div(-mk - r, P.ps);
                    hi = i + floor_div(mk - r, P.ps);
                });
            }
        });
        b.finish(S);
    }
    complete(S, 1, P.row_ptr, P.windows, dense_min_width);
}

bool build_transposed_band(const HostPlan& P, BandStream& S, int dense_min_width) {
    S = BandStream();
    const bool consecutive = TILE_LON % P.ps == 0;
    BandBuilder b;
    for (int first = 0; first < P.nlat_in; first += TILE_LAT)
        for (int r = 0; r < (consecutive ? 1 : P.ps); ++r) {
            merge_group(P.t_row_ptr, P.t_windows, first, P.nlat_in, dense_min_width, [&](int lat, const int (&m)[TILE_LAT]) {
                // Output point w is a partner of input column c iff c - w*ps lies in [-m, m].  Consecutive: c = c0 + i, so
                // w - c0/ps in [ceil((i - m)/ps), floor((i + m)/ps)].  By residue: c = ps*(u0+i) + r, so w - u0 in
                // [i + ceil((r - m)/ps), i + floor((r + m)/ps)].
                b.add_whole(lat * P.nlon_out, 0.f, m, P.nlon_out);
                b.add_band(lat * P.nlon_out, 0.f, m, [&](int mk, int i, int& lo, int& hi) {
                    lo = consecutive ? ceil_div(i - mk, P.ps) : i + ceil_div(r - mk, P.ps);
                    hi = consecutive ? floor_div(i + mk, P.ps) : i + floor_div(r + mk, P.ps);
                });
            });
            b.finish(S);
        }
    complete(S, consecutive ? 1 : P.ps, P.t_row_ptr, P.t_windows, dense_min_width);
    return consecutive;
}

}  // namespace sna
