// Band-limited staging forms of a plan's streams: the basis of the band the energies cover, the choice
// of block length and rank, and the rule that picks a form (or plain frames) for a staging ring.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/tacaw.h"
#include "tacaw_internal.cuh"
#include "tacaw_plan.cuh"

using namespace tacaw;

namespace {

// First halves (u < B/2) of the k most concentrated discrete prolate spheroidal sequences of one parity,
// length B, full bandwidth beta cycles per sample: eigenvectors of Slepian's tridiagonal matrix (diagonal
// ((B-1-2u)/2)^2 cos(pi beta), off-diagonal u (B-u)/2), which splits by symmetry into an even and an odd
// problem of size B/2; the largest eigenvalues belong to the most concentrated sequences.  Eigenvalues by
// bisection on the count of negative pivots of (A - x), each vector by inverse iteration.
class Prolate {
public:
    Prolate(int B, double beta, int parity) : H(B / 2), d(H), o(H, 0.0) {
        for (int u = 0; u < H; ++u) {
            const double c = 0.5 * (B - 1 - 2 * u);
            d[u] = c * c * std::cos(M_PI * beta);
            if (u > 0) o[u] = 0.5 * u * (B - u);   // between u - 1 and u
        }
        d[H - 1] += (parity ? -0.5 : 0.5) * H * (B - H);
        lo = hi = d[0];
        for (int u = 0; u < H; ++u) {
            const double r = o[u] + (u + 1 < H ? o[u + 1] : 0.0);
            lo = std::min(lo, d[u] - r);
            hi = std::max(hi, d[u] + r);
        }
    }
    // first halves of the n most concentrated sequences, the whole sequences of unit norm (norm sqrt(1/2))
    std::vector<std::vector<double>> vectors(int n) const {
        n = std::min(n, H);
        // all eigenvalues side by side, four to a pass: each count is a chain of divisions, which the others overlap
        constexpr int L = 4;
        const int m = (n + L - 1) / L * L;
        std::vector<double> a(m, lo), b(m, hi);
        for (int i = 0; i < 24; ++i) {   // to 2^-24 of the range, below the gaps (range / B and less) by 2^10 and more
            for (int k0 = 0; k0 < m; k0 += L) {
                double x[L], q[L], above[L];
                for (int k = 0; k < L; ++k) {
                    x[k] = 0.5 * (a[k0 + k] + b[k0 + k]);
                    q[k] = 1.0;
                    above[k] = 0.0;
                }
                for (int u = 0; u < H; ++u) {
                    const double o2 = o[u] * o[u], du = d[u];   // (o[0] = 0)
                    for (int k = 0; k < L; ++k) {
                        double t = du - x[k] - o2 / q[k];
                        t = t == 0.0 ? 1e-300 : t;
                        above[k] += t > 0.0 ? 1.0 : 0.0;        // positive pivots of A - x: eigenvalues above x
                        q[k] = t;
                    }
                }
                for (int k = 0; k < L; ++k) (above[k] > k0 + k ? a : b)[k0 + k] = x[k];
            }
        }
        std::vector<std::vector<double>> out;
        Factors f;
        for (int k = 0; k < n; ++k) {
            const double shift = 0.5 * (a[k] + b[k]) + 1e-11 * (hi - lo);   // off the eigenvalue: the solves stay finite
            std::vector<double> v(H);
            for (int u = 0; u < H; ++u) v[u] = 1.0 + 0.01 * (u % 7);   // no symmetry that could hide a vector
            f.factor(*this, shift);
            for (int it = 0; it < 5; ++it) {
                f.solve(v);
                double s = 0.0;
                for (double t : v) s += t * t;
                for (double &t : v) t *= std::sqrt(0.5 / s);
            }
            out.push_back(v);
        }
        return out;
    }

private:
    int H;
    std::vector<double> d, o;
    double lo, hi;
    // A - x by Gaussian elimination with row exchanges: the multiplier of each step, and the upper rows
    // (1 / a, b, c at columns u, u+1, u+2)
    struct Factors {
        std::vector<double> m, r, b, c;
        std::vector<char> swapped;
        void factor(const Prolate &A, double x) {
            const int H = A.H;
            m.assign(H, 0.0);
            r.assign(H, 0.0);
            b.assign(H, 0.0);
            c.assign(H, 0.0);
            swapped.assign(H, 0);
            double p = A.d[0] - x, q = H > 1 ? A.o[1] : 0.0;   // row u as eliminated so far
            for (int u = 0; u + 1 < H; ++u) {
                const double l = A.o[u + 1], dn = A.d[u + 1] - x, on = u + 2 < H ? A.o[u + 2] : 0.0;
                if (std::fabs(p) >= std::fabs(l)) {
                    r[u] = 1.0 / (p == 0.0 ? 1e-300 : p);
                    b[u] = q;
                    m[u] = l * r[u];
                    p = dn - m[u] * q;
                    q = on;
                } else {
                    swapped[u] = 1;
                    r[u] = 1.0 / l;
                    b[u] = dn;
                    c[u] = on;
                    m[u] = p * r[u];
                    p = q - m[u] * dn;
                    q = -m[u] * on;
                }
            }
            r[H - 1] = 1.0 / (p == 0.0 ? 1e-300 : p);
        }
        // v <- (A - x)^-1 v
        void solve(std::vector<double> &v) const {
            const int H = (int)v.size();
            for (int u = 0; u + 1 < H; ++u) {
                if (swapped[u]) std::swap(v[u], v[u + 1]);
                v[u + 1] -= m[u] * v[u];
            }
            for (int u = H - 1; u >= 0; --u) {
                double t = v[u];
                if (u + 1 < H) t -= b[u] * v[u + 1];
                if (u + 2 < H) t -= c[u] * v[u + 2];
                v[u] = t * r[u];
            }
        }
    };
};

// About the rank band_basis finds at kBandTol for x = beta B degrees of freedom (x from 1 to 50).
int rank_guess(double x) { return (int)std::ceil(x + 8.5 + 1.6 * std::log(std::max(1.0, x))); }

// Basis [B/2][R] of the band |d| <= beta/2 (a row: R/2 even vectors, R/2 odd) of the least rank R that
// the push kernels take whose residual over the band stays within tol; R = 0 if none does.  The residual
// is the part of exp(-2 pi i d (u - c)) outside the basis, relative to its norm, checked on a grid of
// d that holds the band's edge, where it is largest.
std::vector<double> band_basis(int B, double beta, double tol, int min_rank, int max_rank, int *rank) {
    const int H = B / 2, kD = 9;
    const Prolate even(B, beta, 0), odd(B, beta, 1);
    const int most = std::min(max_rank, B - 4), guess = std::min(most, rank_guess(beta * B) + 4);
    std::vector<std::vector<double>> ev = even.vectors(guess / 2 + 1), ov = odd.vectors(guess / 2 + 1);
    std::vector<std::vector<double>> vec, res(2 * kD, std::vector<double>(H));
    for (int i = 0; i < kD; ++i)
        for (int u = 0; u < H; ++u) {
            const double ph = 2.0 * M_PI * (0.5 * beta * i / (kD - 1)) * (u - 0.5 * (B - 1));
            res[2 * i][u] = std::cos(ph);
            res[2 * i + 1][u] = std::sin(ph);
        }
    *rank = 0;
    for (int R = min_rank; R <= most; R += 4) {
        if (R / 2 > (int)ev.size()) {
            ev = even.vectors(most / 2);
            ov = odd.vectors(most / 2);
        }
        while ((int)vec.size() < R) {
            const int par = (int)vec.size() & 1;
            vec.push_back((par ? ov : ev)[vec.size() / 2]);
            for (int i = 0; i < kD; ++i) {
                std::vector<double> &r = res[2 * i + par];
                double dot = 0.0;
                for (int u = 0; u < H; ++u) dot += 2.0 * vec.back()[u] * r[u];
                for (int u = 0; u < H; ++u) r[u] -= dot * vec.back()[u];
            }
        }
        double worst = 0.0;
        for (int i = 0; i < kD; ++i) {
            double e = 0.0;
            for (int u = 0; u < H; ++u) e += 2.0 * (res[2 * i][u] * res[2 * i][u] + res[2 * i + 1][u] * res[2 * i + 1][u]);
            worst = std::max(worst, std::sqrt(e / B));
        }
        if (worst <= tol) {
            *rank = R;
            break;
        }
    }
    std::vector<double> basis((size_t)H * *rank);
    for (int u = 0; u < H; ++u)
        for (int q = 0; q < *rank; ++q) basis[(size_t)u * *rank + q] = vec[q < *rank / 2 ? 2 * q : 2 * q - *rank + 1][u];
    return basis;
}

// Reconstruction error allowed at the band's edge, relative to the norm of the exponential.  It acts on
// the part of a block outside the band only (inside, the error is its square), beside operand roundings
// of 2^-17 an element on the split path and FP32 sums of thousands of terms on the FP32 path.
constexpr double kBandTol = 1e-7;

}  // namespace

namespace tacaw {
const std::vector<double> &BandCache::basis(int B, double beta, int min_rank, int max_rank, int *rank) {
    for (const Entry &e : entries)
        if (e.B == B && e.beta == beta && e.max_rank == max_rank) {
            *rank = e.rank;
            return e.v;
        }
    Entry e{B, max_rank, 0, beta, {}};
    e.v = band_basis(B, beta, kBandTol, min_rank, max_rank, &e.rank);
    *rank = e.rank;
    entries.push_back(std::move(e));
    return entries.back().v;
}
}  // namespace tacaw

namespace {

// Segments and rings shorter than this keep staging frames: their passes are bound by launches.
constexpr int kBandMinT = 512;

// Times a (row, frame), in picoseconds, of a ring whose pushes have n frames, staged as frames and as blocks of B
// whose contraction costs `work` products: fitted to measurements (2^16 to 2^20 rows, 8 to 64 frames a push, 60
// to 1000 energies).  A push of frames 2.65 + 8 / n and 3 us a launch (0.5 more where it parts the 16-byte
// chunks of 4 frames); a push of whole blocks 2.3 + 8 / n and 4 us a launch, and 3.7 for the share of the frames
// that passes through the carry; the contraction 0.0139 (split) or 0.142 (FP32) a product, a tenth more on
// coefficients (shorter sums, drained more often).
struct FormCost {
    double product, rows;
    int Nw_pad;
    FormCost(const tacaw_plan_s *p, const Stream &s)
        : product(p->prec == TACAW_PREC_SPLIT_BF16 ? 0.0139 : 0.142), rows((double)s.M), Nw_pad(s.Nw_pad) {}
    double frames(int n) const {
        return 0.97 * (2.65 + 8.0 / n + 3e6 / (rows * n) + (n % 4 ? 0.5 : 0.0) + product * Nw_pad);
    }
    // first: frames of the ring's first push (the end of one that began in the ring before it, or n)
    double blocks(int n, int B, double work, int first) const {
        // share of the frames that wait in the carry, taking the ring's other pushes to have n frames too: the first
        // push's odd frames in each for whole blocks, all but the completing push's for parts of a block, all for
        // other sizes below a block (they drift against the blocks), a block's worth for longer ones
        const double f = n % B == 0 ? (double)(first % B) / n
                         : B % n == 0 && first == n ? 1.0 - (double)n / B
                         : n < B ? 1.0 : (double)B / n;
        return 2.3 + 8.0 / std::max(n, 32) + 4e6 / (rows * n) + 3.7 * f + 1.1 * product * work;
    }
};

// Whether the rule can pick blocks of B over frames and over s's forms so far for a push of some length (a
// ring's first push has up to `most` frames).  Beyond two blocks both the launches' difference and the shares
// carried fall with n, so the lengths up to there, the longest whole number of blocks and the four longest
// (chunks parted or not) decide.
bool ever_picked(const FormCost &c, const Stream &s, int B, double work, int most) {
    auto picks = [&](int n) {
        if (n < 1 || n > most) return false;
        double best = c.frames(n);
        for (int i = 0; i < s.n_band; ++i) best = std::min(best, c.blocks(n, s.band[i].B, s.band[i].work, n));
        return c.blocks(n, B, work, n) < best;
    };
    for (int n = 1; n <= 4 * B; ++n)
        if (picks(n)) return true;
    return picks(most / B * B) || picks(most) || picks(most - 1) || picks(most - 2) || picks(most - 3);
}

// Two-level contraction of a form's coefficients (split path): superblock length S and rank r an energy
// tile, for the least complex products a (row, frame): R / B of the first level's columns, r / S of the
// energies, and 200 a coefficient written and read (16 bytes at the copy rate against 0.0128 ps a
// product).  S = 0 where the direct sum over coefficients costs less than 1.18 times the best.  Measured
// contractions, direct and two-level: 400 energies (work 208, 166) 6.3 and 4.1 ms on 2^20 rows x 2048
// frames; 1000 energies (378, 222) 11.8 and 5.0 ms on 2^18 rows x 8192 frames.
std::vector<double> choose_levels(const Stream &s, BandForm &b, std::vector<double> *centre, BandCache &cache) {
    std::vector<double> best_w;
    double width = 0.0;
    const double dt = s.d.dt_fs * 1e-3 / kPlanck_meV_ps;
    for (int g = 0; g < s.n_wt; ++g) {
        const auto mm = std::minmax_element(s.E.begin() + (size_t)g * s.wt,
                                            s.E.begin() + std::min((size_t)(g + 1) * s.wt, s.E.size()));
        centre->push_back(0.5 * (*mm.first + *mm.second) * dt);
        width = std::max(width, (*mm.second - *mm.first) * dt);
    }
    const int ring = std::min(s.ring, s.T);
    const double best = (double)b.R / b.B * s.Nw_pad / 1.18;
    // the better length by the estimated rank, then its basis
    int best_S = 0;
    auto cost_of = [&](int S, int r, int *wt1, int *n1) {
        const int cols = s.n_wt * r;
        *n1 = (cols + kDrainMaxOmegaTile - 1) / kDrainMaxOmegaTile;
        *wt1 = (int)round_up((cols + *n1 - 1) / *n1, 16);
        return (double)b.R / b.B * (*n1 * (*wt1 + 8)) + (double)r / S * s.Nw_pad + 200.0 * cols / S;
    };
    int wt1 = 0, n1 = 0;
    double estimate = best;
    for (int S : {256, 512}) {
        if (S % b.B || S / b.B * b.R % 32 || S > ring || (s.needs_acc && s.ring % S)) continue;
        const int r = rank_guess(width * S);
        if (r > 56) continue;
        const double c = cost_of(S, (int)round_up(r, 8), &wt1, &n1);
        if (c < estimate) {
            estimate = c;
            best_S = S;
        }
    }
    if (!best_S) return best_w;
    const int S = best_S;
    int r = 0;
    const std::vector<double> &w = cache.basis(S, std::max(width, 1e-6), 4, 56, &r);
    if (r == 0) return best_w;
    // (the first level stores sectors of eight columns: other ranks are padded with zero vectors)
    const int rp = (int)round_up(r, 8), z_slots = (int)round_up((int64_t)((ring + S - 1) / S) * rp, 32);
    const double cost = cost_of(S, rp, &wt1, &n1);
    if (cost >= best || b.z_begin() + s.n_wt * z_slots > s.ring) return best_w;
    best_w.assign((size_t)(S / 2) * rp, 0.0);
    for (int u = 0; u < S / 2; ++u)
        for (int q = 0; q < r; ++q) best_w[(size_t)u * rp + (q < r / 2 ? q : q - r / 2 + rp / 2)] = w[(size_t)u * r + q];
    b.work = cost;
    b.S = S;
    b.r = rp;
    b.z_slots = z_slots;
    b.wt1 = wt1;
    b.n_wt1 = n1;
    return best_w;
}

}  // namespace

namespace tacaw {

tacaw_status build_band_forms(tacaw_plan_s *p, Stream &s, int64_t room_bytes, BandCache &cache, cudaStream_t st,
                              int only) {
    const bool split = p->prec == TACAW_PREC_SPLIT_BF16;
    if (p->in_place || (split && p->bf != 32) || s.T < kBandMinT) return TACAW_OK;
    const double dt_ps = s.d.dt_fs * 1e-3;
    double lo = s.E[0], hi = s.E[0];
    for (double e : s.E) {
        if (!(std::fabs(e) < 1e12)) return TACAW_OK;
        lo = std::min(lo, e);
        hi = std::max(hi, e);
    }
    const double beta = (hi - lo) * dt_ps / kPlanck_meV_ps;
    if (!(beta < 0.5)) return TACAW_OK;   // no form pays (R / B near 1)
    const double fc = 0.5 * (lo + hi) * dt_ps / kPlanck_meV_ps;
    const FormCost cost(p, s);
    const int most = std::min(s.ring, s.T);
    for (int B : {128, 64, 32}) {
        if (only && B != only) continue;
        if (!project_shape_ok(B, 8, split) || (s.needs_acc && s.ring % B)) continue;   // flushes end between blocks
        // no basis, tables or memory for what no push would use, first by the least work it could have (the rank is
        // no more than 2 below the guess; two levels of ranks of 8), then by what it has: on small plans the
        // launches' difference alone decides, and these are most of their creation
        const double ratio = (double)std::max(8, rank_guess(beta * B) - 4) / B;
        double least = ratio * s.Nw_pad;
        if (split) least = std::min(least, ratio * 8 * s.n_wt + 8.0 / 512 * s.Nw_pad);
        if (!only && !ever_picked(cost, s, B, least, most)) continue;
        int R = 0;
        const std::vector<double> &basis = cache.basis(B, std::max(beta, 1e-6), 8, 48, &R);
        if (basis.empty() || !project_shape_ok(B, R, split)) continue;
        const int blocks = (std::min(s.ring, s.T) + B - 1) / B;
        BandForm b;
        b.B = B;
        b.R = R;
        b.beta = beta;
        b.slots = split ? (int)round_up((int64_t)blocks * R, 32) : blocks * R;
        // behind the coefficients the ring's staging area holds the carry (8 B bytes a row) and, on the
        // split path (4 bytes a slot and row in A_hi), a scale a row
        if (b.slots + (split ? 2 * B + 1 : B) > s.ring) continue;
        BandTableArgs ba{};
        ba.B = B;
        ba.R = R;
        ba.fc = fc;
        ba.ring = s.ring;
        ba.slots = b.slots;
        ba.rounds = (s.T + s.ring - 1) / s.ring;
        b.work = (double)R / B * s.Nw_pad;
        std::vector<double> centre, w;
        if (split) w = choose_levels(s, b, &centre, cache);
        if (!only && !ever_picked(cost, s, B, b.work, most)) continue;
        // one allocation: twiddles, first-level table, responses (FP64), basis (FP64), modulation, the second
        // level's basis, group centres and each energy's
        const int K = b.S ? b.r : R;
        const size_t rows = (size_t)ba.rounds * (b.S ? b.z_slots : b.slots), n = basis.size();
        const size_t tp = (size_t)round_up(s.T, B), n1 = (size_t)b.wt1 * b.n_wt1;
        const size_t tw = rows * s.Nw_pad * 8;   // bytes of B_hi, of B_lo, or of B32
        const size_t t1 = b.S ? (size_t)b.S / B * R * n1 * 8 : 0;   // of T_hi, of T_lo
        const size_t bytes = (split ? 2 : 1) * tw + 2 * t1 +
                             ((size_t)K * s.Nw + n + tp + w.size() + centre.size() + s.Nw) * 8 + tp / B;
        if ((int64_t)bytes > room_bytes) continue;
        unsigned char *mem = nullptr;
        if (!dev_alloc(p, &mem, bytes)) break;   // no memory for this form's tables: frames, or the form built before
        room_bytes -= (int64_t)bytes;
        unsigned char *q = mem;
        if (split) {
            b.B_hi = reinterpret_cast<__nv_bfloat16 *>(q);
            b.B_lo = reinterpret_cast<__nv_bfloat16 *>(q + tw);
            q += 2 * tw;
            b.T_hi = reinterpret_cast<__nv_bfloat16 *>(q);
            b.T_lo = reinterpret_cast<__nv_bfloat16 *>(q + t1);
            q += 2 * t1;
        } else {
            b.B32 = reinterpret_cast<float2 *>(q);
            q += tw;
        }
        double *d_resp = reinterpret_cast<double *>(q);
        double *d_basis = d_resp + (size_t)K * s.Nw;
        b.mod = reinterpret_cast<float2 *>(d_basis + n);
        double *d_w = reinterpret_cast<double *>(b.mod + tp), *d_centre = d_w + w.size(), *d_cj = d_centre + centre.size();
        b.growth = reinterpret_cast<unsigned char *>(d_cj + s.Nw);
        b.basis.assign(basis.begin(), basis.end());
        CU_CHECK(p, cudaMemcpy(d_basis, basis.data(), sizeof(double) * n, cudaMemcpyHostToDevice), "basis");
        ba.basis = d_basis;
        const TableArgs ta = stream_table_args(s, p->bf);
        CU_CHECK(p, launch_band_mod(ta, ba, b.mod, st), "band modulation");
        if (split) CU_CHECK(p, launch_band_growth(ta, ba, b.mod, b.growth, st), "band window growth");
        if (b.S) {
            // first level, then the tiles' twiddles as those of blocks of S frames about each tile's centre
            std::vector<double> cj(s.Nw);
            for (int j = 0; j < s.Nw; ++j) cj[j] = centre[j / s.wt];
            CU_CHECK(p, cudaMemcpy(d_w, w.data(), sizeof(double) * w.size(), cudaMemcpyHostToDevice), "basis");
            CU_CHECK(p, cudaMemcpy(d_centre, centre.data(), sizeof(double) * centre.size(), cudaMemcpyHostToDevice), "centres");
            CU_CHECK(p, cudaMemcpy(d_cj, cj.data(), sizeof(double) * s.Nw, cudaMemcpyHostToDevice), "centres");
            BandMergeArgs ma{};
            ma.b = ba;
            ma.S = b.S;
            ma.r = b.r;
            ma.groups = s.n_wt;
            ma.cols_pad = (int)n1;
            ma.w = d_w;
            ma.fg = d_centre;
            CU_CHECK(p, launch_band_merge(ma, b.T_hi, b.T_lo, st), "band merge table");
            ba.B = b.S;
            ba.R = b.r;
            ba.basis = d_w;
            ba.fcj = d_cj;
            ba.slots = b.z_slots;
        }
        CU_CHECK(p, launch_band_response(ta, ba, d_resp, st), "band response");
        CU_CHECK(p, launch_band_twiddles(ta, ba, d_resp, b.B_hi, b.B_lo, b.B32, st), "band twiddles");
        s.band[s.n_band++] = b;
        s.shift_mean = !s.d.subtract_mean;
    }
    return TACAW_OK;
}

void share_band_forms(const Stream &from, Stream &s) {
    std::copy(from.band, from.band + kBandForms, s.band);
    s.n_band = from.n_band;
    s.shift_mean = from.shift_mean;
}

// The form with the least time (FormCost).  Both sides at the line: six partitions pushed 16 frames at a time,
// 300 energies: frames 14.9 + 20.1 ms, blocks of 32 with half their frames carried 21.2 + 11.0 ms.
int choose_form(const tacaw_plan_s *p, const Stream &s, int n, int first, bool band_only) {
    const FormCost c(p, s);
    double best = band_only ? HUGE_VAL : c.frames(n);
    int form = -1;
    for (int i = 0; i < s.n_band; ++i) {
        const double cost = c.blocks(n, s.band[i].B, s.band[i].work, first);
        if (cost < best) {
            best = cost;
            form = i;
        }
    }
    return form;
}

}  // namespace tacaw
