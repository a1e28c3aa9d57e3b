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
    // the k-th sequence's first half, the whole sequence of unit norm (norm sqrt(1/2))
    std::vector<double> vector(int k) const {
        double a = lo, b = hi;   // the k-th largest eigenvalue
        for (int i = 0; i < 80 && b - a > 4e-16 * std::max(std::fabs(a), std::fabs(b)); ++i) {
            const double x = 0.5 * (a + b);
            (above(x) > k ? a : b) = x;
        }
        const double x = 0.5 * (a + b) + 1e-13 * (hi - lo);   // off the eigenvalue: the solves stay finite
        std::vector<double> v(H, 1.0);
        for (int u = 0; u < H; ++u) v[u] += 0.01 * (u % 7);   // no symmetry that could hide a vector
        for (int it = 0; it < 4; ++it) {
            solve(x, v);
            double n = 0.0;
            for (double t : v) n += t * t;
            for (double &t : v) t *= std::sqrt(0.5 / n);
        }
        return v;
    }

private:
    int H;
    std::vector<double> d, o;
    double lo, hi;
    // eigenvalues above x: positive pivots of A - x
    int above(double x) const {
        int n = 0;
        double q = 1.0;
        for (int u = 0; u < H; ++u) {
            q = d[u] - x - (u ? o[u] * o[u] / q : 0.0);
            if (q == 0.0) q = 1e-300;
            n += q > 0.0;
        }
        return n;
    }
    // v <- (A - x)^-1 v, Gaussian elimination with row exchanges (three diagonals above)
    void solve(double x, std::vector<double> &v) const {
        std::vector<double> a(H), b(H, 0.0), c(H, 0.0);   // the current upper rows: a b c at columns u, u+1, u+2
        double p = d[0] - x, q = H > 1 ? o[1] : 0.0;       // row u as eliminated so far
        for (int u = 0; u < H; ++u) {
            if (u + 1 == H) {
                a[u] = p == 0.0 ? 1e-300 : p;
                break;
            }
            const double l = o[u + 1], dn = d[u + 1] - x, on = u + 2 < H ? o[u + 2] : 0.0;
            if (std::fabs(p) >= std::fabs(l)) {
                a[u] = p == 0.0 ? 1e-300 : p;
                b[u] = q;
                const double m = l / a[u];
                p = dn - m * q;
                q = on;
                v[u + 1] -= m * v[u];
            } else {
                a[u] = l;
                b[u] = dn;
                c[u] = on;
                const double m = p / l;
                p = q - m * dn;
                q = -m * on;
                const double t = v[u];
                v[u] = v[u + 1];
                v[u + 1] = t - m * v[u];
            }
        }
        for (int u = H - 1; u >= 0; --u) {
            double t = v[u];
            if (u + 1 < H) t -= b[u] * v[u + 1];
            if (u + 2 < H) t -= c[u] * v[u + 2];
            v[u] = t / a[u];
        }
    }
};

// Basis [B/2][R] of the band |d| <= beta/2 (a row: R/2 even vectors, R/2 odd) of the least rank R that
// the push kernels take whose residual over the band stays within tol; R = 0 if none does.  The residual
// is the part of exp(-2 pi i d (u - c)) outside the basis, relative to its norm, checked on a grid of
// d that holds the band's edge, where it is largest.
std::vector<double> band_basis(int B, double beta, double tol, bool split, int *rank) {
    const int H = B / 2, kD = 9;
    const Prolate even(B, beta, 0), odd(B, beta, 1);
    std::vector<std::vector<double>> vec, res(2 * kD, std::vector<double>(H));
    for (int i = 0; i < kD; ++i)
        for (int u = 0; u < H; ++u) {
            const double ph = 2.0 * M_PI * (0.5 * beta * i / (kD - 1)) * (u - 0.5 * (B - 1));
            res[2 * i][u] = std::cos(ph);
            res[2 * i + 1][u] = std::sin(ph);
        }
    *rank = 0;
    for (int R = 4; R == 4 || project_shape_ok(B, R, split); R += 4) {
        while ((int)vec.size() < R) {
            const int par = (int)vec.size() & 1;
            vec.push_back((par ? odd : even).vector((int)vec.size() / 2));
            for (int i = 0; i < kD; ++i) {
                std::vector<double> &r = res[2 * i + par];
                double dot = 0.0;
                for (int u = 0; u < H; ++u) dot += 2.0 * vec.back()[u] * r[u];
                for (int u = 0; u < H; ++u) r[u] -= dot * vec.back()[u];
            }
        }
        if (R < 8) continue;
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

// Segments and rings shorter than this keep staging frames: their passes are bound by launches.
constexpr int kBandMinT = 512;


}  // namespace

namespace tacaw {

tacaw_status build_band_forms(tacaw_plan_s *p, Stream &s, int64_t room_bytes, cudaStream_t st) {
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
    for (int B : {32, 64, 128}) {
        if (!project_shape_ok(B, 8, split) || (s.needs_acc && s.ring % B)) continue;   // flushes end between blocks
        int R = 0;
        const std::vector<double> basis = band_basis(B, std::max(beta, 1e-6), kBandTol, split, &R);
        if (R == 0) continue;
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
        // one allocation: twiddles, responses (FP64), basis (FP64), modulation
        const size_t rows = (size_t)ba.rounds * b.slots, n = basis.size(), tp = (size_t)round_up(s.T, B);
        const size_t tw = rows * s.Nw_pad * 8;   // bytes of B_hi, of B_lo, or of B32
        const size_t bytes = (split ? 2 : 1) * tw + ((size_t)R * s.Nw + n + tp) * 8;
        if ((int64_t)bytes > room_bytes) continue;
        unsigned char *mem = nullptr;
        if (!dev_alloc(p, &mem, bytes)) break;   // no memory for this form's tables: frames, or the form built before
        room_bytes -= (int64_t)bytes;
        unsigned char *q = mem;
        if (split) {
            b.B_hi = reinterpret_cast<__nv_bfloat16 *>(q);
            b.B_lo = reinterpret_cast<__nv_bfloat16 *>(q + tw);
            q += 2 * tw;
        } else {
            b.B32 = reinterpret_cast<float2 *>(q);
            q += tw;
        }
        double *d_resp = reinterpret_cast<double *>(q);
        double *d_basis = d_resp + (size_t)R * s.Nw;
        b.mod = reinterpret_cast<float2 *>(d_basis + n);
        b.basis.assign(basis.begin(), basis.end());
        CU_CHECK(p, cudaMemcpy(d_basis, basis.data(), sizeof(double) * n, cudaMemcpyHostToDevice), "basis");
        ba.basis = d_basis;
        const TableArgs ta = stream_table_args(s, p->bf);
        CU_CHECK(p, launch_band_mod(ta, ba, b.mod, st), "band modulation");
        CU_CHECK(p, launch_band_response(ta, ba, d_resp, st), "band response");
        CU_CHECK(p, launch_band_twiddles(ta, ba, d_resp, b.B_hi, b.B_lo, b.B32, st), "band twiddles");
        s.band[s.n_band++] = b;
    }
    return TACAW_OK;
}

// The form with the least time a (row, frame), from measurements in picoseconds on 2^18 rows (16 to 64
// frames a push; 60 to 1000 energies): a push of frames 2.7 + 24 / n (5.7 where n is no multiple of 4 and
// takes the unaligned conversion); a push of whole blocks 2.2 + 36 / n, and where it ends inside blocks
// 3.2 for the share of the frames that pass through the carry and 16 / n for the extra launch's rows; the
// contraction 0.0128 (split) or 0.142 (FP32) an energy, times 1.25 or 1.12 R / B on coefficients (shorter
// sums under the same epilogue).
int choose_form(const tacaw_plan_s *p, const Stream &s, int n) {
    const bool split = p->prec == TACAW_PREC_SPLIT_BF16;
    const double energies = (split ? 0.0128 : 0.142) * s.Nw_pad, stretch = split ? 1.25 : 1.12;
    double best = 0.97 * ((n % 4 == 0 || !split ? 2.7 + 24.0 / n : 5.7) + energies);
    int form = -1;
    for (int i = 0; i < s.n_band; ++i) {
        const BandForm &b = s.band[i];
        // share of the frames that wait in the carry, taking the ring's other pushes to be like its first:
        // none for whole blocks, all but the completing push's for parts of a block, all for other sizes
        // below a block (they drift against the blocks), a block's worth for longer ones
        const double f = n % b.B == 0 ? 0.0 : b.B % n == 0 ? 1.0 - (double)n / b.B : n < b.B ? 1.0 : (double)b.B / n;
        const double push = 2.2 + 36.0 / std::max(n, 32) + (f > 0.0 ? 3.2 * f + 16.0 / n : 0.0);
        const double cost = push + stretch * b.R / b.B * energies;
        if (cost < best) {
            best = cost;
            form = i;
        }
    }
    return form;
}

}  // namespace tacaw
