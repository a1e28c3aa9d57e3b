// Window and twiddle tables (built once per plan, on the GPU, in FP64).
//
// Phase of energy j at frame t: theta_jt = 2 pi frac(c_j t), c_j = E_j dt / h cycles per
// frame (App. B: energies are resolved up to eps = h/(2 dt)).  The fractional part is
// taken in FP64; on an FFT grid (E_j = j h/(T dt)) it is the exact integer form
// ((j t) mod T) / T.  Trigonometry is CUDA's FP64 sincospi/cospi.
// Windows follow Sec. III.A / App. A (scipy's periodic forms; length-1 windows are [1]).
#include "tacaw_internal.cuh"

namespace tacaw {

enum { WIN_RECT = 0, WIN_HANN = 1, WIN_GAUSS = 2, WIN_TUKEY = 3, WIN_BLACKMANHARRIS = 4, WIN_KAISER = 5,
       WIN_CHEBWIN = 6 };

// Modified Bessel function I0 by its power series sum_k ((x/2)^k / k!)^2, FP64 (x <= 60)
__device__ double bessel_i0(double x) {
    const double q = 0.25 * x * x;
    double term = 1.0, total = 1.0;
    for (int k = 1; k < 200; ++k) {
        term *= q / ((double)k * (double)k);
        total += term;
        if (term <= 1e-18 * total) break;
    }
    return total;
}

__device__ double window_value(const TableArgs &a, int t) {
    const int kind = a.window, T = a.T;
    const double param = a.window_param;
    if (T == 1) return 1.0;
    switch (kind) {
        case WIN_RECT:
            return 1.0;
        case WIN_HANN:
            return 0.5 - 0.5 * cospi(2.0 * (double)t / (double)T);
        case WIN_GAUSS: {
            double s = param > 0.0 ? param : (double)T / 6.0;
            double z = ((double)t - 0.5 * (double)T) / s;
            return exp(-0.5 * z * z);
        }
        case WIN_TUKEY: {
            double alpha = param;
            if (alpha <= 0.0) return 1.0;
            if (alpha >= 1.0) return 0.5 - 0.5 * cospi(2.0 * (double)t / (double)T);
            double edge = alpha * (double)T / 2.0;
            if ((double)t < edge) return 0.5 * (1.0 - cospi((double)t / edge));
            if ((double)t > (double)T - edge) return 0.5 * (1.0 - cospi((double)(T - t) / edge));
            return 1.0;
        }
        case WIN_BLACKMANHARRIS: {
            const double x = 2.0 * (double)t / (double)T;   // in units of pi
            return 0.35875 - 0.48829 * cospi(x) + 0.14128 * cospi(2.0 * x) - 0.01168 * cospi(3.0 * x);
        }
        case WIN_KAISER: {
            const double u = 2.0 * (double)t / (double)T - 1.0;
            const double r = 1.0 - u * u;
            return bessel_i0(param * sqrt(r > 0.0 ? r : 0.0)) / bessel_i0(param);
        }
        case WIN_CHEBWIN:
            return a.win_table ? a.win_table[t] : 1.0;
    }
    return 1.0;
}

// exp(-i theta_jt) = (cos, -sin) of 2 pi f, f = frac(c_j t) in [0, 1)
__device__ void twiddle(const TableArgs &a, int j, int t, double &c, double &s) {
    double f;
    if (a.fft_bins) {
        long long r = ((long long)j * (long long)t) % (long long)a.T;
        f = (double)r / (double)a.T;
    } else {
        double x = a.cj[j] * (double)t;
        f = x - floor(x);
    }
    sincospi(2.0 * f, &s, &c);
}

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// fp16 pieces (split-FP16 path), stored in the bf16-typed table as raw 16-bit patterns;
// |B| <= 1, so no scaling: residuals below the fp16 normal range keep an absolute
// resolution of 2^-24, far below the 2^-22 relative resolution of the largest twiddles
__device__ __forceinline__ void split_f16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
    const __half h = __float2half_rn(x);
    const __half l = __float2half_rn(x - __half2float(h));
    hi = __ushort_as_bfloat16(__half_as_ushort(h));
    lo = __ushort_as_bfloat16(__half_as_ushort(l));
}

// One thread per (energy j < Nw_pad, frame t < T_pad).  Rows 2j and 2j+1 of block t/bf
// (rows of 2*bf bf16) receive, at elements 2(t%bf) and 2(t%bf)+1, the real embedding of
// B = w_t exp(-i theta):
//   row 2j   : ( Re B, -Im B)  ->  Re Psi_j = Re psi Re B - Im psi Im B
//   row 2j+1 : ( Im B,  Re B)  ->  Im Psi_j = Re psi Im B + Im psi Re B
template <bool F16>
__global__ void twiddles_split_kernel(TableArgs a, __nv_bfloat16 *B_hi, __nv_bfloat16 *B_lo) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    int t = blockIdx.y * blockDim.y + threadIdx.y;
    if (j >= a.Nw_pad || t >= a.T_pad) return;
    double br = 0.0, bi = 0.0;
    if (j < a.Nw && t < a.T) {
        double c, s;
        twiddle(a, j, t, c, s);
        double w = window_value(a, t);
        br = w * c;
        bi = -w * s;
    }
    const int bf = a.block_frames;
    const int kb = t / bf, tt = t % bf;
    const size_t rows = 2 * (size_t)a.Nw_pad;
    // word tt (a bf16 pair) of rows 2j and 2j+1; pre-swizzled rows keep their 16-byte chunks
    // where the tensor core's shared-memory swizzle of the row width expects them
    const int cpr = bf >> 2;
    const int sw0 = a.swz ? (int)(((2 * j * cpr) >> 3) & (cpr - 1)) : 0;
    const int sw1 = a.swz ? (int)((((2 * j + 1) * cpr) >> 3) & (cpr - 1)) : 0;
    const int w0 = (((tt >> 2) ^ sw0) << 2) | (tt & 3), w1 = (((tt >> 2) ^ sw1) << 2) | (tt & 3);
    const size_t r0 = ((size_t)kb * rows + 2 * (size_t)j) * (2 * bf) + 2 * w0;
    const size_t r1 = ((size_t)kb * rows + 2 * (size_t)j + 1) * (2 * bf) + 2 * w1;
    float v0[2] = {(float)br, (float)(-bi)};
    float v1[2] = {(float)bi, (float)br};
    for (int e = 0; e < 2; ++e) {
        __nv_bfloat16 h, l;
        if (F16) split_f16(v0[e], h, l);
        else split_bf16(v0[e], h, l);
        B_hi[r0 + e] = h;
        B_lo[r0 + e] = l;
        if (F16) split_f16(v1[e], h, l);
        else split_bf16(v1[e], h, l);
        B_hi[r1 + e] = h;
        B_lo[r1 + e] = l;
    }
}

// Table of the adjoint's back-projection C[m, t] = sum_j G[m, j] conj(B[t, j]): frames are the
// output columns and energies the contraction.  One thread per (energy j < e_pad, frame
// t < t_rows); b = conj(w_t exp(-i theta_jt)) = w_t exp(+i theta_jt) goes to elements 2(j%32),
// 2(j%32)+1 of rows 2t and 2t+1 of block j/32 (rows of 32 bf16 pairs, pre-swizzled):
//   row 2t   : ( Re b, -Im b)  ->  Re C_t = Re G Re b - Im G Im b
//   row 2t+1 : ( Im b,  Re b)  ->  Im C_t = Re G Im b + Im G Re b
__global__ void twiddles_adjoint_split_kernel(TableArgs a, int t_rows, int e_pad, __nv_bfloat16 *B_hi,
                                              __nv_bfloat16 *B_lo) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y * blockDim.y + threadIdx.y;
    if (j >= e_pad || t >= t_rows) return;
    double br = 0.0, bi = 0.0;
    if (j < a.Nw && t < a.T) {
        double c, s;
        twiddle(a, j, t, c, s);
        const double w = window_value(a, t);
        br = w * c;
        bi = w * s;
    }
    const int kb = j / 32, jj = j % 32;
    const size_t rows = 2 * (size_t)t_rows;
    const int r0 = 2 * t, r1 = 2 * t + 1;
    // 128-byte rows: chunk c of row r stored at c ^ (r mod 8)
    const int w0 = (((jj >> 2) ^ (r0 & 7)) << 2) | (jj & 3), w1 = (((jj >> 2) ^ (r1 & 7)) << 2) | (jj & 3);
    const size_t o0 = ((size_t)kb * rows + (size_t)r0) * 64 + 2 * (size_t)w0;
    const size_t o1 = ((size_t)kb * rows + (size_t)r1) * 64 + 2 * (size_t)w1;
    const float v0[2] = {(float)br, (float)(-bi)};
    const float v1[2] = {(float)bi, (float)br};
    for (int e = 0; e < 2; ++e) {
        __nv_bfloat16 h, l;
        split_bf16(v0[e], h, l);
        B_hi[o0 + e] = h;
        B_lo[o0 + e] = l;
        split_bf16(v1[e], h, l);
        B_hi[o1 + e] = h;
        B_lo[o1 + e] = l;
    }
}

__global__ void twiddles_fp32_kernel(TableArgs a, float2 *B32) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    int t = blockIdx.y * blockDim.y + threadIdx.y;
    if (j >= a.Nw_pad || t >= a.T_pad) return;
    float2 v = make_float2(0.f, 0.f);
    if (j < a.Nw && t < a.T) {
        double c, s;
        twiddle(a, j, t, c, s);
        double w = window_value(a, t);
        v = make_float2((float)(w * c), (float)(-w * s));
    }
    B32[(size_t)t * a.Nw_pad + j] = v;
}

// W(E_j) = sum_t w_t exp(-i theta_jt), one block per energy, fixed-order tree reduction.
__global__ void window_transform_kernel(TableArgs a, float2 *Wc) {
    const int j = blockIdx.x;
    double sr = 0.0, si = 0.0;
    for (int t = threadIdx.x; t < a.T; t += blockDim.x) {
        double c, s;
        twiddle(a, j, t, c, s);
        double w = window_value(a, t);
        sr += w * c;
        si -= w * s;
    }
    __shared__ double rr[256], ri[256];
    rr[threadIdx.x] = sr;
    ri[threadIdx.x] = si;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
            rr[threadIdx.x] += rr[threadIdx.x + h];
            ri[threadIdx.x] += ri[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) Wc[j] = make_float2((float)rr[0], (float)ri[0]);
}

__global__ void window_values_kernel(TableArgs a, float *w) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < a.T) w[t] = (float)window_value(a, t);
}

// ---- band-limited staging form ----------------------------------------------------------
// Psi_j = sum_t y_t w_t exp(-2 pi i c_j t) block by block: with t = t0 + u inside a block of B frames,
// centre c = (B-1)/2, and m[t] = w_t exp(-2 pi i f_c (u - c)),
//   sum_u y w exp(-2 pi i c_j t) = exp(-2 pi i c_j (t0 + c)) sum_u (m y)_u exp(-2 pi i (c_j - f_c)(u - c))
// and the last exponential, |c_j - f_c| <= beta/2, is expanded on the R basis vectors v_q (real,
// orthonormal, even or odd): its coefficients are q_resp[q][j] = sum_u v_q[u] exp(-2 pi i d (u - c)),
//   even: 2 sum_{u < B/2} v cos(2 pi d (u - c)),   odd: -2 i sum_{u < B/2} v sin(2 pi d (u - c)).

__global__ void band_mod_kernel(TableArgs a, int B, double fc, int n, float2 *mod) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    float2 v = make_float2(0.f, 0.f);
    if (t < a.T) {
        double c, s;
        sincospi(2.0 * fc * ((double)(t % B) - 0.5 * (double)(B - 1)), &s, &c);
        const double w = window_value(a, t);
        v = make_float2((float)(w * c), (float)(-w * s));
    }
    mod[t] = v;
}

// One CTA per ring of `per` blocks (n in all): exponents of the blocks' largest |mod|, then of the ring's over them.
__global__ void band_growth_kernel(int B, int per, int n, int total, const float2 *mod, unsigned char *growth) {
    constexpr int kZero = -1000;                      // a block of zeros
    __shared__ int top;
    const int b0 = blockIdx.x * per, b1 = min(b0 + per, n);
    auto exponent = [&](int blk) {
        float w = 0.f;
        for (int u = 0; u < B && blk * B + u < total; ++u)
            w = fmaxf(w, fmaxf(fabsf(mod[blk * B + u].x), fabsf(mod[blk * B + u].y)));
        return w > 0.f ? ilogbf(w) : kZero;
    };
    if (threadIdx.x == 0) top = kZero;
    __syncthreads();
    for (int blk = b0 + (int)threadIdx.x; blk < b1; blk += blockDim.x) atomicMax(&top, exponent(blk));
    __syncthreads();
    for (int blk = b0 + (int)threadIdx.x; blk < b1; blk += blockDim.x) {
        const int x = exponent(blk);
        growth[blk] = (unsigned char)(x == kZero ? 0 : min(top - x, 255));
    }
}

// (c, s) of the next place along an even grid of angles: rotation by the step's (cd, sd), whose FP64 rounding over up
// to 512 steps stays below 1e-13 (an FP64 sincospi at each was most of the tables' time)
__device__ __forceinline__ void rotate(double &c, double &s, double cd, double sd) {
    const double x = c * cd - s * sd;
    s = s * cd + c * sd;
    c = x;
}

// one thread per (energy, basis vector); a.cj holds c_j for FFT grids too
__global__ void band_response_kernel(TableArgs a, BandTableArgs b, double *q_resp) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y;
    if (j >= a.Nw) return;
    const double d = a.cj[j] - (b.fcj ? b.fcj[j] : b.fc);
    double acc = 0.0, c, s, cd, sd;
    sincospi(-d * (double)(b.B - 1), &s, &c);
    sincospi(2.0 * d, &sd, &cd);
    for (int u = 0; u < b.B / 2; ++u) {
        acc += b.basis[u * b.R + q] * (q >= b.R / 2 ? -2.0 * s : 2.0 * c);
        rotate(c, s, cd, sd);
    }
    q_resp[(size_t)q * a.Nw + j] = acc;
}

// One thread per (energy j < Nw_pad, block): the R table rows of block k of flush f.  The split path
// takes fp16 pieces (|B| is at most about sqrt(B)).
__global__ void band_twiddles_kernel(TableArgs a, BandTableArgs b, const double *q_resp, __nv_bfloat16 *B_hi,
                                     __nv_bfloat16 *B_lo, float2 *B32) {
    const int per = (b.slots + b.R - 1) / b.R;      // blocks a flush's table rows hold (the last may be padding)
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y * blockDim.y + threadIdx.y;
    if (j >= a.Nw_pad || n >= b.rounds * per) return;
    const int f = n / per, k = n % per;
    const long long t0 = (long long)f * b.ring + (long long)k * b.B;
    const bool in = j < a.Nw && k * b.B < b.ring && t0 < a.T;
    double c = 0.0, s = 0.0;
    if (in) {
        // phase at the block's centre, in half frames: c_j (2 t0 + B - 1) / 2
        const long long h = 2 * t0 + b.B - 1;
        if (a.fft_bins) {
            const long long r = ((long long)j * h) % (2LL * a.T);
            sincospi((double)r / (double)a.T, &s, &c);
        } else {
            const double x = a.cj[j] * 0.5 * (double)h;
            sincospi(2.0 * (x - floor(x)), &s, &c);
        }
    }
    const size_t rows = 2 * (size_t)a.Nw_pad;
    const int n0 = 2 * j, n1 = 2 * j + 1;
    for (int q = 0; q < b.R && k * b.R + q < b.slots; ++q) {
        const double g = in ? q_resp[(size_t)q * a.Nw + j] : 0.0;
        // (c - i s) g, times i for the odd vectors (whose q_resp is the imaginary part)
        const bool odd = q >= b.R / 2;
        const float br = (float)(odd ? s * g : c * g), bi = (float)(odd ? c * g : -s * g);
        const int row = f * b.slots + k * b.R + q;
        if (B32) {
            B32[(size_t)row * a.Nw_pad + j] = make_float2(br, bi);
            continue;
        }
        const int kb = row / 32, tt = row % 32;
        const int w0 = (((tt >> 2) ^ (n0 & 7)) << 2) | (tt & 3), w1 = (((tt >> 2) ^ (n1 & 7)) << 2) | (tt & 3);
        const size_t r0 = ((size_t)kb * rows + (size_t)n0) * 64 + 2 * (size_t)w0;
        const size_t r1 = ((size_t)kb * rows + (size_t)n1) * 64 + 2 * (size_t)w1;
        const float v0[2] = {br, -bi}, v1[2] = {bi, br};
        for (int e = 0; e < 2; ++e) {
            __nv_bfloat16 h, l;
            split_f16(v0[e], h, l);
            B_hi[r0 + e] = h;
            B_lo[r0 + e] = l;
            split_f16(v1[e], h, l);
            B_hi[r1 + e] = h;
            B_lo[r1 + e] = l;
        }
    }
}

// Second-level coefficient p of energy group g over a superblock: sum_t x_t w_p[t] exp(-2 pi i f_g (t - (S-1)/2)),
// x_t = exp(2 pi i f_c (u - c)) sum_q z[k, q] v_q[u] for t = k B + u.  One thread per (column g r + p, slot k R + q).
__global__ void band_merge_kernel(BandMergeArgs m, __nv_bfloat16 *T_hi, __nv_bfloat16 *T_lo) {
    const int col = blockIdx.x * blockDim.x + threadIdx.x, slot = blockIdx.y * blockDim.y + threadIdx.y;
    const int B = m.b.B, R = m.b.R;
    if (col >= m.cols_pad || slot >= m.S / B * R) return;
    double ar = 0.0, ai = 0.0;
    if (col < m.groups * m.r) {
        const int g = col / m.r, p = col % m.r, k = slot / R, q = slot % R;
        const double fg = m.fg[g], c0 = 0.5 * (double)(B - 1);
        const bool odd_v = q >= R / 2, odd_w = p >= m.r / 2;
        double sr = 0.0, si = 0.0, s, c, sd, cd;
        sincospi(-2.0 * (m.b.fc - fg) * c0, &s, &c);
        sincospi(2.0 * (m.b.fc - fg), &sd, &cd);
        for (int u = 0; u < B; ++u) {
            const double v = u < B / 2 ? m.b.basis[u * R + q] : (odd_v ? -1.0 : 1.0) * m.b.basis[(B - 1 - u) * R + q];
            const int t = k * B + u;
            const double w = t < m.S / 2 ? m.w[t * m.r + p] : (odd_w ? -1.0 : 1.0) * m.w[(m.S - 1 - t) * m.r + p];
            sr += v * w * c;
            si += v * w * s;
            rotate(c, s, cd, sd);
        }
        sincospi(-2.0 * fg * ((double)(k * B) + c0 - 0.5 * (double)(m.S - 1)), &s, &c);
        ar = sr * c - si * s;
        ai = sr * s + si * c;
    }
    const int kb = slot / 32, tt = slot % 32, n0 = 2 * col, n1 = 2 * col + 1;
    const int w0 = (((tt >> 2) ^ (n0 & 7)) << 2) | (tt & 3), w1 = (((tt >> 2) ^ (n1 & 7)) << 2) | (tt & 3);
    const size_t rows = 2 * (size_t)m.cols_pad;
    const size_t r0 = ((size_t)kb * rows + (size_t)n0) * 64 + 2 * (size_t)w0;
    const size_t r1 = ((size_t)kb * rows + (size_t)n1) * 64 + 2 * (size_t)w1;
    const float v0[2] = {(float)ar, (float)(-ai)}, v1[2] = {(float)ai, (float)ar};
    for (int e = 0; e < 2; ++e) {
        __nv_bfloat16 h, l;
        split_f16(v0[e], h, l);
        T_hi[r0 + e] = h;
        T_lo[r0 + e] = l;
        split_f16(v1[e], h, l);
        T_hi[r1 + e] = h;
        T_lo[r1 + e] = l;
    }
}

cudaError_t launch_band_merge(const BandMergeArgs &m, __nv_bfloat16 *T_hi, __nv_bfloat16 *T_lo, cudaStream_t st) {
    const int slots = m.S / m.b.B * m.b.R;
    band_merge_kernel<<<dim3((m.cols_pad + 31) / 32, (slots + 3) / 4), dim3(32, 4), 0, st>>>(m, T_hi, T_lo);
    return cudaGetLastError();
}

cudaError_t launch_band_mod(const TableArgs &t, const BandTableArgs &b, float2 *mod, cudaStream_t st) {
    const int n = (t.T + b.B - 1) / b.B * b.B;
    band_mod_kernel<<<(n + 127) / 128, 128, 0, st>>>(t, b.B, b.fc, n, mod);
    return cudaGetLastError();
}

cudaError_t launch_band_growth(const TableArgs &t, const BandTableArgs &b, const float2 *mod, unsigned char *growth,
                               cudaStream_t st) {
    const int n = (t.T + b.B - 1) / b.B;
    band_growth_kernel<<<b.rounds, 256, 0, st>>>(b.B, b.rounds > 1 ? b.ring / b.B : n, n, n * b.B, mod, growth);
    return cudaGetLastError();
}

cudaError_t launch_band_response(const TableArgs &t, const BandTableArgs &b, double *q_resp, cudaStream_t st) {
    band_response_kernel<<<dim3((t.Nw + 63) / 64, b.R), 64, 0, st>>>(t, b, q_resp);
    return cudaGetLastError();
}

cudaError_t launch_band_twiddles(const TableArgs &t, const BandTableArgs &b, const double *q_resp,
                                 __nv_bfloat16 *B_hi, __nv_bfloat16 *B_lo, float2 *B32, cudaStream_t st) {
    const dim3 blk(32, 8);
    const dim3 grd((t.Nw_pad + 31) / 32, (b.rounds * ((b.slots + b.R - 1) / b.R) + 7) / 8);
    band_twiddles_kernel<<<grd, blk, 0, st>>>(t, b, q_resp, B_hi, B_lo, B32);
    return cudaGetLastError();
}

cudaError_t launch_twiddles_split(const TableArgs &t, __nv_bfloat16 *B_hi, __nv_bfloat16 *B_lo, int f16,
                                  cudaStream_t st) {
    dim3 blk(32, 8);
    dim3 grd((t.Nw_pad + 31) / 32, (t.T_pad + 7) / 8);
    if (f16)
        twiddles_split_kernel<true><<<grd, blk, 0, st>>>(t, B_hi, B_lo);
    else
        twiddles_split_kernel<false><<<grd, blk, 0, st>>>(t, B_hi, B_lo);
    return cudaGetLastError();
}

cudaError_t launch_twiddles_adjoint_split(const TableArgs &t, int t_rows, int e_pad, __nv_bfloat16 *B_hi,
                                          __nv_bfloat16 *B_lo, cudaStream_t st) {
    dim3 blk(32, 8);
    dim3 grd((e_pad + 31) / 32, (t_rows + 7) / 8);
    twiddles_adjoint_split_kernel<<<grd, blk, 0, st>>>(t, t_rows, e_pad, B_hi, B_lo);
    return cudaGetLastError();
}

cudaError_t launch_twiddles_fp32(const TableArgs &t, float2 *B32, cudaStream_t st) {
    dim3 blk(32, 8);
    dim3 grd((t.Nw_pad + 31) / 32, (t.T_pad + 7) / 8);
    twiddles_fp32_kernel<<<grd, blk, 0, st>>>(t, B32);
    return cudaGetLastError();
}

cudaError_t launch_window_transform(const TableArgs &t, float2 *Wc, cudaStream_t st) {
    window_transform_kernel<<<t.Nw, 256, 0, st>>>(t, Wc);
    return cudaGetLastError();
}

cudaError_t launch_window_values(const TableArgs &t, float *w, cudaStream_t st) {
    window_values_kernel<<<(t.T + 255) / 256, 256, 0, st>>>(t, w);
    return cudaGetLastError();
}

}  // namespace tacaw
