// Syndrome and 8-dimensional reconciliation kernels.
//
// * qcldpc_syndrome: s = H x over GF(2) for the QC expansion of Sec. III-C,
//   one thread per word of 32 check nodes or, where rows are short, per check.
// * qcldpc_bob_message_8d / qcldpc_llr_8d: Sec. II-C. Bob sends M = U Y with
//   U_j = (-1)^{C_j}; Alice divides, R = M X^{-1} = M conj(X) / |X|^2, and
//   with sigma_N^2 = 8 sigma_Z^2 / |X|^2 the channel LLR of Step 1 of
//   Algorithm 1 becomes Q = 2R / sigma_N^2 = (M conj(X)) snr / 4: |X|^2
//   cancels, so the kernel needs one octonion product per block of eight.
//
// Octonions are pairs of quaternions with Cayley-Dickson doubling
// (p,q)(r,s) = (p r - conj(s) q, s p + q conj(r)); quaternions multiply by
// Hamilton's rule. One thread owns one block of eight floats, loaded and
// stored as two 16-byte vectors; the work is a pure stream (12 bytes per bit
// for the LLR map), bounded by HBM bandwidth.
#include "qcldpc_internal.cuh"

namespace {

struct Quat {
    float w, x, y, z;
};

__device__ __forceinline__ Quat qmul(Quat a, Quat b) {
    Quat r;
    r.w = a.w * b.w - a.x * b.x - a.y * b.y - a.z * b.z;
    r.x = a.w * b.x + a.x * b.w + a.y * b.z - a.z * b.y;
    r.y = a.w * b.y - a.x * b.z + a.y * b.w + a.z * b.x;
    r.z = a.w * b.z + a.x * b.y - a.y * b.x + a.z * b.w;
    return r;
}

__device__ __forceinline__ Quat qconj(Quat a) { return Quat{a.w, -a.x, -a.y, -a.z}; }
__device__ __forceinline__ Quat qadd(Quat a, Quat b) {
    return Quat{a.w + b.w, a.x + b.x, a.y + b.y, a.z + b.z};
}
__device__ __forceinline__ Quat qsub(Quat a, Quat b) {
    return Quat{a.w - b.w, a.x - b.x, a.y - b.y, a.z - b.z};
}
__device__ __forceinline__ Quat q4(float4 v) { return Quat{v.x, v.y, v.z, v.w}; }
__device__ __forceinline__ float4 f4(Quat q) { return make_float4(q.w, q.x, q.y, q.z); }

// (p, q)(r, s) = (p r - conj(s) q, s p + q conj(r))
__device__ __forceinline__ void omul(Quat p, Quat q, Quat r, Quat s, Quat &lo, Quat &hi) {
    lo = qsub(qmul(p, r), qmul(qconj(s), q));
    hi = qadd(qmul(s, p), qmul(q, qconj(r)));
}

// `len` (1 to 32) bits of a packed row from bit v on, in the low bits of the
// result. Reads only words that hold one of them.
__device__ __forceinline__ uint32_t bit_window(const uint32_t *__restrict__ words, int64_t v, int len) {
    const int64_t w = v >> 5;
    const int s = (int)(v & 31);
    const uint32_t lo = __ldg(words + w);
    const uint32_t hi = s + len > 32 ? __ldg(words + w + 1) : 0u;
    const uint32_t x = __funnelshift_r(lo, hi, s);
    return len == 32 ? x : x & ((1u << len) - 1u);
}

// One thread per packed word of 32 checks. Checks of one base row are
// consecutive, and circulant (col, shift) gives them consecutive bits of the
// column from (i + shift) mod Z on, so a word is the XOR of one 32-bit window
// per circulant (two where the window wraps at Z): two loads and a funnel
// shift serve 32 checks. A word that straddles base rows is put together from
// one segment per row. Bounded by launch latency and the L2's window reads.
// With one thread and one bit load per check and circulant, Bob's message,
// syndrome and Alice's LLRs of 16 frames of n = 10^6 took 149 us together;
// with words they take 63 us (the two maps' 320 MB alone need 47 us of HBM).
__global__ void __launch_bounds__(128) syndrome_kernel(const __grid_constant__ qc::Table T,
                                                       const uint32_t *__restrict__ bits,
                                                       uint32_t *__restrict__ syn,
                                                       int64_t words_n, int64_t words_m) {
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= words_m) return;
    const int Z = T.Z;
    const int64_t m = (int64_t)T.mb * Z;
    const uint32_t *fb = bits + (int64_t)blockIdx.y * words_n;
    int64_t c = w * 32;
    int r = (int)(c / Z), i = (int)(c - (int64_t)r * Z);
    uint32_t out = 0;
    for (int pos = 0; pos < 32 && c < m;) {
        const int len = min(32 - pos, Z - i);
        const int ke = T.row_ptr[r + 1];
        uint32_t par = 0;
        for (int k = T.row_ptr[r]; k < ke; k++) {
            const qc::RowEnt e = T.rows[k];
            const int64_t col0 = (int64_t)e.col * Z;
            int j = i + e.shift;
            if (j >= Z) j -= Z;
            const int first = min(len, Z - j);  // bits before the wrap
            par ^= bit_window(fb, col0 + j, first);
            if (first < len) par ^= bit_window(fb, col0, len - first) << first;
        }
        out |= par << pos;
        pos += len;
        c += len;
        i = 0;
        r++;
    }
    syn[(int64_t)blockIdx.y * words_m + w] = out;
}

// One thread per check, results packed with a warp ballot: for rows so short
// that a word of the other form would walk many of them one after the other.
__global__ void __launch_bounds__(256) syndrome_bit_kernel(const __grid_constant__ qc::Table T,
                                                           const uint32_t *__restrict__ bits,
                                                           uint32_t *__restrict__ syn,
                                                           int64_t words_n, int64_t words_m) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int Z = T.Z;
    const bool on = c < (int64_t)T.mb * Z;
    const uint32_t *fb = bits + (int64_t)blockIdx.y * words_n;
    uint32_t par = 0;
    if (on) {
        const int r = (int)(c / Z), i = (int)(c - (int64_t)r * Z);
        const int ke = T.row_ptr[r + 1];
        for (int k = T.row_ptr[r]; k < ke; k++) {
            const qc::RowEnt e = T.rows[k];
            int j = i + e.shift;
            if (j >= Z) j -= Z;
            const int64_t v = (int64_t)e.col * Z + j;
            par ^= __ldg(fb + (v >> 5)) >> (v & 31) & 1u;
        }
    }
    const uint32_t word = __ballot_sync(0xffffffffu, par);
    if ((threadIdx.x & 31) == 0 && on) syn[(int64_t)blockIdx.y * words_m + (c >> 5)] = word;
}

// Whether a syndrome call takes the word form. A word meets `seg` rows at most
// (it starts at a multiple of gcd(Z, 32) in a row) and its thread reads their
// circulants one after the other, so the word form's latency grows with their
// product. A few thousand checks of 7 circulants took it 53 us at Z = 1, 10.3 at
// 8 and 15 (28 reads), 6.2 at 16 (14), and the bit form 4.8 (the call's host
// time) at each of them. Up to 18 reads the word form is at most 1.5 us behind
// there and ahead from a few hundred thousand checks on (one multi-edge frame,
// Z = 625, 16 reads: 6.2 and 10.3 us). Above a million checks the number of
// reads counts, and the word form is ahead from Z = 6 on (Z = 8, 7 circulants,
// 6.4 million checks: 37 and 62 us), not below (Z = 4, 3 circulants, 3.2
// million: 28.7 and 20.6).
bool syndrome_by_words(const qc::Table &T, int n_frames) {
    int g = 1;
    while (g < 32 && T.Z % (2 * g) == 0) g *= 2;
    const int seg = 1 + (32 - g + T.Z - 1) / T.Z;
    return seg * T.max_row_deg <= 18 || (seg <= 6 && (int64_t)n_frames * T.mb * T.Z >= 1 << 20);
}

__global__ void __launch_bounds__(256) bob8_kernel(const float4 *__restrict__ y,
                                                   const uint32_t *__restrict__ bits,
                                                   float4 *__restrict__ out, int64_t n_blocks) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
         b += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t byte = (__ldg(bits + (b >> 2)) >> (8 * (b & 3))) & 0xffu;
        float u[8];
#pragma unroll
        for (int j = 0; j < 8; j++) u[j] = ((byte >> j) & 1u) ? -1.0f : 1.0f;
        const Quat up{u[0], u[1], u[2], u[3]}, uq{u[4], u[5], u[6], u[7]};
        const Quat yr = q4(__ldcs(y + 2 * b)), ys = q4(__ldcs(y + 2 * b + 1));
        Quat lo, hi;
        omul(up, uq, yr, ys, lo, hi);
        out[2 * b] = f4(lo);
        out[2 * b + 1] = f4(hi);
    }
}

__global__ void __launch_bounds__(256) llr8_kernel(const float4 *__restrict__ x,
                                                   const float4 *__restrict__ m,
                                                   float4 *__restrict__ llr, float scale,
                                                   int64_t n_blocks) {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n_blocks;
         b += (int64_t)gridDim.x * blockDim.x) {
        const Quat mp = q4(__ldg(m + 2 * b)), mq = q4(__ldg(m + 2 * b + 1));
        const Quat xp = q4(__ldcs(x + 2 * b)), xq = q4(__ldcs(x + 2 * b + 1));
        // conj of the octonion (xp, xq) is (conj xp, -xq)
        const Quat cp = qconj(xp);
        const Quat cq{-xq.w, -xq.x, -xq.y, -xq.z};
        Quat lo, hi;
        omul(mp, mq, cp, cq, lo, hi);
        llr[2 * b] = make_float4(lo.w * scale, lo.x * scale, lo.y * scale, lo.z * scale);
        llr[2 * b + 1] = make_float4(hi.w * scale, hi.x * scale, hi.y * scale, hi.z * scale);
    }
}

// d in {1, 2, 4}: reals, complex numbers (Cayley-Dickson doubling of the
// reals) and quaternions (Hamilton's rule). Bob: M = U Y. Alice:
// Q = (M conj(X)) * 2 snr / d (sigma_N^2 = d sigma_Z^2 / |X|^2, so |X|^2
// cancels as in the 8-D map).
template <int D>
__device__ __forceinline__ void bob_block(uint32_t neg, const float *yy, float *o) {
    float u[D];
#pragma unroll
    for (int j = 0; j < D; j++) u[j] = ((neg >> j) & 1u) ? -1.0f : 1.0f;
    if constexpr (D == 1) {
        o[0] = u[0] * yy[0];
    } else if constexpr (D == 2) {  // (a + ib)(c + id)
        o[0] = u[0] * yy[0] - u[1] * yy[1];
        o[1] = u[0] * yy[1] + u[1] * yy[0];
    } else {
        const Quat r = qmul(Quat{u[0], u[1], u[2], u[3]}, Quat{yy[0], yy[1], yy[2], yy[3]});
        o[0] = r.w;
        o[1] = r.x;
        o[2] = r.y;
        o[3] = r.z;
    }
}

template <int D>
__device__ __forceinline__ void llr_block(const float *m, const float *x, float scale, float *o) {
    if constexpr (D == 1) {
        o[0] = m[0] * x[0] * scale;
    } else if constexpr (D == 2) {  // M conj(X) = (a + ib)(c - id)
        const float a = m[0], bb = m[1], c = x[0], d = x[1];
        o[0] = (a * c + bb * d) * scale;
        o[1] = (bb * c - a * d) * scale;
    } else {
        const Quat r = qmul(Quat{m[0], m[1], m[2], m[3]}, qconj(Quat{x[0], x[1], x[2], x[3]}));
        o[0] = r.w * scale;
        o[1] = r.x * scale;
        o[2] = r.y * scale;
        o[3] = r.z * scale;
    }
}

// One thread takes V consecutive values: V = 4 (one 16-byte vector of each
// array, and one nibble of the bits) when every float buffer is 16-byte
// aligned, else V = D. The last n % 4 values of the vector form (d = 1, 2)
// are taken block by block by the first threads. A pure stream, bounded by
// HBM and, below a few million values, by the calls themselves: message,
// syndrome and LLRs of 4 frames of n = 10^6, d = 2, went from 45.0 to 30.6 us
// with the word-wise syndrome and these loads.
template <int D, bool VEC>
__global__ void __launch_bounds__(256) bob_d_kernel(const float *__restrict__ y,
                                                    const uint32_t *__restrict__ bits,
                                                    float *__restrict__ out, int64_t n) {
    constexpr int V = VEC ? 4 : D;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nv = n / V;
    for (int64_t b = tid; b < nv; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v0 = b * V;
        const uint32_t neg = __ldg(bits + (v0 >> 5)) >> (v0 & 31);
        float yy[V], o[V];
        if constexpr (VEC) {
            const float4 q = __ldcs(reinterpret_cast<const float4 *>(y) + b);
            yy[0] = q.x, yy[1] = q.y, yy[2] = q.z, yy[3] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < V; j++) yy[j] = __ldg(y + v0 + j);
        }
#pragma unroll
        for (int j = 0; j < V; j += D) bob_block<D>(neg >> j, yy + j, o + j);
        if constexpr (VEC) {
            reinterpret_cast<float4 *>(out)[b] = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int j = 0; j < V; j++) out[v0 + j] = o[j];
        }
    }
    if constexpr (V > D) {
        const int64_t v0 = nv * V + tid * D;
        if (v0 < n) {
            const uint32_t neg = __ldg(bits + (v0 >> 5)) >> (v0 & 31);
            float yy[D], o[D];
#pragma unroll
            for (int j = 0; j < D; j++) yy[j] = __ldg(y + v0 + j);
            bob_block<D>(neg, yy, o);
#pragma unroll
            for (int j = 0; j < D; j++) out[v0 + j] = o[j];
        }
    }
}

template <int D, bool VEC>
__global__ void __launch_bounds__(256) llr_d_kernel(const float *__restrict__ x,
                                                    const float *__restrict__ m,
                                                    float *__restrict__ llr, float scale, int64_t n) {
    constexpr int V = VEC ? 4 : D;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nv = n / V;
    for (int64_t b = tid; b < nv; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v0 = b * V;
        float mm[V], xx[V], o[V];
        if constexpr (VEC) {
            const float4 p = __ldg(reinterpret_cast<const float4 *>(m) + b);
            const float4 q = __ldcs(reinterpret_cast<const float4 *>(x) + b);
            mm[0] = p.x, mm[1] = p.y, mm[2] = p.z, mm[3] = p.w;
            xx[0] = q.x, xx[1] = q.y, xx[2] = q.z, xx[3] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < V; j++) mm[j] = __ldg(m + v0 + j), xx[j] = __ldg(x + v0 + j);
        }
#pragma unroll
        for (int j = 0; j < V; j += D) llr_block<D>(mm + j, xx + j, scale, o + j);
        if constexpr (VEC) {
            reinterpret_cast<float4 *>(llr)[b] = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int j = 0; j < V; j++) llr[v0 + j] = o[j];
        }
    }
    if constexpr (V > D) {
        const int64_t v0 = nv * V + tid * D;
        if (v0 < n) {
            float mm[D], xx[D], o[D];
#pragma unroll
            for (int j = 0; j < D; j++) mm[j] = __ldg(m + v0 + j), xx[j] = __ldg(x + v0 + j);
            llr_block<D>(mm, xx, scale, o);
#pragma unroll
            for (int j = 0; j < D; j++) llr[v0 + j] = o[j];
        }
    }
}

int stream_grid(int64_t n_blocks) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
    int64_t g = (n_blocks + 255) / 256;
    const int64_t cap = (int64_t)sms * 8;  // 8 resident blocks of 256 per SM
    if (g > cap) g = cap;
    return (int)(g > 0 ? g : 1);
}

}  // namespace

extern "C" int qcldpc_syndrome(const qcldpc_code *code, const uint32_t *bits_dev,
                               uint32_t *syn_dev, int n_frames, qcldpc_stream_t stream) {
    using namespace qc;
    if (!code || !bits_dev || !syn_dev || n_frames < 0)
        return fail(QCLDPC_E_INVAL, "syndrome: NULL argument or negative frame count");
    if (!aligned(bits_dev, 4) || !aligned(syn_dev, 4))
        return fail(QCLDPC_E_ALIGN, "syndrome: buffers must be 4-byte aligned");
    if (n_frames > 65535) return fail(QCLDPC_E_INVAL, "syndrome: more than 65535 frames");
    if (n_frames == 0) return QCLDPC_OK;
    if (int st = upload_tables(const_cast<qcldpc_code *>(code))) return st;
    const int64_t words_n = (code->n + 31) / 32, words_m = (code->m + 31) / 32;
    const bool words = syndrome_by_words(code->tab, n_frames);
    const int nt = words ? 128 : 256;
    const int64_t threads = words ? words_m : code->m;
    dim3 grid((unsigned)((threads + nt - 1) / nt), (unsigned)n_frames);
    auto kernel = words ? syndrome_kernel : syndrome_bit_kernel;
    kernel<<<grid, nt, 0, (cudaStream_t)stream>>>(code->tab, bits_dev, syn_dev, words_n, words_m);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "syndrome: launch");
    return QCLDPC_OK;
}

extern "C" int qcldpc_bob_message_8d(const float *y_dev, const uint32_t *bits_dev, int64_t n,
                                     float *m_dev, qcldpc_stream_t stream) {
    using namespace qc;
    if (!y_dev || !bits_dev || !m_dev || n < 0 || n % 8 != 0)
        return fail(QCLDPC_E_INVAL, "bob_message_8d: NULL argument or n not a multiple of 8");
    if (!aligned(y_dev, 16) || !aligned(m_dev, 16) || !aligned(bits_dev, 4))
        return fail(QCLDPC_E_ALIGN, "bob_message_8d: floats must be 16-byte aligned");
    if (n == 0) return QCLDPC_OK;
    const int64_t nb = n / 8;
    bob8_kernel<<<stream_grid(nb), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const float4 *>(y_dev), bits_dev, reinterpret_cast<float4 *>(m_dev), nb);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "bob_message_8d: launch");
    return QCLDPC_OK;
}

extern "C" int qcldpc_llr_8d(const float *x_dev, const float *m_dev, int64_t n, float snr,
                             float *llr_dev, qcldpc_stream_t stream) {
    using namespace qc;
    if (!x_dev || !m_dev || !llr_dev || n < 0 || n % 8 != 0 || !(snr > 0.0f))
        return fail(QCLDPC_E_INVAL, "llr_8d: NULL argument, n not a multiple of 8, or snr <= 0");
    if (!aligned(x_dev, 16) || !aligned(m_dev, 16) || !aligned(llr_dev, 16))
        return fail(QCLDPC_E_ALIGN, "llr_8d: buffers must be 16-byte aligned");
    if (n == 0) return QCLDPC_OK;
    const int64_t nb = n / 8;
    llr8_kernel<<<stream_grid(nb), 256, 0, (cudaStream_t)stream>>>(
        reinterpret_cast<const float4 *>(x_dev), reinterpret_cast<const float4 *>(m_dev),
        reinterpret_cast<float4 *>(llr_dev), snr * 0.25f, nb);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "llr_8d: launch");
    return QCLDPC_OK;
}

extern "C" int qcldpc_bob_message(int d, const float *y_dev, const uint32_t *bits_dev, int64_t n,
                                  float *m_dev, qcldpc_stream_t stream) {
    using namespace qc;
    if (d == 8) return qcldpc_bob_message_8d(y_dev, bits_dev, n, m_dev, stream);
    if ((d != 1 && d != 2 && d != 4) || !y_dev || !bits_dev || !m_dev || n < 0 || n % d != 0)
        return fail(QCLDPC_E_INVAL, "bob_message: d must be 1, 2, 4 or 8 and n a multiple of d");
    if (!aligned(y_dev, 4) || !aligned(m_dev, 4) || !aligned(bits_dev, 4))
        return fail(QCLDPC_E_ALIGN, "bob_message: buffers must be 4-byte aligned");
    if (n == 0) return QCLDPC_OK;
    const bool vec = aligned(y_dev, 16) && aligned(m_dev, 16);
    const int grid = stream_grid(vec ? (n + 3) / 4 : n / d);
    void (*kernel)(const float *, const uint32_t *, float *, int64_t) =
        d == 1 ? (vec ? bob_d_kernel<1, true> : bob_d_kernel<1, false>)
        : d == 2 ? (vec ? bob_d_kernel<2, true> : bob_d_kernel<2, false>) : (vec ? bob_d_kernel<4, true> : bob_d_kernel<4, false>);
    kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(y_dev, bits_dev, m_dev, n);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "bob_message: launch");
    return QCLDPC_OK;
}

extern "C" int qcldpc_llr(int d, const float *x_dev, const float *m_dev, int64_t n, float snr,
                          float *llr_dev, qcldpc_stream_t stream) {
    using namespace qc;
    if (d == 8) return qcldpc_llr_8d(x_dev, m_dev, n, snr, llr_dev, stream);
    if ((d != 1 && d != 2 && d != 4) || !x_dev || !m_dev || !llr_dev || n < 0 || n % d != 0 ||
        !(snr > 0.0f))
        return fail(QCLDPC_E_INVAL, "llr: d must be 1, 2, 4 or 8, n a multiple of d, snr > 0");
    if (!aligned(x_dev, 4) || !aligned(m_dev, 4) || !aligned(llr_dev, 4))
        return fail(QCLDPC_E_ALIGN, "llr: buffers must be 4-byte aligned");
    if (n == 0) return QCLDPC_OK;
    const float scale = 2.0f * snr / (float)d;
    const bool vec = aligned(x_dev, 16) && aligned(m_dev, 16) && aligned(llr_dev, 16);
    const int grid = stream_grid(vec ? (n + 3) / 4 : n / d);
    void (*kernel)(const float *, const float *, float *, float, int64_t) =
        d == 1 ? (vec ? llr_d_kernel<1, true> : llr_d_kernel<1, false>)
        : d == 2 ? (vec ? llr_d_kernel<2, true> : llr_d_kernel<2, false>) : (vec ? llr_d_kernel<4, true> : llr_d_kernel<4, false>);
    kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(x_dev, m_dev, llr_dev, scale, n);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "llr: launch");
    return QCLDPC_OK;
}
