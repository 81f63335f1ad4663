// FP32 SIMT path of the potential: forward message passing and the force
// adjoint.
//
// The filter w_ij = fc(d) phi(d) and its derivative dw/dd depend on the pair's
// distance only: they are the same for (i, j) and (j, i) and do not depend on
// the features. So an evaluation computes both once per unordered pair and
// layer (k_pair_filter, register-blocked GEMMs over tiles of 128 pairs), and
// the passes over the directed pairs are gathers over each atom's own row:
//   forward   m_i = sum_j w_ij * u_j
//   backward  ubar_i = sum_j w_ij * mbar_j,  F_i = sum_j dE/dd_ij rhat_ij
// around one pass over the unordered pairs per layer,
//   dE/dd_ij = g_ij . dw/dd_ij,  g_ij = mbar_i * u_j + mbar_j * u_i (symmetric).
// One warp per atom, the row's pairs in a fixed order, no atomics on results:
// deterministic and independent of the launch shape.
//
// At layer 0, u_j is one row per species, and where that pays (kMinFactorAtoms)
// the second product of the filter is taken out of the sums: rows fc SiLU(a)
// are summed per atom and neighbour species, and multiplied by W2 once each
// (k_gather_species; the adjoint alike in k_pair_dedd).
// 12,288-atom water, when it came: forces with virial 748 -> 692 us, 3 fs step
// 1.00 -> 0.93 ms (701 us and 0.95 ms now).
//
// Against recomputing the filter per directed pair in each pass (20,480 and
// 10,240 flop per directed pair and layer), this is 20,480 flop per unordered
// pair and layer in all, and w, dw/dd travel through memory (512 bytes per
// unordered pair and layer at F = 64, written once, w read four times and
// dw/dd once). Big model, 12,288-atom water, one evaluation: 3.48 -> 0.57 ms
// (edge passes 3.36 -> 0.43 ms); 192 atoms: 0.61 -> 0.158 ms.
#include <cuda_bf16.h>

#include <algorithm>

#include "f32x2.cuh"
#include "internal.cuh"

namespace dmts {

namespace {

// Bessel functions e_k(d) = pref sin(k pi d / rc) / d, k < K <= KP (zero from
// K on), their derivatives, the cosine cutoff and its derivative.
template <int KP>
__device__ __forceinline__ void basis_pair(float d, int K, float pi_over_rc, float pref, float* e, float* de,
                                           float& fc, float& dfc) {
    float s1, c1;
    sincospif(d * (pi_over_rc * 0.31830988618379067f), &s1, &c1);
    float inv_d = 1.0f / d;
    float sk = s1, skm1 = 0.f, ck = c1, ckm1 = 1.f;
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        float kw = (float)(k + 1) * pi_over_rc;
        e[k] = k < K ? pref * sk * inv_d : 0.f;
        de[k] = k < K ? pref * (kw * ck - sk * inv_d) * inv_d : 0.f;
        float sn = 2.f * c1 * sk - skm1;
        float cn = 2.f * c1 * ck - ckm1;
        skm1 = sk; sk = sn;
        ckm1 = ck; ck = cn;
    }
    fc = 0.5f * (c1 + 1.0f);
    dfc = -0.5f * pi_over_rc * s1;
}

// fc'(d), as basis_pair has it
__device__ __forceinline__ float cutoff_deriv(float d, float pi_over_rc) {
    return -0.5f * pi_over_rc * sinpif(d * (pi_over_rc * 0.31830988618379067f));
}

// ------------------------------------------------------------ embedding
// h^0 = A[Z_i] and u^0 = h^0 W_in^0 of every atom and, behind them, the same
// of each species, to h_spec and u_spec.
template <int F>
__global__ void k_embed(PotArgs a, float* __restrict__ h_spec, float* __restrict__ u_spec) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    int i = t / F, f = t % F;
    if (i >= a.n_atoms + a.n_species) return;
    const bool atom = i < a.n_atoms;
    int z = atom ? a.species[i] : i - a.n_atoms;
    const float* A = a.P + a.off.A + z * F;
    const float* W = a.P + a.off.W_in[0];
    float acc = 0.f;
    for (int k = 0; k < F; ++k) acc += __ldg(A + k) * __ldg(W + k * F + f);
    if (!atom) {
        h_spec[z * F + f] = __ldg(A + f);
        u_spec[z * F + f] = acc;
        return;
    }
    a.h[(size_t)i * F + f] = __ldg(A + f);
    a.u_next[(size_t)i * F + f] = acc;
    if (a.um_u_out)
        *reinterpret_cast<__nv_bfloat16*>(a.um_u_out + (size_t)i * F * 4 + (f >> 4) * 64 + (f & 15) * 2) =
            __float2bfloat16_rn(acc);
}

// ------------------------------------------------------------ unordered pairs
// The unordered pairs of the list, one entry (i, j), j > i, each, and for
// every directed pair e the number pid[e] of its entry. A row's columns
// ascend, so its pairs with j > i are a suffix. A block takes a range of
// entries for its 8 atoms, one per warp, with one atomic (the order of the
// ranges varies from run to run and no result depends on it); the entry's
// number goes to its own directed pair and, found by bisection in row j, to the
// reverse one.
constexpr int kIdxWarps = 8;

__global__ void __launch_bounds__(kIdxWarps * 32) k_pair_index(PotArgs a, PairFilter pf) {
    __shared__ int w_sum[kIdxWarps];
    __shared__ int blk;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kIdxWarps + w;
    int total = 0;                                       // pairs with j > i, and the end of the row
    long long end = 0;
    if (i < a.n_atoms) {
        const long long beg = min((long long)a.row_ptr[i], a.e_cap);
        end = min((long long)a.row_ptr[i + 1], a.e_cap);
        for (long long e = beg + lane; e < end; e += 32) total += a.col[e] > i ? 1 : 0;
    }
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0) w_sum[w] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
        int sum = 0;
        for (int k = 0; k < kIdxWarps; ++k) sum += w_sum[k];
        blk = sum ? atomicAdd(pf.count, sum) : 0;
    }
    __syncthreads();
    int base = blk;
    for (int k = 0; k < w; ++k) base += w_sum[k];
    for (int t = lane; t < total; t += 32) {
        const int e = (int)end - total + t;
        const int j = DMTS_IDX(a.col[e], a.n_atoms, a.check), p = base + t;
        if (p >= pf.cap) continue;                       // a truncated (overflowed) list: the call is redone
        pf.pairs[p] = make_int2(i, j);
        pf.pid[e] = p;
        int lo = (int)min((long long)a.row_ptr[j], a.e_cap);
        const int hi = (int)min((long long)a.row_ptr[j + 1], a.e_cap);
        int n = hi - lo;
        while (n > 0) {                                  // first column of row j that is >= i
            const int h = n >> 1;
            if (a.col[lo + h] < i) { lo += h + 1; n -= h + 1; }
            else n = h;
        }
        if (lo < hi && a.col[lo] == i) pf.pid[lo] = p;
    }
}

// ------------------------------------------------------------ filter of every pair
// w = fc phi and dw/dd = fc' phi + fc (SiLU'(a) (e' W1)) W2, with
// a = e W1 + b1 and phi = SiLU(a) W2 + b2, for tiles of 128 pairs.
//
// Bound by FP32 FMA issue: 2 (2 KP F + 2 F F) flop per pair and layer against
// 512 bytes written (F = 64): 639,638 directed pairs, two layers, the first one
// without its second product, 7.9 GFLOP in 215 us (cold, ncu: FMA pipe 57 %, issue
// 52 %, 279 MB written). Each thread owns 8 pairs x 4 features of both
// products that share a weight matrix (64 accumulators), as packed f32x2
// operations over two pairs: one FFMA2 for two FMAs leaves issue slots for the
// operand loads (five 16-byte shared loads per 64 FMAs). The hidden layer is
// kept [feature][pair] with a row stride of 132 floats: the four hidden
// features of a thread are F / 4 apart, so that the eight lanes of a 16-byte
// store phase fall into distinct banks, while its four output features are
// adjacent, so that a row of w is written as whole 128-byte lines.
// SiLU takes the ordinary division, as the per-atom kernels do (an approximate
// one: forces with virial of 12,288 atoms 701 -> 675 us, but two ulp instead of
// half a one, and zero for activations from -88.7 to -87.4).
template <int F, int KP>
struct FiltTile {
    static constexpr int FG = F / 4;                     // feature groups of 4
    static constexpr int TP = 128;                       // pairs per tile
    static constexpr int NT = TP / 8 * FG;               // threads: 8 pairs x 4 features each
    static constexpr int TS = TP + 4;
    float W1[KP * F];                                    // [k][4 fg + c] = W1[k][fg + FG c]
    float b1[F];                                         // permuted alike
    float W2[F * F];
    float b2[F];
    float B[KP * TS], D[KP * TS];                        // basis and derivative, [k][pair]
    float S[F * TS], Q[F * TS];                          // SiLU(a), SiLU'(a) (e' W1), [feature][pair]
    float fc[2][TP], dfc[2][TP];                         // two tiles in turn
};

// acc[p][c] += A[k][p0 + 2p, + 1] W[k][f0 + c] for two operands that share W
template <int KIN, int TS, int WS, int UNROLL>
__device__ __forceinline__ void gemm_pair(const float* A0, const float* A1, const float* W, f2::f32x2 (&x)[4][4],
                                          f2::f32x2 (&y)[4][4]) {
#pragma unroll UNROLL
    for (int k = 0; k < KIN; ++k) {
        const ulonglong2 s01 = *reinterpret_cast<const ulonglong2*>(A0 + k * TS);
        const ulonglong2 s23 = *reinterpret_cast<const ulonglong2*>(A0 + k * TS + 4);
        const ulonglong2 q01 = *reinterpret_cast<const ulonglong2*>(A1 + k * TS);
        const ulonglong2 q23 = *reinterpret_cast<const ulonglong2*>(A1 + k * TS + 4);
        const float4 w4 = *reinterpret_cast<const float4*>(W + k * WS);
        const f2::f32x2 s[4] = {s01.x, s01.y, s23.x, s23.y}, q[4] = {q01.x, q01.y, q23.x, q23.y};
        const f2::f32x2 w[4] = {f2::splat(w4.x), f2::splat(w4.y), f2::splat(w4.z), f2::splat(w4.w)};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                x[p][c] = f2::fma(s[p], w[c], x[p][c]);
                y[p][c] = f2::fma(q[p], w[c], y[p][c]);
            }
    }
}

// With HID (layer 0 by species) layer 0 stops before the second product:
// the rows are fc SiLU(a) and its derivative q = fc' SiLU(a) + fc SiLU'(a) (e' W1),
// and fc goes to pf.se until the backward pass overwrites it. There each
// thread's four hidden features are adjacent (W1 and b1 unpermuted), as the
// rows are written from the first product's registers.
template <int F, int KP, bool HID>
__global__ void __launch_bounds__(FiltTile<F, KP>::NT, F == 64 ? 2 : 4) k_pair_filter(PotArgs a, PairFilter pf, int K,
                                                                                      int l0, int l1, int a0, int a1) {
    using T = FiltTile<F, KP>;
    constexpr int TP = T::TP, TS = T::TS, FG = T::FG, NT = T::NT;
    extern __shared__ float4 smem4[];
    T& S = *reinterpret_cast<T*>(smem4);
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int fg = (F == 64 ? (wp & 1) * 8 : 0) + (lane & 7);
    const int p0 = 8 * ((F == 64 ? wp >> 1 : wp) * 4 + (lane >> 3));
    const int f0 = 4 * fg;
    // the pairs: the unordered ones, or (chunked) the directed pairs of atoms a0 .. a1
    const bool half = pf.chunk_atoms == 0;
    const long long e_beg = half ? 0 : min((long long)a.row_ptr[a0], a.e_cap);
    const long long n_pairs = half ? min((long long)*pf.count, pf.cap)
                                   : min(min((long long)a.row_ptr[a1], a.e_cap) - e_beg, pf.cap);
    const long long tiles = (n_pairs + TP - 1) / TP, units = tiles * (l1 - l0);
    int cur = -1, buf = 0;
    // The thread's pair of the next tile (pair tid mod TP): atom indices loaded
    // at the start of a tile, positions before its second product.
    const int lp = tid & (TP - 1);
    int ni = -1, nj = 0;
    uint4 qi = make_uint4(0, 0, 0, 0), qj = qi;
    auto load_pair = [&](long long u) {
        const long long p = u < units ? u % tiles * TP + lp : n_pairs;
        ni = -1;
        if (p >= n_pairs) return;
        if (half) {
            const int2 ij = pf.pairs[p];
            ni = DMTS_IDX(ij.x, a.n_atoms, a.check);
            nj = DMTS_IDX(ij.y, a.n_atoms, a.check);
        } else {
            ni = DMTS_IDX(a.recv[e_beg + p], a.n_atoms, a.check);
            nj = DMTS_IDX(a.col[e_beg + p], a.n_atoms, a.check);
        }
    };
    auto load_pos = [&]() {
        if (ni < 0) return;
        qi = a.q[ni];
        qj = a.q[nj];
    };
    load_pair(blockIdx.x);
    load_pos();
    for (long long unit = blockIdx.x; unit < units; unit += gridDim.x, buf ^= 1) {
        const int l = l0 + (int)(unit / tiles);
        const long long t0 = (unit - (l - l0) * tiles) * TP;
        const bool hid = HID && l == 0;
        if (l != cur) {                                  // this layer's weights
            __syncthreads();
            for (int t = tid; t < KP * F; t += NT) {
                const int k = t / F, r = t % F, f = hid ? r : (r >> 2) + FG * (r & 3);
                S.W1[t] = k < K ? __ldg(a.P + a.off.W1[l] + k * F + f) : 0.f;
            }
            for (int t = tid; t < F; t += NT) S.b1[t] = __ldg(a.P + a.off.b1[l] + (hid ? t : (t >> 2) + FG * (t & 3)));
            if (!hid) {
                for (int t = tid; t < F * F; t += NT) S.W2[t] = __ldg(a.P + a.off.W2[l] + t);
                for (int t = tid; t < F; t += NT) S.b2[t] = __ldg(a.P + a.off.b2[l] + t);
            }
            cur = l;
        }
        {
            float eb[KP], db[KP], fc = 0.f, dfc = 0.f;
            if (ni >= 0) {
                const float3 r = edge_vec(qi, qj, a.frame[qi.w].qscale);
                const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
                basis_pair<KP>(d, K, a.pi_over_rc, a.bessel_pref, eb, db, fc, dfc);
            } else {
#pragma unroll
                for (int k = 0; k < KP; ++k) eb[k] = db[k] = 0.f;
            }
            // with two threads per pair (F = 64) one writes the basis, the other its derivative
            if (NT == TP || tid < TP) {
#pragma unroll
                for (int k = 0; k < KP; ++k) S.B[k * TS + lp] = eb[k];
                S.fc[buf][lp] = fc;
            }
            if (NT == TP || tid >= TP) {
#pragma unroll
                for (int k = 0; k < KP; ++k) S.D[k * TS + lp] = db[k];
                S.dfc[buf][lp] = dfc;
            }
            if (hid && tid < TP && t0 + lp < n_pairs) pf.se[t0 + lp] = fc;
        }
        load_pair(unit + gridDim.x);
        __syncthreads();
        f2::f32x2 x[4][4], y[4][4];
        {
            const float4 b = *reinterpret_cast<const float4*>(S.b1 + f0);
            const float bc[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    x[p][c] = f2::splat(bc[c]);
                    y[p][c] = 0ull;
                }
            gemm_pair<KP, TS, F, KP>(S.B + p0, S.D + p0, S.W1 + f0, x, y);
            if (hid) {
                load_pos();
                const size_t row0 = (size_t)(half ? l : 0) * 2 * pf.cap;
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const long long r = t0 + p0 + p;
                    if (r >= n_pairs) break;
                    const float fc = S.fc[buf][p0 + p], dfc = S.dfc[buf][p0 + p];
                    float s[4], q[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float v = (p & 1) ? f2::hi(x[p >> 1][c]) : f2::lo(x[p >> 1][c]);
                        const float t = (p & 1) ? f2::hi(y[p >> 1][c]) : f2::lo(y[p >> 1][c]);
                        float sg;
                        s[c] = silu_f(v, sg);
                        q[c] = dfc * s[c] + fc * (sg * (1.f + v * (1.f - sg)) * t);
                    }
                    float* w = pf.w + (row0 + r) * F + f0;
                    *reinterpret_cast<float4*>(w) = make_float4(fc * s[0], fc * s[1], fc * s[2], fc * s[3]);
                    __stcs(reinterpret_cast<float4*>(w + (size_t)pf.cap * F), make_float4(q[0], q[1], q[2], q[3]));
                }
                __syncthreads();                         // B and D are rewritten by the next tile
                continue;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {                // hidden feature fg + FG c of the thread's 8 pairs
                float s[8], q[8];
#pragma unroll
                for (int p = 0; p < 8; ++p) {
                    const float v = (p & 1) ? f2::hi(x[p >> 1][c]) : f2::lo(x[p >> 1][c]);
                    const float t = (p & 1) ? f2::hi(y[p >> 1][c]) : f2::lo(y[p >> 1][c]);
                    float sg;
                    s[p] = silu_f(v, sg);
                    q[p] = sg * (1.f + v * (1.f - sg)) * t;
                }
                float* ds = S.S + (fg + FG * c) * TS + p0;
                float* dq = S.Q + (fg + FG * c) * TS + p0;
                *reinterpret_cast<float4*>(ds) = make_float4(s[0], s[1], s[2], s[3]);
                *reinterpret_cast<float4*>(ds + 4) = make_float4(s[4], s[5], s[6], s[7]);
                *reinterpret_cast<float4*>(dq) = make_float4(q[0], q[1], q[2], q[3]);
                *reinterpret_cast<float4*>(dq + 4) = make_float4(q[4], q[5], q[6], q[7]);
            }
        }
        __syncthreads();
        load_pos();
        {
            const float4 b = *reinterpret_cast<const float4*>(S.b2 + f0);
            const float bc[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    x[p][c] = f2::splat(bc[c]);
                    y[p][c] = 0ull;
                }
            gemm_pair<F, TS, F, 4>(S.S + p0, S.Q + p0, S.W2 + f0, x, y);
            const size_t row0 = (size_t)(half ? l : 0) * 2 * pf.cap;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const long long r = t0 + p0 + p;
                if (r >= n_pairs) break;
                const float fc = S.fc[buf][p0 + p], dfc = S.dfc[buf][p0 + p];
                float ph[4], ps[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    ph[c] = (p & 1) ? f2::hi(x[p >> 1][c]) : f2::lo(x[p >> 1][c]);
                    ps[c] = (p & 1) ? f2::hi(y[p >> 1][c]) : f2::lo(y[p >> 1][c]);
                }
                float* w = pf.w + (row0 + r) * F + f0;
                *reinterpret_cast<float4*>(w) = make_float4(fc * ph[0], fc * ph[1], fc * ph[2], fc * ph[3]);
                __stcs(reinterpret_cast<float4*>(w + (size_t)pf.cap * F),
                       make_float4(dfc * ph[0] + fc * ps[0], dfc * ph[1] + fc * ps[1], dfc * ph[2] + fc * ps[2],
                                   dfc * ph[3] + fc * ps[3]));
            }
        }
        // the next tile's basis, SiLU and fc tiles: B and D were last read before the
        // second barrier, fc alternates, S and Q are written after the next first barrier
    }
}

// ------------------------------------------------------------ gathers
// One warp per atom; a row of F floats is read by F / 4 lanes, 16 bytes each,
// so one warp instruction reads 2 (F = 64) or 4 (F = 32) whole rows: w_ij and
// v_j, 512 bytes per directed pair at F = 64 (639,638 pairs: 39 us, 8.4 TB/s
// through L2). Bound by the latency of those rows: the next 32 pairs' indices
// are loaded, and their w rows (mostly in DRAM by then) sent for, while the
// present ones are summed.
// At layer 0, u_j = A[Z_j] W_in depends on the species only: its row is read
// at the first atom of that species (first_of), a few rows that stay in L1.
// Blocks that run on one SM one after another take adjacent atoms
// (gather_range), whose neighbours' rows they share in L1.

// The atoms of this block: block b of a grid of kSmCount x per blocks takes
// range (b mod kSmCount) per + b / kSmCount, so that blocks kSmCount apart,
// which the hardware mostly gives to the same SM, are neighbours.
__device__ __forceinline__ void gather_range(int n_per_cta, int a0, int a1, int& first, int& last) {
    const int per = gridDim.x / kSmCount;
    const int r = per > 0 ? (int)(blockIdx.x % kSmCount) * per + (int)(blockIdx.x / kSmCount) : (int)blockIdx.x;
    first = min(a1, a0 + r * n_per_cta);
    last = min(a1, first + n_per_cta);
}

// Filter row of directed pair e, or -1 if there is none: after an overflow
// (the call will be redone) a pair may lack its entry, and a stale number is
// recognised by the pair stored there.
__device__ __forceinline__ int filter_row(const PotArgs& a, const PairFilter& pf, long long e, long long e_beg, int i,
                                          int j, bool overflow) {
    if (pf.chunk_atoms) return e - e_beg < pf.cap ? (int)(e - e_beg) : -1;
    const int p = pf.pid[e];
    if (!overflow) return DMTS_IDX(p, pf.cap, a.check);
    if (p < 0 || p >= pf.cap) return -1;
    const int2 ij = pf.pairs[p];
    return ij.x == min(i, j) && ij.y == max(i, j) ? p : -1;
}

__device__ __forceinline__ float4 ld4(const float* p, int row, int F) {
    return __ldg(reinterpret_cast<const float4*>(p + (size_t)(unsigned int)row * F));
}

// Starts moving row p of an [.][F] array into L2.
template <int F>
__device__ __forceinline__ void prefetch_row(const float* base, int p) {
#pragma unroll
    for (int k = 0; k < F; k += 32) asm volatile("prefetch.global.L2 [%0];" :: "l"(base + (size_t)(unsigned int)p * F + k));
}

// out_i = sum_j w_ij * v_j over atom i's row: the messages (v = u) or, in the
// backward pass above layer 0, ubar (v = mbar). FWD: the forward pass, which
// at layer 0 also sums the pair repulsion, 1/2 phi(d_ij) per directed pair.
template <int F, bool FWD>
__global__ void __launch_bounds__(kThreads) k_gather(PotArgs a, PairFilter pf, const float* __restrict__ v, int a0,
                                                     int a1) {
    constexpr int LPR = F / 4, RPI = 32 / LPR;
    const int lane = threadIdx.x & 31, sub = lane / LPR, ch = lane % LPR;
    const bool overflow = a.check[kFlagOverflow] != 0;
    const bool l0 = FWD && a.layer == 0, rep_on = l0 && a.energy;
    const float* W0 = pf.w + (size_t)(pf.chunk_atoms ? 0 : a.layer) * 2 * pf.cap * F;
    const float* W = W0 + 4 * ch;
    const float* V = v + 4 * ch;
    const long long e_beg = min((long long)a.row_ptr[a0], a.e_cap);
    int first, last;
    gather_range(a.atoms_per_cta, a0, a1, first, last);
    for (int i = first + (threadIdx.x >> 5); i < last; i += kThreads / 32) {
        const long long beg = min((long long)a.row_ptr[i], a.e_cap), end = min((long long)a.row_ptr[i + 1], a.e_cap);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float rep = 0.f;
        const uint4 qi = a.q[i];
        const float qscale = a.frame[qi.w].qscale;
        int nj = 0, nv = 0, np = -1;                     // the lane's pair of the next chunk
        auto load = [&](long long e) {
            np = -1;
            if (e < end) {
                nj = DMTS_IDX(a.col[e], a.n_atoms, a.check);
                np = filter_row(a, pf, e, e_beg, i, nj, overflow);
                if (np >= 0) prefetch_row<F>(W0, np);
                nv = l0 ? a.first_of[nj] : nj;
            }
        };
        load(beg + lane);
        for (long long b = beg; b < end; b += 32) {
            const int p = np, jv = nv;                   // rows of w (-1: no pair) and v
            uint4 qj = qi;                               // (used after the rows' loads have been issued)
            if (rep_on && b + lane < end) qj = a.q[nj];
            load(b + 32 + lane);
            const int n = (int)min(32ll, end - b);
#pragma unroll 8
            for (int k = 0; k < n; k += RPI) {
                const int pk = __shfl_sync(0xffffffffu, p, k + sub);
                const int jk = __shfl_sync(0xffffffffu, jv, k + sub);
                const float4 w = ld4(W, max(pk, 0), F), x = ld4(V, jk, F);
                if (pk >= 0) {
                    acc.x += w.x * x.x;
                    acc.y += w.y * x.y;
                    acc.z += w.z * x.z;
                    acc.w += w.w * x.w;
                }
            }
            if (rep_on && b + lane < end) {
                const float3 r = edge_vec(qi, qj, qscale);
                const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
                rep += 0.5f * rep_phi(d, a.rep_a, a.rep_inv_rho, a.rep_rc, a.rep_pi_over_rc, nullptr);
            }
        }
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
            acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (sub == 0) *reinterpret_cast<float4*>(a.msg_out + (size_t)i * F + 4 * ch) = acc;
        if (rep_on) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rep += __shfl_xor_sync(0xffffffffu, rep, o);
            if (lane == 0) a.erep[i] = rep;
        }
    }
}

// Layer 0 by species: u_j depends on the neighbour's species only, so
// m_i = sum_s u_s * (T_is W2 + t_is b2) with T_is = sum_{j of species s} fc SiLU(a_ij)
// and t_is = sum_{j of species s} fc_ij, and the filter's second product runs
// once per atom and species (in the per-atom kernel) instead of once per
// pair: 2 F^2 flop of 9 to 26 unordered pairs against 2 S F^2. One warp per
// atom, as k_gather, without the rows of v; the sums take selected values, as a
// branch on the species splits the rows of one instruction (12,288 atoms,
// forces with virial 683 -> 676 us).
template <int F, int NS>
__global__ void __launch_bounds__(kThreads) k_gather_species(PotArgs a, PairFilter pf, int a0, int a1) {
    constexpr int LPR = F / 4, RPI = 32 / LPR;
    const int lane = threadIdx.x & 31, sub = lane / LPR, ch = lane % LPR;
    const bool overflow = a.check[kFlagOverflow] != 0;
    const bool rep_on = a.energy != 0;
    const float* W = pf.w + 4 * ch;
    const long long e_beg = min((long long)a.row_ptr[a0], a.e_cap);
    int first, last;
    gather_range(a.atoms_per_cta, a0, a1, first, last);
    for (int i = first + (threadIdx.x >> 5); i < last; i += kThreads / 32) {
        const long long beg = min((long long)a.row_ptr[i], a.e_cap), end = min((long long)a.row_ptr[i + 1], a.e_cap);
        float4 acc[NS];
        float fsum[NS], rep = 0.f;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            acc[s] = make_float4(0.f, 0.f, 0.f, 0.f);
            fsum[s] = 0.f;
        }
        const uint4 qi = a.q[i];
        const float qscale = a.frame[qi.w].qscale;
        int nj = 0, nz = -1, np = -1;                    // the lane's pair of the next chunk
        auto load = [&](long long e) {
            np = nz = -1;
            if (e < end) {
                nj = DMTS_IDX(a.col[e], a.n_atoms, a.check);
                np = filter_row(a, pf, e, e_beg, i, nj, overflow);
                if (np >= 0) {
                    prefetch_row<F>(pf.w, np);
                    nz = a.species[nj];
                }
            }
        };
        load(beg + lane);
        for (long long b = beg; b < end; b += 32) {
            const int p = np, z = nz;                    // row and species of j (-1: no pair)
            float fc = 0.f;                              // (fc and qj: used after the rows' loads have been issued)
            uint4 qj = qi;
            if (p >= 0) fc = pf.se[p];
            if (rep_on && b + lane < end) qj = a.q[nj];
            load(b + 32 + lane);
            const int n = (int)min(32ll, end - b);
#pragma unroll 8
            for (int k = 0; k < n; k += RPI) {
                const int pk = __shfl_sync(0xffffffffu, p, k + sub);
                const int zk = __shfl_sync(0xffffffffu, z, k + sub);
                const float4 w = ld4(W, max(pk, 0), F);
#pragma unroll
                for (int s = 0; s < NS; ++s) {           // (selected values: the rows of an instruction do not diverge)
                    acc[s].x += zk == s ? w.x : 0.f;
                    acc[s].y += zk == s ? w.y : 0.f;
                    acc[s].z += zk == s ? w.z : 0.f;
                    acc[s].w += zk == s ? w.w : 0.f;
                }
            }
#pragma unroll
            for (int s = 0; s < NS; ++s) fsum[s] += z == s ? fc : 0.f;
            if (rep_on && b + lane < end) {
                const float3 r = edge_vec(qi, qj, qscale);
                const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
                rep += 0.5f * rep_phi(d, a.rep_a, a.rep_inv_rho, a.rep_rc, a.rep_pi_over_rc, nullptr);
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (s >= a.n_species) break;
#pragma unroll
            for (int o = LPR; o < 32; o <<= 1) {
                acc[s].x += __shfl_xor_sync(0xffffffffu, acc[s].x, o);
                acc[s].y += __shfl_xor_sync(0xffffffffu, acc[s].y, o);
                acc[s].z += __shfl_xor_sync(0xffffffffu, acc[s].z, o);
                acc[s].w += __shfl_xor_sync(0xffffffffu, acc[s].w, o);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) fsum[s] += __shfl_xor_sync(0xffffffffu, fsum[s], o);
            const size_t row = (size_t)i * a.n_species + s;
            if (sub == 0) *reinterpret_cast<float4*>(a.spec_row + row * F + 4 * ch) = acc[s];
            if (lane == 0) a.spec_sum[row] = fsum[s];
        }
        if (rep_on) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rep += __shfl_xor_sync(0xffffffffu, rep, o);
            if (lane == 0) a.erep[i] = rep;
        }
    }
}

// s[k] of the LPR lanes of a row, summed over those lanes by halving exchanges
// (LPR - 1 shuffles): lane ch is left with the sum of s[ch] in s[0].
template <int LPR>
__device__ __forceinline__ void halving_sum(float (&s)[LPR], int ch) {
#pragma unroll
    for (int m = LPR / 2; m > 0; m >>= 1) {
        const bool up = (ch & m) != 0;
#pragma unroll
        for (int k = 0; k < m; ++k) {
            const float give = up ? s[k] : s[k + m], keep = up ? s[k + m] : s[k];
            s[k] = keep + __shfl_xor_sync(0xffffffffu, give, m);
        }
    }
}

// One pair's share of atom i's force, dE/dd rhat, and (NV = 9) of its virial,
// W_ab = -1/2 sum_directed dE/dd d rhat_a rhat_b (xx yy zz xy xz yz).
template <int NV>
__device__ __forceinline__ void add_force(float (&fv)[NV], float se, float rx, float ry, float rz, float d) {
    fv[0] += se * rx;
    fv[1] += se * ry;
    fv[2] += se * rz;
    if constexpr (NV == 9) {
        const float hv = -0.5f * se * d;
        fv[3] += hv * rx * rx; fv[4] += hv * ry * ry; fv[5] += hv * rz * rz;
        fv[6] += hv * rx * ry; fv[7] += hv * rx * rz; fv[8] += hv * ry * rz;
    }
}

template <int NV>
__device__ __forceinline__ void store_force(const PotArgs& a, int i, float (&fv)[NV], int lane, int accumulate) {
#pragma unroll
    for (int c = 0; c < NV; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fv[c] += __shfl_xor_sync(0xffffffffu, fv[c], o);
    if (lane != 0) return;
#pragma unroll
    for (int c = 0; c < NV; ++c) {
        float* f = c < 3 ? a.force + (size_t)c * a.n_atoms + i : a.vir6 + (size_t)i * 6 + c - 3;
        *f = accumulate ? *f + fv[c] : fv[c];
    }
}

// ------------------------------------------------------------ dE/dd of every pair
// se = g . dw/dd, g = mbar_i * u_j + mbar_j * u_i: symmetric in (i, j), so once
// per unordered pair; at layer 0 plus the repulsion's derivative. The layers
// add up in pf.se (add). (In atom rows, both directions of every pair with the
// ubar sum alongside: 100 and 69 us for layers 1 and 0 of the big model on
// 12,288-atom water; so, with k_gather and k_pair_force: 70 and 47.) A warp takes 32 consecutive pairs: their dw/dd rows
// are contiguous, and consecutive pairs mostly share atom i. The products of
// a row of lanes are partial sums in registers, one per row instruction; the
// sum of pair RPI ch + sub ends in lane (sub, ch).
// SPEC (layer 0 by species): se = (Y_i,zj + Y_j,zi) . q + fc' (B_i,zj + B_j,zi) with
// the per-atom kernel's Y_is = W2 (mbar_i * u_s) and B_is = b2 . (mbar_i * u_s): three
// rows per pair instead of five.
template <int F, bool L0, bool SPEC>
__global__ void __launch_bounds__(kThreads, F == 64 ? 3 : 4) k_pair_dedd(PotArgs a, PairFilter pf, int a0, int a1, int add) {
    constexpr int LPR = F / 4, RPI = 32 / LPR;
    const int lane = threadIdx.x & 31, sub = lane / LPR, ch = lane % LPR;
    const bool half = pf.chunk_atoms == 0;
    const long long e_beg = half ? 0 : min((long long)a.row_ptr[a0], a.e_cap);
    const long long n_pairs = half ? min((long long)*pf.count, pf.cap)
                                   : min(min((long long)a.row_ptr[a1], a.e_cap) - e_beg, pf.cap);
    const float* DW = pf.w + (size_t)((half ? a.layer : 0) * 2 + 1) * pf.cap * F + 4 * ch;
    const float* U = a.u + 4 * ch;
    const float* MB = a.mbar + 4 * ch;
    const float* Y = a.spec_row + 4 * ch;
    const long long step = (long long)gridDim.x * (kThreads / 32) * 32;
    int ni = 0, nj = 0;
    auto load_pair = [&](long long p) {                  // atoms of pair p (the atoms of the chunk's first pair past the end)
        if (p >= n_pairs) return;
        if (half) {
            const int2 ij = pf.pairs[p];
            ni = DMTS_IDX(ij.x, a.n_atoms, a.check);
            nj = DMTS_IDX(ij.y, a.n_atoms, a.check);
        } else {
            ni = DMTS_IDX(a.recv[e_beg + p], a.n_atoms, a.check);
            nj = DMTS_IDX(a.col[e_beg + p], a.n_atoms, a.check);
        }
    };
    const int own = RPI * ch + sub;                      // this lane's pair of a chunk
    long long p0 = ((long long)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 32;
    load_pair(p0 + own);
    for (; p0 < n_pairs; p0 += step) {
        const int i = ni, j = nj;
        int iu = i, ju = j;
        if (SPEC) {                                       // rows of Y
            iu = i * a.n_species + a.species[j];
            ju = j * a.n_species + a.species[i];
        } else if (L0) {
            iu = a.first_of[i];
            ju = a.first_of[j];
        }
        load_pair(p0 + step + own);
        const int n = (int)min(32ll, n_pairs - p0);
        float s[LPR];
#pragma unroll
        for (int k = 0; k < LPR; ++k) {
            s[k] = 0.f;
            if (RPI * k < n) {                            // warp-uniform
                const int src = sub * LPR + k;
                const int row = min(RPI * k + sub, n - 1);
                if constexpr (SPEC) {
                    const int iy = __shfl_sync(0xffffffffu, iu, src), jy = __shfl_sync(0xffffffffu, ju, src);
                    const float4 q = __ldcs(reinterpret_cast<const float4*>(DW + (p0 + row) * F));
                    const float4 yi = ld4(Y, iy, F), yj = ld4(Y, jy, F);
                    float t = (yi.x + yj.x) * q.x;
                    t += (yi.y + yj.y) * q.y;
                    t += (yi.z + yj.z) * q.z;
                    t += (yi.w + yj.w) * q.w;
                    s[k] = t;
                    continue;
                }
                const int ik = __shfl_sync(0xffffffffu, i, src), jk = __shfl_sync(0xffffffffu, j, src);
                const int iuk = L0 ? __shfl_sync(0xffffffffu, iu, src) : ik;
                const int juk = L0 ? __shfl_sync(0xffffffffu, ju, src) : jk;
                const float4 dw = __ldcs(reinterpret_cast<const float4*>(DW + (p0 + row) * F));
                const float4 ui = ld4(U, iuk, F), uj = ld4(U, juk, F), mi = ld4(MB, ik, F), mj = ld4(MB, jk, F);
                float t = (mi.x * uj.x + mj.x * ui.x) * dw.x;
                t += (mi.y * uj.y + mj.y * ui.y) * dw.y;
                t += (mi.z * uj.z + mj.z * ui.z) * dw.z;
                t += (mi.w * uj.w + mj.w * ui.w) * dw.w;
                s[k] = t;
            }
        }
        halving_sum<LPR>(s, ch);
        if (own < n) {
            float se = s[0];
            if (L0) {
                const uint4 qi = a.q[i];
                const float3 r = edge_vec(qi, a.q[j], a.frame[qi.w].qscale);
                const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
                if (SPEC) se += cutoff_deriv(d, a.pi_over_rc) * (a.spec_sum[iu] + a.spec_sum[ju]);
                float dphi;
                (void)rep_phi(d, a.rep_a, a.rep_inv_rho, a.rep_rc, a.rep_pi_over_rc, &dphi);
                se += dphi;
            }
            float* out = pf.se + p0 + own;
            *out = add ? *out + se : se;
        }
    }
}

// F_i = sum_j dE/dd_ij rhat_ij over atom i's row, and (NV = 9) the per-atom
// virial; one warp per atom, one pair per lane.
template <int NV>
__global__ void __launch_bounds__(kThreads) k_pair_force(PotArgs a, PairFilter pf, int a0, int a1, int accumulate) {
    const int lane = threadIdx.x & 31;
    const bool overflow = a.check[kFlagOverflow] != 0;
    const long long e_beg = min((long long)a.row_ptr[a0], a.e_cap);
    int first, last;
    gather_range(a.atoms_per_cta, a0, a1, first, last);
    for (int i = first + (threadIdx.x >> 5); i < last; i += kThreads / 32) {
        const long long beg = min((long long)a.row_ptr[i], a.e_cap), end = min((long long)a.row_ptr[i + 1], a.e_cap);
        const uint4 qi = a.q[i];
        const float qscale = a.frame[qi.w].qscale;
        float fv[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) fv[c] = 0.f;
        for (long long e = beg + lane; e < end; e += 32) {
            const int j = DMTS_IDX(a.col[e], a.n_atoms, a.check);
            const int p = filter_row(a, pf, e, e_beg, i, j, overflow);
            const float3 r = edge_vec(qi, a.q[j], qscale);
            const float d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
            const float inv = 1.0f / d;
            const float rx = r.x * inv, ry = r.y * inv, rz = r.z * inv;
            const float se = p >= 0 ? pf.se[p] : 0.f;
            add_force<NV>(fv, se, rx, ry, rz, d);
        }
        store_force<NV>(a, i, fv, lane, accumulate);
    }
    // every reader of the pair count has finished: zero for the next index
    if (!pf.chunk_atoms && blockIdx.x == 0 && threadIdx.x == 0) *pf.count = 0;
}

// One-layer models: dE/dd, force and (NV = 9) virial in one pass over each
// atom's row, every pair's dE/dd evaluated in both directions: at F = 32 that
// costs no more than the two passes above (12,288-atom water, small model:
// 18.5 against 18.9 us; 192 atoms: 8 against 14 us).
template <int F, int NV>
__global__ void __launch_bounds__(kThreads, NV == 3 ? 3 : 2) k_row_force(PotArgs a, PairFilter pf, int a0, int a1) {
    constexpr int LPR = F / 4, RPI = 32 / LPR;
    const int lane = threadIdx.x & 31, sub = lane / LPR, ch = lane % LPR;
    const bool overflow = a.check[kFlagOverflow] != 0;
    const float* DW = pf.w + (size_t)pf.cap * F + 4 * ch;
    const float* U = a.u + 4 * ch;
    const float* MB = a.mbar + 4 * ch;
    const long long e_beg = min((long long)a.row_ptr[a0], a.e_cap);
    int first, last;
    gather_range(a.atoms_per_cta, a0, a1, first, last);
    for (int i = first + (threadIdx.x >> 5); i < last; i += kThreads / 32) {
        const long long beg = min((long long)a.row_ptr[i], a.e_cap), end = min((long long)a.row_ptr[i + 1], a.e_cap);
        const uint4 qi = a.q[i];
        const float qscale = a.frame[qi.w].qscale;
        const float4 ui = ld4(U, i, F), mi = ld4(MB, i, F);
        float fv[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) fv[c] = 0.f;
        for (long long b = beg; b < end; b += 32) {
            const long long e = b + RPI * ch + sub;       // this lane's pair of the chunk
            int j = i, ju = i, p = -1;
            float rx = 0.f, ry = 0.f, rz = 0.f, d = 1.f;
            if (e < end) {
                j = DMTS_IDX(a.col[e], a.n_atoms, a.check);
                p = filter_row(a, pf, e, e_beg, i, j, overflow);
                const float3 r = edge_vec(qi, a.q[j], qscale);
                d = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
                const float inv = 1.0f / d;
                rx = r.x * inv; ry = r.y * inv; rz = r.z * inv;
                ju = a.first_of[j];
            }
            const int n = (int)min(32ll, end - b);
            float s[LPR];
#pragma unroll
            for (int k = 0; k < LPR; ++k) {
                s[k] = 0.f;
                if (RPI * k < n) {                        // warp-uniform
                    const int src = sub * LPR + k;
                    const int pk = __shfl_sync(0xffffffffu, p, src), jk = __shfl_sync(0xffffffffu, j, src);
                    const int juk = __shfl_sync(0xffffffffu, ju, src);
                    const float4 dw = ld4(DW, max(pk, 0), F), uj = ld4(U, juk, F), mj = ld4(MB, jk, F);
                    float t = (mi.x * uj.x + mj.x * ui.x) * dw.x;
                    t += (mi.y * uj.y + mj.y * ui.y) * dw.y;
                    t += (mi.z * uj.z + mj.z * ui.z) * dw.z;
                    t += (mi.w * uj.w + mj.w * ui.w) * dw.w;
                    s[k] = pk >= 0 ? t : 0.f;
                }
            }
            halving_sum<LPR>(s, ch);
            if (e < end) {
                float dphi;
                (void)rep_phi(d, a.rep_a, a.rep_inv_rho, a.rep_rc, a.rep_pi_over_rc, &dphi);
                add_force<NV>(fv, s[0] + dphi, rx, ry, rz, d);
            }
        }
        store_force<NV>(a, i, fv, lane, a.accumulate);
    }
    if (!pf.chunk_atoms && blockIdx.x == 0 && threadIdx.x == 0) *pf.count = 0;
}

// ------------------------------------------------------------ launches
// Filters of layers l0 .. l1 - 1 for the unordered pairs, or (chunked) the
// directed pairs of atoms a0 .. a1 - 1. Persistent: two CTAs of 256 threads
// per SM at F = 64, four of 128 at F = 32 (shared memory and registers).
template <int F, int KP, bool HID>
void filter_go(const PotArgs& a, int K, int l0, int l1, int a0, int a1, cudaStream_t s) {
    using T = FiltTile<F, KP>;
    smem_opt_in((const void*)k_pair_filter<F, KP, HID>, (int)sizeof(T));
    const long long tiles = (a.filter.cap + T::TP - 1) / T::TP * (l1 - l0);
    const int grid = (int)std::min<long long>(tiles, (long long)kSmCount * (F == 64 ? 2 : 4));
    k_pair_filter<F, KP, HID><<<std::max(1, grid), T::NT, sizeof(T), s>>>(a, a.filter, K, l0, l1, a0, a1);
    count_launch();
}

template <int F>
void filters(const PotArgs& a, int K, int l0, int l1, int a0, int a1, cudaStream_t s) {
    if (a.spec_row && l0 == 0) {
        if (K <= 8) filter_go<F, 8, true>(a, K, l0, l1, a0, a1, s);
        else filter_go<F, 16, true>(a, K, l0, l1, a0, a1, s);
    } else {
        if (K <= 8) filter_go<F, 8, false>(a, K, l0, l1, a0, a1, s);
        else filter_go<F, 16, false>(a, K, l0, l1, a0, a1, s);
    }
}

// Blocks for the atoms a0 .. a1 - 1: a multiple of the SM count once there are
// that many (gather_range).
inline int gather_blocks(const PotArgs& a, int a0, int a1) {
    const int n = (a1 - a0 + a.atoms_per_cta - 1) / a.atoms_per_cta;
    return n < kSmCount ? n : (n + kSmCount - 1) / kSmCount * kSmCount;
}

template <int F>
void fwd_gather(const PotArgs& a, int a0, int a1, cudaStream_t s) {
    const int grid = gather_blocks(a, a0, a1);
    if (a.layer > 0 || !a.spec_row) k_gather<F, true><<<grid, kThreads, 0, s>>>(a, a.filter, a.u, a0, a1);
    else if (a.n_species <= 2) k_gather_species<F, 2><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1);
    else k_gather_species<F, kMaxFactorSpecies><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1);
    count_launch();
}

template <int F>
void fwd_go(const PotArgs& a, int K, cudaStream_t s) {
    if (!a.filter.chunk_atoms) {
        if (a.layer == 0) {                              // the filters of every layer at once
            k_pair_index<<<(a.n_atoms + kIdxWarps - 1) / kIdxWarps, kIdxWarps * 32, 0, s>>>(a, a.filter);
            count_launch();
            filters<F>(a, K, 0, a.n_layers, 0, a.n_atoms, s);
        }
        fwd_gather<F>(a, 0, a.n_atoms, s);
        return;
    }
    for (int a0 = 0; a0 < a.n_atoms; a0 += a.filter.chunk_atoms) {
        const int a1 = std::min(a.n_atoms, a0 + a.filter.chunk_atoms);
        filters<F>(a, K, a.layer, a.layer + 1, a0, a1, s);
        fwd_gather<F>(a, a0, a1, s);
    }
}

// The forces need every layer's dE/dd: summed over the layers per unordered
// pair, then one pass; chunked, one pass per layer and chunk.
template <int F>
void bwd_go(const PotArgs& a, int K, cudaStream_t s) {
    const bool half = !a.filter.chunk_atoms;
    const int step = half ? a.n_atoms : a.filter.chunk_atoms;
    const bool top = a.layer == a.n_layers - 1;
    for (int a0 = 0; a0 < a.n_atoms; a0 += step) {
        const int a1 = std::min(a.n_atoms, a0 + step), grid = gather_blocks(a, a0, a1);
        if (!half) filters<F>(a, K, a.layer, a.layer + 1, a0, a1, s);
        const int warps = (int)std::min<long long>((a.filter.cap + 31) / 32, (long long)kSmCount * 8 * (F == 64 ? 3 : 4));
        const int pgrid = (warps + kThreads / 32 - 1) / (kThreads / 32);
        if (a.n_layers == 1) {
            if (a.virial) k_row_force<F, 9><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1);
            else k_row_force<F, 3><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1);
            count_launch();
            continue;
        }
        if (a.layer == 0) {
            if (a.spec_row) k_pair_dedd<F, true, true><<<pgrid, kThreads, 0, s>>>(a, a.filter, a0, a1, half && !top);
            else k_pair_dedd<F, true, false><<<pgrid, kThreads, 0, s>>>(a, a.filter, a0, a1, half && !top);
        } else {
            k_pair_dedd<F, false, false><<<pgrid, kThreads, 0, s>>>(a, a.filter, a0, a1, half && !top);
            k_gather<F, false><<<grid, kThreads, 0, s>>>(a, a.filter, a.mbar, a0, a1);
            count_launch();
        }
        count_launch();
        if (half && a.layer > 0) continue;
        const int acc = half ? 0 : a.accumulate;
        if (a.virial) k_pair_force<9><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1, acc);
        else k_pair_force<3><<<grid, kThreads, 0, s>>>(a, a.filter, a0, a1, acc);
        count_launch();
    }
}

}  // namespace

void launch_embed(const PotArgs& a, int F, float* h_spec, float* u_spec, cudaStream_t s) {
    if (a.n_atoms == 0) return;
    int total = (a.n_atoms + a.n_species) * F;
    if (F == 64) k_embed<64><<<(total + 255) / 256, 256, 0, s>>>(a, h_spec, u_spec);
    else k_embed<32><<<(total + 255) / 256, 256, 0, s>>>(a, h_spec, u_spec);
    count_launch();
}

void launch_edge_fwd_f32(const PotArgs& a, int F, int K, cudaStream_t s) {
    if (a.n_atoms == 0) return;
    if (F == 64) fwd_go<64>(a, K, s);
    else fwd_go<32>(a, K, s);
}

void launch_edge_bwd_f32(const PotArgs& a, int F, int K, cudaStream_t s) {
    if (a.n_atoms == 0) return;
    if (F == 64) bwd_go<64>(a, K, s);
    else bwd_go<32>(a, K, s);
}

// ------------------------------------------------------------ reductions
// Per-system FP64 sums in a fixed order (deterministic): one CTA per system,
// strided partial sums, then fixed-shape shuffle trees (deterministic).
template <int NT>
__global__ void __launch_bounds__(NT) k_system_sum(int n_sys, const int* __restrict__ off,
                                                  const double* __restrict__ v, double* __restrict__ out,
                                                  int stride) {
    __shared__ double wsum[NT / 32];
    const int s = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double acc = 0.0;
    for (int i = off[s] + threadIdx.x; i < off[s + 1]; i += NT) acc += v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) wsum[w] = acc;
    __syncthreads();
    if (w == 0) {
        double t = lane < NT / 32 ? wsum[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) out[(size_t)s * stride] = t;
    }
}

// A few large systems: each system's values in kSumChunks consecutive
// chunks, one CTA per chunk (fixed-order partial sums); the CTA of a system
// that finishes last adds the partials in chunk order and clears the
// system's counter. The FP64 additions spread over many SMs.
template <int NT>
__global__ void __launch_bounds__(NT) k_system_sum_split(const int* __restrict__ off, const double* __restrict__ v,
                                                        double* __restrict__ out, int stride,
                                                        double* __restrict__ part, unsigned int* __restrict__ ctr) {
    __shared__ double wsum[NT / 32];
    __shared__ bool last;
    const int s = blockIdx.y, b = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int begin = off[s], end = off[s + 1];
    const int per = (end - begin + kSumChunks - 1) / kSumChunks;
    const int lo = begin + b * per, hi = min(end, lo + per);
    double acc = 0.0;
    for (int i = lo + threadIdx.x; i < hi; i += NT) acc += v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) wsum[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < NT / 32; ++k) t += wsum[k];
        part[(size_t)s * kSumChunks + b] = t;
        __threadfence();
        last = atomicAdd(&ctr[s], 1u) == (unsigned int)kSumChunks - 1u;
    }
    __syncthreads();
    if (last && w == 0) {
        __threadfence();
        double u = 0.0;
        for (int k = lane; k < kSumChunks; k += 32) u += __ldcg(part + (size_t)s * kSumChunks + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) u += __shfl_down_sync(0xffffffffu, u, o);
        if (lane == 0) {
            out[(size_t)s * stride] = u;
            ctr[s] = 0u;
        }
    }
}

void launch_system_sum(int n_sys, const int* atom_offset, const double* per_atom, double* out,
                       int stride, const SumScratch& sc, cudaStream_t s) {
    if (n_sys <= kSumMaxSplit && sc.part) {
        k_system_sum_split<256><<<dim3(kSumChunks, n_sys), 256, 0, s>>>(atom_offset, per_atom, out, stride, sc.part,
                                                                         sc.ctr);
    } else if (n_sys <= 8) {
        // one CTA per system: wide for a single large system, narrow for many molecules
        k_system_sum<1024><<<n_sys, 1024, 0, s>>>(n_sys, atom_offset, per_atom, out, stride);
    } else {
        k_system_sum<64><<<n_sys, 64, 0, s>>>(n_sys, atom_offset, per_atom, out, stride);
    }
    count_launch();
}

__global__ void k_virial_sum(int n_sys, const int* __restrict__ off, const float* __restrict__ v6,
                             double* __restrict__ out) {
    __shared__ double sh[6][128];
    int s = blockIdx.x;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int i = off[s] + threadIdx.x; i < off[s + 1]; i += blockDim.x)
        for (int c = 0; c < 6; ++c) acc[c] += (double)v6[(size_t)i * 6 + c];
    for (int c = 0; c < 6; ++c) sh[c][threadIdx.x] = acc[c];
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 6; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double* o = out + (size_t)s * 9;
        o[0] = sh[0][0]; o[4] = sh[1][0]; o[8] = sh[2][0];
        o[1] = o[3] = sh[3][0];
        o[2] = o[6] = sh[4][0];
        o[5] = o[7] = sh[5][0];
    }
}

// A few large systems: as k_system_sum_split, for the six components at once
// (FP64 additions run at two lanes per SM and clock: in one block, the virial of
// 12,288 atoms made the call 752 -> 808 us).
__global__ void __launch_bounds__(128) k_virial_split(const int* __restrict__ off, const float* __restrict__ v6,
                                                      double* __restrict__ out, double* __restrict__ part,
                                                      unsigned int* __restrict__ ctr) {
    __shared__ double wsum[4][6];
    __shared__ bool last;
    const int s = blockIdx.y, b = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int begin = off[s], end = off[s + 1];
    const int per = (end - begin + kSumChunks - 1) / kSumChunks;
    const int lo = begin + b * per, hi = min(end, lo + per);
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int i = lo + threadIdx.x; i < hi; i += 128)
#pragma unroll
        for (int c = 0; c < 6; ++c) acc[c] += (double)v6[(size_t)i * 6 + c];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], o);
        if (lane == 0) wsum[w][c] = acc[c];
    }
    __syncthreads();
    double* p = part + ((size_t)s * kSumChunks + b) * 6;
    if (threadIdx.x < 6) {
        p[threadIdx.x] = (wsum[0][threadIdx.x] + wsum[1][threadIdx.x]) + (wsum[2][threadIdx.x] + wsum[3][threadIdx.x]);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctr[s], 1u) == (unsigned int)kSumChunks - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    __shared__ double tot[6];
    if (threadIdx.x < 6) {
        double t = 0.0;
        for (int k = 0; k < kSumChunks; ++k) t += __ldcg(part + ((size_t)s * kSumChunks + k) * 6 + threadIdx.x);
        tot[threadIdx.x] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double* o = out + (size_t)s * 9;
        o[0] = tot[0]; o[4] = tot[1]; o[8] = tot[2];
        o[1] = o[3] = tot[3];
        o[2] = o[6] = tot[4];
        o[5] = o[7] = tot[5];
        ctr[s] = 0u;
    }
}

void launch_virial_sum(int n_sys, const int* atom_offset, const float* vir6, double* out, const SumScratch& sc,
                       cudaStream_t s) {
    if (n_sys <= kSumMaxSplit && sc.part)
        k_virial_split<<<dim3(kSumChunks, n_sys), 128, 0, s>>>(atom_offset, vir6, out, sc.part, sc.ctr);
    else
        k_virial_sum<<<n_sys, 128, 0, s>>>(n_sys, atom_offset, vir6, out);
    count_launch();
}

}  // namespace dmts
