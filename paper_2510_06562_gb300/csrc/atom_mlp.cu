// Per-atom MLPs of the potential (FP32, register-blocked SIMT), run after the
// edge passes have produced the per-atom sums: in the FP32 mode, and in the
// BF16 mode for models narrower than F = 64 (wider ones use the tensor-core
// kernels of atom_tc.cu):
//
//   forward, layer l:   z = m U1 + c1;  h <- h + SiLU(z) U2 + c2;
//                       l < L-1:  u^{l+1} = h W_in^{l+1}
//                       l = L-1:  q = h R1 + d1;  E_i = SiLU(q) . R2 + d2 + e0[Z_i] + E_rep,i
//                                 and the first adjoint steps:
//                                 gh = (SiLU'(q) * R2) R1^T;  mbar^l = ((gh U2^T) * SiLU'(z)) U1^T
//   backward, layer l >= 1:  gh <- gh + ubar^l W_in^{l T};
//                            mbar^{l-1} = ((gh U2^{l-1 T}) * SiLU'(z^{l-1})) U1^{l-1 T}
//
// Layer 0 reads h^0 = A[Z_i] from the per-atom copy built once per parameter
// upload. A CTA takes A = 8, 16 or 32 atoms; each stage is an [A x F] x [F x F]
// product, each thread owning RA = A / 8 atoms x RF features (4 at F = 64; 2
// at F = 32, so that the narrow model still has 4 warps per CTA). Inputs stay in their
// natural [atom][k] layout in shared memory. The weight matrices (row-major;
// the transposed ones are copies prepared on the host) all stream in at the
// start, or, at 32 atoms per CTA, where their shared memory costs residency
// (3.5 % of a 3 fs step of 100,000 atoms), the next stage's while the current
// one computes.
#include <cuda_bf16.h>

#include "internal.cuh"

namespace dmts {

namespace {

template <int F, int RA_>
struct AtomTile {
    static constexpr int RA = RA_;          // atoms per thread
    static constexpr int A = 8 * RA;        // atoms per CTA
    static constexpr int RF = F >= 64 ? 4 : 2;  // features per thread
    static constexpr int FG = F / RF;       // feature groups
    static constexpr int NT = (A / RA) * FG; // threads per CTA: 128
    static constexpr int XS = F + 4;        // row stride of per-atom rows [a][k]
    static constexpr int WS = F + 4;        // row stride of staged weights [k][f]
    static constexpr bool PRE = RA < 4;     // every matrix in its own buffer, loaded at the start
    static constexpr int smem(int slots) { return (2 * A * XS + (PRE ? slots : 2) * F * WS) * 4; }
    static_assert(FG <= 32 && 32 % FG == 0, "an atom's feature groups are lanes of one warp");
};

__device__ __forceinline__ float sig(float x) { return 1.0f / (1.0f + __expf(-x)); }

__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// RF consecutive floats (RF = 2 or 4, aligned to RF floats) to and from registers.
template <int RF>
__device__ __forceinline__ void ld_vec(float (&d)[RF], const float* s) {
    if constexpr (RF == 4) {
        const float4 x = *reinterpret_cast<const float4*>(s);
        d[0] = x.x; d[1] = x.y; d[2] = x.z; d[3] = x.w;
    } else {
        const float2 x = *reinterpret_cast<const float2*>(s);
        d[0] = x.x; d[1] = x.y;
    }
}
template <int RF>
__device__ __forceinline__ void st_vec(float* d, const float (&v)[RF]) {
    if constexpr (RF == 4) *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
    else *reinterpret_cast<float2*>(d) = make_float2(v[0], v[1]);
}

// Weight buffers of the forward kernel: one each (PRE), or two in turn by the slot's parity
// (layer 0 by species, which is never the last layer, has W2 in the place of R1^T).
enum WSlot { kU1, kU2, kOut, kR1T, kU2T, kU1T, kSlots, kW2 = kR1T };

// Start copying the row-major F x F matrix W into Ws [F][WS]; joins the next commit group.
template <int F, int RA>
__device__ __forceinline__ void copy_w(float* Ws, const float* __restrict__ W) {
    using T = AtomTile<F, RA>;
    for (int t = threadIdx.x; t < F * F / 4; t += T::NT) {
        const int r = t / (F / 4), c = (t % (F / 4)) * 4;
        cp_async16(Ws + r * T::WS + c, W + (size_t)r * F + c);
    }
}

// The same as a commit group of its own.
template <int F, int RA>
__device__ __forceinline__ void stage_w(float* Ws, const float* __restrict__ W) {
    copy_w<F, RA>(Ws, W);
    cp_commit();
}

// Start copying rows base .. base + A - 1 of the [N][F] array src into X [A][XS]
// (rows past N are zero); joins the next commit group.
template <int F, int RA>
__device__ __forceinline__ void stage_rows(float* X, const float* __restrict__ src, int base, int n_atoms) {
    using T = AtomTile<F, RA>;
    for (int t = threadIdx.x; t < T::A * F / 4; t += T::NT) {
        const int a = t / (F / 4), c = (t % (F / 4)) * 4;
        if (base + a < n_atoms) cp_async16(X + a * T::XS + c, src + (size_t)(base + a) * F + c);
        else *reinterpret_cast<float4*>(X + a * T::XS + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// acc[a][f] = sum_k X[a0 + a][k] * Ws[k][f0 + f], k ascending.
template <int F, int RA>
__device__ __forceinline__ void gemm_blk(const float* X, const float* Ws, int a0, int f0,
                                         float (&acc)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF]) {
    using T = AtomTile<F, RA>;
#pragma unroll
    for (int a = 0; a < T::RA; ++a)
#pragma unroll
        for (int f = 0; f < T::RF; ++f) acc[a][f] = 0.f;
#pragma unroll 4
    for (int k = 0; k < F; k += 4) {
        float xv[T::RA][4];
#pragma unroll
        for (int a = 0; a < T::RA; ++a) ld_vec<4>(xv[a], X + (a0 + a) * T::XS + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float w[T::RF];
            ld_vec<T::RF>(w, Ws + (k + kk) * T::WS + f0);
#pragma unroll
            for (int a = 0; a < T::RA; ++a)
#pragma unroll
                for (int f = 0; f < T::RF; ++f) acc[a][f] += xv[a][kk] * w[f];
        }
    }
}

// The same for species s of the [N][n_species][F] sums.
template <int F, int RA>
__device__ __forceinline__ void stage_species(float* X, const float* __restrict__ src, int s, int n_species, int base,
                                              int n_atoms) {
    using T = AtomTile<F, RA>;
    for (int t = threadIdx.x; t < T::A * F / 4; t += T::NT) {
        const int a = t / (F / 4), c = (t % (F / 4)) * 4;
        if (base + a < n_atoms) cp_async16(X + a * T::XS + c, src + ((size_t)(base + a) * n_species + s) * F + c);
        else *reinterpret_cast<float4*>(X + a * T::XS + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

template <int F, int RA>
__device__ __forceinline__ void put_rows(float* X, int a0, int f0,
                                         const float (&v)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF]) {
    using T = AtomTile<F, RA>;
#pragma unroll
    for (int a = 0; a < T::RA; ++a) st_vec<T::RF>(X + (a0 + a) * T::XS + f0, v[a]);
}

template <int F, int RA>
__device__ __forceinline__ void store_rows(float* __restrict__ dst, int base, int n_atoms, int a0, int f0,
                                           const float (&v)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF]) {
    using T = AtomTile<F, RA>;
#pragma unroll
    for (int a = 0; a < T::RA; ++a) {
        const int i = base + a0 + a;
        if (i < n_atoms) st_vec<T::RF>(dst + (size_t)i * F + f0, v[a]);
    }
}

// BF16 copy of the same block into interleaved rows (F * 4 bytes per atom;
// per 16 features 16 u values then 16 mbar values, half 0 or 1).
template <int F, int RA>
__device__ __forceinline__ void store_rows_bf16(unsigned char* __restrict__ dst, int half, int base, int n_atoms,
                                                int a0, int f0, const float (&v)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF]) {
    using T = AtomTile<F, RA>;
    if (!dst) return;
#pragma unroll
    for (int a = 0; a < T::RA; ++a) {
        const int i = base + a0 + a;
        if (i >= n_atoms) continue;
        unsigned char* row = dst + (size_t)i * F * 4 + (f0 >> 4) * 64 + half * 32 + (f0 & 15) * 2;
        __nv_bfloat162 lo = __floats2bfloat162_rn(v[a][0], v[a][1]);
        if constexpr (T::RF == 4) {
            __nv_bfloat162 hi = __floats2bfloat162_rn(v[a][2], v[a][3]);
            uint2 w;
            w.x = *reinterpret_cast<uint32_t*>(&lo);
            w.y = *reinterpret_cast<uint32_t*>(&hi);
            *reinterpret_cast<uint2*>(row) = w;
        } else {
            *reinterpret_cast<uint32_t*>(row) = *reinterpret_cast<uint32_t*>(&lo);
        }
    }
}

template <int F, int RA>
__device__ __forceinline__ void load_rows(float (&v)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF], const float* __restrict__ src,
                                          int base, int n_atoms, int a0, int f0) {
    using T = AtomTile<F, RA>;
#pragma unroll
    for (int a = 0; a < T::RA; ++a) {
        const int i = base + a0 + a;
        if (i < n_atoms) {
            ld_vec<T::RF>(v[a], src + (size_t)i * F + f0);
        } else {
#pragma unroll
            for (int f = 0; f < T::RF; ++f) v[a][f] = 0.f;
        }
    }
}

// Transposed F x F copies: W_in^T, U1^T, U2^T of every layer, then R1^T.
__device__ __forceinline__ const float* wt_of(const PotArgs& p, int F, int l, int which) {
    return p.PT + ((size_t)3 * l + which) * F * F;
}
__device__ __forceinline__ const float* r1t_of(const PotArgs& p, int F) {
    return p.PT + (size_t)3 * p.n_layers * F * F;
}

__device__ __forceinline__ const float* w2t_of(const PotArgs& p, int F) {
    return p.PT + ((size_t)3 * p.n_layers + 1) * F * F;
}

// Layer 0 by species, backward: from the block's mbar^0 (v) the rows
// Y_is = W2 (mbar_i * u_s) and scalars B_is = b2 . (mbar_i * u_s) of every
// species s, over the forward pass's sums. W holds W2^T; A0 and A1 are row
// buffers, A0 free on entry, A1 read by the preceding product.
template <int F, int RA>
__device__ __forceinline__ void species_adjoint(const PotArgs& p, float* A0, float* A1, const float* W, int base, int a0,
                                                int f0, const float (&v)[AtomTile<F, RA>::RA][AtomTile<F, RA>::RF]) {
    using T = AtomTile<F, RA>;
    float b2[T::RF];
#pragma unroll
    for (int f = 0; f < T::RF; ++f) b2[f] = __ldg(p.P + p.off.b2[0] + f0 + f);
    for (int s = 0; s < p.n_species; ++s) {
        float x[T::RA][T::RF], y[T::RA][T::RF], part[T::RA];
#pragma unroll
        for (int a = 0; a < T::RA; ++a) part[a] = 0.f;
#pragma unroll
        for (int f = 0; f < T::RF; ++f) {
            const float us = __ldg(p.u_spec + s * F + f0 + f);
#pragma unroll
            for (int a = 0; a < T::RA; ++a) {
                x[a][f] = v[a][f] * us;
                part[a] += x[a][f] * b2[f];
            }
        }
        put_rows<F, RA>(A0, a0, f0, x);
#pragma unroll
        for (int a = 0; a < T::RA; ++a)
#pragma unroll
            for (int o = T::FG / 2; o > 0; o >>= 1) part[a] += __shfl_xor_sync(0xffffffffu, part[a], o);
        __syncthreads();
        gemm_blk<F, RA>(A0, W, a0, f0, y);
#pragma unroll
        for (int a = 0; a < T::RA; ++a) {
            const int i = base + a0 + a;
            if (i >= p.n_atoms) continue;
            const size_t row = (size_t)i * p.n_species + s;
            st_vec<T::RF>(p.spec_row + row * F + f0, y[a]);
            if (f0 == 0) p.spec_sum[row] = part[a];
        }
        float* t = A0; A0 = A1; A1 = t;
    }
}

template <int F, int RA, bool SPEC>
__global__ void __launch_bounds__(AtomTile<F, RA>::NT) k_atom_fwd(PotArgs p, const float* __restrict__ msg) {
    using T = AtomTile<F, RA>;
    extern __shared__ float4 smem4[];
    float* X = reinterpret_cast<float*>(smem4);      // [A][XS]
    float* Y = X + T::A * T::XS;                     // [A][XS]
    float* Wb = Y + T::A * T::XS;                    // weight buffers [F][WS]
    auto W = [&](int slot) { return Wb + (T::PRE ? slot : slot & 1) * F * T::WS; };
    __shared__ float sE[T::A];
    __shared__ float sBias[4][F];                    // c1, c2 of this layer; d1, R2 (last layer)
    const int l = p.layer;
    const int base = blockIdx.x * T::A;
    const int tid = threadIdx.x, fg = tid % T::FG, ag = tid / T::FG;
    const int f0 = T::RF * fg, a0 = T::RA * ag;
    const float* P = p.P;
    const bool last = (l == p.n_layers - 1);
    float z[T::RA][T::RF], v[T::RA][T::RF], h[T::RA][T::RF];

    const bool by_species = SPEC && l == 0;          // the messages are formed here (below)
    if (by_species) {
        stage_species<F, RA>(X, p.spec_row, 0, p.n_species, base, p.n_atoms);
        stage_w<F, RA>(W(kW2), P + p.off.W2[0]);                         // group: first species' sums + W2
    } else {
        stage_rows<F, RA>(X, msg, base, p.n_atoms);
        stage_w<F, RA>(W(kU1), P + p.off.U1[l]);                         // group: message rows + U1
    }
    if constexpr (T::PRE) {                                              // group: all other matrices
        if (by_species) copy_w<F, RA>(W(kU1), P + p.off.U1[l]);
        copy_w<F, RA>(W(kU2), P + p.off.U2[l]);
        copy_w<F, RA>(W(kOut), last ? P + p.off.R1 : P + p.off.W_in[l + 1]);
        if (last) {
            copy_w<F, RA>(W(kR1T), r1t_of(p, F));
            copy_w<F, RA>(W(kU2T), wt_of(p, F, l, 2));
            copy_w<F, RA>(W(kU1T), wt_of(p, F, l, 1));
        }
        cp_commit();
    } else {
        if (by_species) stage_w<F, RA>(W(kU1), P + p.off.U1[l]);         // group: U1
        else stage_w<F, RA>(W(kU2), P + p.off.U2[l]);                    // group: U2
    }
    load_rows<F, RA>(h, p.h_in, base, p.n_atoms, a0, f0);
    // the small per-layer vectors and the per-atom energy constants, loaded while the copies run
    for (int t = tid; t < F; t += T::NT) {
        sBias[0][t] = __ldg(P + p.off.c1[l] + t);
        sBias[1][t] = __ldg(P + p.off.c2[l] + t);
        if (last) {
            sBias[2][t] = __ldg(P + p.off.d1 + t);
            sBias[3][t] = __ldg(P + p.off.R2 + t);
        }
    }
    // After a tensor-core forward pass that left its split rows to this kernel
    // (fused_fixup): a row split across 128-pair tiles gets the head tile's
    // last carry slot plus the later tiles' first slots, in tile order, and a
    // row without pairs zeros (the order and sums of the separate fix-up pass).
    auto split_row = [&](int i, long long& t0, long long& t1) -> int {   // 0: in one tile, 1: split, 2: empty
        const long long r0 = min((long long)p.row_ptr[i], p.e_cap), r1 = min((long long)p.row_ptr[i + 1], p.e_cap);
        if (r1 <= r0) return 2;
        t0 = r0 >> 7;
        t1 = (r1 - 1) >> 7;
        return t0 == t1 ? 0 : 1;
    };
    double e_const = 0.0;                            // d2 + e0[Z_i] + E_rep,i of atom base + tid
    if (tid < T::A && base + tid < p.n_atoms && p.energy && (last || (p.fused_fixup && l == 0))) {
        const int i = base + tid;
        float erep = 0.f;
        if (l == 0 && p.fused_fixup) {               // E_rep,i is a scalar slot of the layer-0 pass
            long long t0 = 0, t1 = 0;
            const int k = split_row(i, t0, t1);
            if (k == 0) {
                erep = p.erep[i];
            } else if (k == 1) {
                erep = p.carry[(2 * t0 + 1) * (long long)p.carry_w + F];
                for (long long u = t0 + 1; u <= t1; ++u) erep += p.carry[2 * u * (long long)p.carry_w + F];
            }
            p.erep[i] = erep;                        // read again by the last layer of deeper models
        } else {
            erep = p.erep[i];
        }
        if (last) e_const = (double)__ldg(P + p.off.d2) + (double)__ldg(P + p.off.e0 + p.species[i]) + (double)erep;
    }
    if (by_species) {
        // m_i = sum_s u_s * (T_is W2 + t_is b2)
        float m[T::RA][T::RF];
#pragma unroll
        for (int a = 0; a < T::RA; ++a)
#pragma unroll
            for (int f = 0; f < T::RF; ++f) m[a][f] = 0.f;
        float *cur = X, *nxt = Y;
        for (int s = 0; s < p.n_species; ++s) {
            if (s + 1 < p.n_species) {
                stage_species<F, RA>(nxt, p.spec_row, s + 1, p.n_species, base, p.n_atoms);
                cp_commit();
                if (s == 0) cp_wait<2>();                                // (U1 is in flight too)
                else cp_wait<1>();
            } else {
                cp_wait<0>();
            }
            __syncthreads();
            gemm_blk<F, RA>(cur, W(kW2), a0, f0, v);
            float t[T::RA];
#pragma unroll
            for (int a = 0; a < T::RA; ++a)
                t[a] = base + a0 + a < p.n_atoms ? p.spec_sum[(size_t)(base + a0 + a) * p.n_species + s] : 0.f;
#pragma unroll
            for (int f = 0; f < T::RF; ++f) {
                const float us = __ldg(p.u_spec + s * F + f0 + f), b2 = __ldg(P + p.off.b2[0] + f0 + f);
#pragma unroll
                for (int a = 0; a < T::RA; ++a) m[a][f] += us * (v[a][f] + t[a] * b2);
            }
            __syncthreads();                                             // cur (and, at the end, W2) read
            float* sw = cur; cur = nxt; nxt = sw;
        }
        if (!T::PRE) stage_w<F, RA>(W(kU2), P + p.off.U2[l]);            // group: U2
        put_rows<F, RA>(X, a0, f0, m);
    }
    cp_wait<1>();
    __syncthreads();
    if (p.fused_fixup) {
#pragma unroll
        for (int a = 0; a < T::RA; ++a) {
            const int i = base + a0 + a;
            if (i >= p.n_atoms) continue;
            long long t0 = 0, t1 = 0;
            const int k = split_row(i, t0, t1);
            if (k == 0) continue;
            float v[T::RF];
#pragma unroll
            for (int f = 0; f < T::RF; ++f) v[f] = 0.f;
            if (k == 1) {
                ld_vec<T::RF>(v, p.carry + (2 * t0 + 1) * (long long)p.carry_w + f0);
                for (long long u = t0 + 1; u <= t1; ++u) {
                    float w[T::RF];
                    ld_vec<T::RF>(w, p.carry + 2 * u * (long long)p.carry_w + f0);
#pragma unroll
                    for (int f = 0; f < T::RF; ++f) v[f] += w[f];
                }
            }
            st_vec<T::RF>(X + (a0 + a) * T::XS + f0, v);
        }
        __syncthreads();
    }
    gemm_blk<F, RA>(X, W(kU1), a0, f0, z);                               // z = m U1 + c1
#pragma unroll
    for (int f = 0; f < T::RF; ++f) {
        const float c1 = sBias[0][f0 + f];
#pragma unroll
        for (int a = 0; a < T::RA; ++a) {
            z[a][f] += c1;
            v[a][f] = z[a][f] * sig(z[a][f]);
        }
    }
    // a one-layer model read only for its force needs z, h, dE/dh and E_i of no later kernel
    const bool keep = !(p.lean && p.n_layers == 1);
    if (keep) store_rows<F, RA>(p.z, base, p.n_atoms, a0, f0, z);
    put_rows<F, RA>(Y, a0, f0, v);
    __syncthreads();                                                     // U1 read, Y complete
    if (!T::PRE) stage_w<F, RA>(W(kOut), last ? P + p.off.R1 : P + p.off.W_in[l + 1]);
    cp_wait<T::PRE ? 0 : 1>();
    __syncthreads();
    gemm_blk<F, RA>(Y, W(kU2), a0, f0, v);                               // h += SiLU(z) U2 + c2
#pragma unroll
    for (int f = 0; f < T::RF; ++f) {
        const float c2 = sBias[1][f0 + f];
#pragma unroll
        for (int a = 0; a < T::RA; ++a) h[a][f] += v[a][f] + c2;
    }
    if (keep) store_rows<F, RA>(p.h, base, p.n_atoms, a0, f0, h);
    put_rows<F, RA>(X, a0, f0, h);
    __syncthreads();                                                     // U2 read, X complete
    if (!last) {
        cp_wait<0>();
        __syncthreads();
        gemm_blk<F, RA>(X, W(kOut), a0, f0, v);                          // u^{l+1} = h W_in^{l+1}
        store_rows<F, RA>(p.u_next, base, p.n_atoms, a0, f0, v);
        store_rows_bf16<F, RA>(p.um_u_out, 0, base, p.n_atoms, a0, f0, v);
        return;
    }
    if constexpr (!T::PRE) {
        stage_w<F, RA>(W(kR1T), r1t_of(p, F));
        cp_wait<1>();
        __syncthreads();
    }
    gemm_blk<F, RA>(X, W(kOut), a0, f0, v);                              // q = h R1 + d1
    float e_part[T::RA];
#pragma unroll
    for (int a = 0; a < T::RA; ++a) e_part[a] = 0.f;
#pragma unroll
    for (int f = 0; f < T::RF; ++f) {
        const float d1 = sBias[2][f0 + f], r2 = sBias[3][f0 + f];
#pragma unroll
        for (int a = 0; a < T::RA; ++a) {
            const float q = v[a][f] + d1;
            const float s = sig(q);
            e_part[a] += q * s * r2;
            v[a][f] = s * (1.f + q * (1.f - s)) * r2;                  // dE/dq
        }
    }
    // sum the energy terms over the FG threads of this atom group (consecutive lanes)
#pragma unroll
    for (int a = 0; a < T::RA; ++a)
#pragma unroll
        for (int o = T::FG / 2; o > 0; o >>= 1) e_part[a] += __shfl_xor_sync(0xffffffffu, e_part[a], o);
    if (fg == 0)
#pragma unroll
        for (int a = 0; a < T::RA; ++a) sE[a0 + a] = e_part[a];
    put_rows<F, RA>(Y, a0, f0, v);
    __syncthreads();                                                     // R1 read, Y and sE complete
    if (!T::PRE) stage_w<F, RA>(W(kU2T), wt_of(p, F, l, 2));
    static_assert(T::NT >= T::A, "one thread per atom of the tile");
    if (keep && tid < T::A && base + tid < p.n_atoms) p.Ei[base + tid] = (double)sE[tid] + e_const;
    if constexpr (!T::PRE) {
        cp_wait<1>();
        __syncthreads();
    }
    gemm_blk<F, RA>(Y, W(kR1T), a0, f0, v);                              // gh = gq R1^T
    if (keep) store_rows<F, RA>(p.gh, base, p.n_atoms, a0, f0, v);
    put_rows<F, RA>(X, a0, f0, v);
    __syncthreads();                                                     // R1^T read, X complete
    if constexpr (!T::PRE) {
        stage_w<F, RA>(W(kU1T), wt_of(p, F, l, 1));
        cp_wait<1>();
        __syncthreads();
    }
    gemm_blk<F, RA>(X, W(kU2T), a0, f0, v);                              // gy = gh U2^T
#pragma unroll
    for (int a = 0; a < T::RA; ++a)
#pragma unroll
        for (int f = 0; f < T::RF; ++f) {
            const float s = sig(z[a][f]);
            v[a][f] *= s * (1.f + z[a][f] * (1.f - s));
        }
    put_rows<F, RA>(Y, a0, f0, v);
    cp_wait<0>();
    __syncthreads();                                                     // U2^T and X read, Y complete
    gemm_blk<F, RA>(Y, W(kU1T), a0, f0, v);                              // mbar = gz U1^T
    store_rows<F, RA>(p.mbar_out, base, p.n_atoms, a0, f0, v);
    store_rows_bf16<F, RA>(p.um_mbar_out, 1, base, p.n_atoms, a0, f0, v);
}

template <int F, int RA, bool SPEC>
__global__ void __launch_bounds__(AtomTile<F, RA>::NT) k_atom_bwd(PotArgs p, const float* __restrict__ ubar) {
    using T = AtomTile<F, RA>;
    extern __shared__ float4 smem4[];
    float* X = reinterpret_cast<float*>(smem4);
    float* Y = X + T::A * T::XS;
    float* Wb = Y + T::A * T::XS;
    auto W = [&](int slot) { return Wb + (T::PRE ? slot : slot & 1) * F * T::WS; };
    const int l = p.layer;   // >= 1
    const int base = blockIdx.x * T::A;
    const int tid = threadIdx.x, fg = tid % T::FG, ag = tid / T::FG;
    const int f0 = T::RF * fg, a0 = T::RA * ag;
    float v[T::RA][T::RF], g[T::RA][T::RF], z[T::RA][T::RF];
    stage_rows<F, RA>(X, ubar, base, p.n_atoms);
    const bool by_species = SPEC && l == 1;
    stage_w<F, RA>(W(0), wt_of(p, F, l, 0));                             // group: ubar rows + W_in^{l T}
    copy_w<F, RA>(W(1), wt_of(p, F, l - 1, 2));                          // group: U2^{l-1 T} (all other matrices)
    if constexpr (T::PRE) {
        copy_w<F, RA>(W(2), wt_of(p, F, l - 1, 1));
        if (by_species) copy_w<F, RA>(W(3), w2t_of(p, F));
    }
    cp_commit();
    load_rows<F, RA>(g, p.gh, base, p.n_atoms, a0, f0);
    load_rows<F, RA>(z, p.z_prev, base, p.n_atoms, a0, f0);
    cp_wait<1>();
    __syncthreads();
    gemm_blk<F, RA>(X, W(0), a0, f0, v);                                 // ubar W_in^T
#pragma unroll
    for (int a = 0; a < T::RA; ++a)
#pragma unroll
        for (int f = 0; f < T::RF; ++f) g[a][f] += v[a][f];
    store_rows<F, RA>(p.gh, base, p.n_atoms, a0, f0, g);
    put_rows<F, RA>(Y, a0, f0, g);
    if constexpr (!T::PRE) {
        __syncthreads();                                                 // W_in^T read
        stage_w<F, RA>(W(2), wt_of(p, F, l - 1, 1));                     // U1^{l-1 T}
        cp_wait<1>();
    } else {
        cp_wait<0>();
    }
    __syncthreads();                                                     // Y complete
    gemm_blk<F, RA>(Y, W(1), a0, f0, v);                                       // gy = gh U2^T
#pragma unroll
    for (int a = 0; a < T::RA; ++a)
#pragma unroll
        for (int f = 0; f < T::RF; ++f) {
            const float s = sig(z[a][f]);
            v[a][f] *= s * (1.f + z[a][f] * (1.f - s));
        }
    put_rows<F, RA>(X, a0, f0, v);
    cp_wait<0>();
    __syncthreads();                                                     // U2^T and Y read, X complete
    if (by_species && !T::PRE) stage_w<F, RA>(W(3), w2t_of(p, F));
    gemm_blk<F, RA>(X, W(2), a0, f0, v);                                 // mbar^{l-1} = gz U1^T
    store_rows<F, RA>(p.mbar_out, base, p.n_atoms, a0, f0, v);
    store_rows_bf16<F, RA>(p.um_mbar_out, 1, base, p.n_atoms, a0, f0, v);
    if (by_species) {
        cp_wait<0>();                                                    // (visible after the first barrier inside)
        species_adjoint<F, RA>(p, Y, X, W(3), base, a0, f0, v);
    }
}

template <int F, int RA, bool SPEC>
void atom_fwd_go(const PotArgs& p, const float* msg, cudaStream_t s) {
    using T = AtomTile<F, RA>;
    constexpr int bytes = T::smem(kSlots);
    smem_opt_in((const void*)k_atom_fwd<F, RA, SPEC>, bytes);
    k_atom_fwd<F, RA, SPEC><<<(p.n_atoms + T::A - 1) / T::A, T::NT, bytes, s>>>(p, msg);
}

template <int F, int RA, bool SPEC>
void atom_bwd_go(const PotArgs& p, const float* ubar, cudaStream_t s) {
    using T = AtomTile<F, RA>;
    constexpr int bytes = T::smem(SPEC ? 4 : 3);
    smem_opt_in((const void*)k_atom_bwd<F, RA, SPEC>, bytes);
    k_atom_bwd<F, RA, SPEC><<<(p.n_atoms + T::A - 1) / T::A, T::NT, bytes, s>>>(p, ubar);
}

template <int F, int RA>
void atom_go(const PotArgs& p, const float* x, bool fwd, cudaStream_t s) {
    const bool spec = p.spec_row && p.layer == (fwd ? 0 : 1);
    if (fwd) spec ? atom_fwd_go<F, RA, true>(p, x, s) : atom_fwd_go<F, RA, false>(p, x, s);
    else spec ? atom_bwd_go<F, RA, true>(p, x, s) : atom_bwd_go<F, RA, false>(p, x, s);
}

// Atoms per thread: as few as leave one block per SM. The products are then a
// chain of latencies, and a block of 8 atoms walks it in a third of the time
// of one of 32. Blocks of 32 atoms against these, us: FP32 forces of 192 atoms
// 171 -> 158, of 1,536 209 -> 199, of 2,187 230 -> 221, 1 fs step of 1,536
// 164 -> 155; 3 fs step in BF16 (the small model's kernels; steps back to back) of
// 192 atoms 174 -> 170, of 1,536 220 -> 217. At F = 32 the line is 1,824 atoms: at
// 2,187 that step takes 256 in blocks of 16 against 254.
template <int F>
void atom_any(const PotArgs& p, const float* x, bool fwd, cudaStream_t s) {
    if (p.n_atoms <= 8 * kSmCount) atom_go<F, 1>(p, x, fwd, s);
    else if (p.n_atoms <= (F == 64 ? 16 : 12) * kSmCount) atom_go<F, 2>(p, x, fwd, s);
    else atom_go<F, 4>(p, x, fwd, s);
    count_launch();
}

}  // namespace

void launch_atom_fwd(const PotArgs& p, int F, const float* msg, cudaStream_t s) {
    if (p.n_atoms == 0) return;
    if (F == 64) atom_any<64>(p, msg, true, s);
    else atom_any<32>(p, msg, true, s);
}

void launch_atom_bwd(const PotArgs& p, int F, const float* ubar, cudaStream_t s) {
    if (p.n_atoms == 0) return;
    if (F == 64) atom_any<64>(p, ubar, false, s);
    else atom_any<32>(p, ubar, false, s);
}

}  // namespace dmts
