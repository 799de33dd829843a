// PD local step on sm_103a, fused with the RHS assembly: per-tet deformation
// gradient, 3x3 SVD, rotation and volume targets, the per-corner
// right-hand-side contributions (in shared memory), and their deterministic
// sum per vertex into b (or into the residual b - K x).
//
// Paper: Sec. 7.1 (local step; R by polar decomposition, V through the
// three-unknown problem of Eq. vol_pre with targets clamped to >= 0.01),
// Eq. pd_local, Eq. energy (per-element gamma_s, gamma_v).  Ordinarily
// strained elements get both targets as one isotropic function of F^T F;
// inverted and strongly strained ones, and every one in pd_step's frames of the
// direct form (see local_corners), by the SVD and the enumeration of the volume
// problem's candidates (proj3.cuh).
//
// What bounds it: with the SVD path for every element the kernel was bound
// by instruction issue (1,050 thread instructions per element; 25.7 us for
// 390,000 elements, ncu, cold caches).  Without it 18.6 us (640 instructions
// with the vertex sums): the latency of the loads (long-scoreboard stalls, 39 %
// of the warps resident, 2.5 waves); 64-tet blocks, 96-tet blocks and 48
// registers measure within 0.5 % of this.
//
// The serving loop runs the same block code over every resident request in
// one launch (k_b_local_assemble, k_b_assemble_shared).

#include <algorithm>

#include "pd_internal.h"
#include "proj3.cuh"

namespace pdg {

namespace {

using namespace proj;

// Rotation and volume targets of n matrices.  390,000 of them: 25.5 us a call before (one matrix per thread read in
// place, SVD of each), 20-24 us now, of which the host's part is 19; bound by instruction issue (70 %).
// Matrices go through shared memory: consecutive threads read and write consecutive floats of the 36-byte records
// (read in place, a warp's loads touch nine times the lines), and the odd record length is free of bank conflicts.
constexpr int kProjThreads = 128;

__global__ void __launch_bounds__(kProjThreads) k_project(const float* __restrict__ Fin, int n, float* __restrict__ Rout,
                                                          float* __restrict__ Vout, float* __restrict__ sout) {
    __shared__ float buf[21 * kProjThreads];
    const int64_t e0 = (int64_t)blockIdx.x * kProjThreads;
    const int ne = (int)min((int64_t)kProjThreads, n - e0), tid = threadIdx.x;
    for (int l = tid; l < 9 * ne; l += kProjThreads) buf[l] = Fin[9 * e0 + l];
    __syncthreads();
    float F[3][3], R[3][3], V[3][3], s[3];
    const int me = min(tid, ne - 1);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) F[i][j] = buf[9 * me + 3 * i + j];
    Strain S;
    if (strain_of<true>(F, S)) {
        strain_apply<false>(F, S, 1.f, 0.f, R);
        strain_apply<false>(F, S, 0.f, 1.f, V);
        s[0] = S.s1;
        s[1] = S.s2;
        s[2] = S.s3;
    } else {
        float U[3][3], W[3][3], d[3];
        const float one[3] = {1.f, 1.f, 1.f};
        svd3(F, U, s, W);
        udwt(U, one, W, R);
        volume_targets(s, d);
        udwt(U, d, W, V);
    }
    // all three results in their own parts of the buffer: one exchange
    float *bR = buf, *bV = buf + 9 * kProjThreads, *bs = buf + 18 * kProjThreads;
    __syncthreads();           // the inputs have been read
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        bR[9 * tid + i] = R[i / 3][i % 3];
        bV[9 * tid + i] = V[i / 3][i % 3];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) bs[3 * tid + i] = s[i];
    __syncthreads();
    if (Rout)
        for (int l = tid; l < 9 * ne; l += kProjThreads) Rout[9 * e0 + l] = bR[l];
    if (Vout)
        for (int l = tid; l < 9 * ne; l += kProjThreads) Vout[9 * e0 + l] = bV[l];
    if (sout)
        for (int l = tid; l < 3 * ne; l += kProjThreads) sout[3 * e0 + l] = bs[l];
}

// geo holds three float4 rows per tet in SoA blocks:
// geo[t] = (g1, ws), geo[n_t + t] = (g2, wv), geo[2 n_t + t] = (g3, 0), with
// g_k the rows of Dm^-1 and ws = V_e gamma_s, wv = V_e gamma_v; the corner
// vectors are g_1, g_2, g_3 and g_0 = -(g1 + g2 + g3).
struct LocalIn {
    float4 r1, r2, r3, x0, x1, x2, x3;
};

// P = U diag(c) W^T for any element.
template <bool RESID>
__device__ __forceinline__ void svd_targets(const float (&F)[3][3], float ws, float wv, float (&P)[3][3]) {
    float U[3][3], W[3][3], s[3], d[3];
    svd3(F, U, s, W);
    volume_targets(s, d);
    float c[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) c[i] = RESID ? ws * (1.f - s[i]) + wv * (d[i] - s[i]) : ws + wv * d[i];
    udwt(U, c, W, P);
}

// The same out of line, for the rare element beside the fast path (which keeps its registers).
template <bool RESID>
__device__ __noinline__ void svd_targets_rare(const float (&F)[3][3], float ws, float wv, float (&P)[3][3]) {
    svd_targets<RESID>(F, ws, wv, P);
}

// Per-tet corner terms f_c = P g_c with P = U diag(c) W^T: the RHS form
// c_i = w_s + w_v d_i (P = w_s R + w_v V), or the residual form
// c_i = w_s (1 - s_i) + w_v (d_i - s_i) (P = w_s (R - F) + w_v (V - F), the
// elastic part of b - K x without cancellation: F = U diag(s) W^T).
//
// FAST: the SVD-free targets (strain_of).  pd_step's frames of the direct form
// (x = S(b), FP32) do not use them: there the rounding of every local step
// enters the positions at full size (an ulp of a 2 m garment is 4e-5 m/s of
// its velocity), and their trajectories stay what they were.  In the
// correction form it only enters the shrinking correction.  Served frames,
// direct form too, use them: on one domain they were the stepper's bitwise
// and are no longer, with the same error against FP64 (eight slabs and shells
// of 1,008 to 50,700 elements, frames 1, 5 and 30: positions 2.1e-7 .. 1.0e-4
// with, 2.1e-7 .. 1.4e-4 without; velocities 1.3e-5 .. 5.7e-3 and 1.4e-5 ..
// 6.7e-3, the largest on the coarsest one-layer shell).  Six requests with /
// without 42.8 / 46.0 ms; BF16 frame of the 390K shell 1.57 / 1.67 ms; FP32
// frames would gain from it: 390K shell 2.10 -> 2.00 ms, 140K shell 1.00 -> 0.93,
// 10 iterations of the small slab 178 -> 164 us.
template <bool RESID, bool FAST>
__device__ __forceinline__ void local_corners(const LocalIn& L, float (&out)[4][3]) {
    const float e1[3] = {L.x1.x - L.x0.x, L.x1.y - L.x0.y, L.x1.z - L.x0.z};
    const float e2[3] = {L.x2.x - L.x0.x, L.x2.y - L.x0.y, L.x2.z - L.x0.z};
    const float e3[3] = {L.x3.x - L.x0.x, L.x3.y - L.x0.y, L.x3.z - L.x0.z};
    const float g1[3] = {L.r1.x, L.r1.y, L.r1.z};
    const float g2[3] = {L.r2.x, L.r2.y, L.r2.z};
    const float g3[3] = {L.r3.x, L.r3.y, L.r3.z};
    float F[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) F[i][j] = e1[i] * g1[j] + e2[i] * g2[j] + e3[i] * g3[j];
    float P[3][3];
    const float ws = L.r1.w, wv = L.r2.w;
    if (FAST) {
        Strain S;
        if (strain_of<false>(F, S)) strain_apply<RESID>(F, S, ws, wv, P);
        else svd_targets_rare<RESID>(F, ws, wv, P);
    } else {
        svd_targets<RESID>(F, ws, wv, P);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        out[1][i] = P[i][0] * g1[0] + P[i][1] * g1[1] + P[i][2] * g1[2];
        out[2][i] = P[i][0] * g2[0] + P[i][1] * g2[1] + P[i][2] * g2[2];
        out[3][i] = P[i][0] * g3[0] + P[i][1] * g3[1] + P[i][2] * g3[2];
        out[0][i] = -(out[1][i] + out[2][i] + out[3][i]);
    }
}

// Fused local step and RHS assembly.  Tets are cut into blocks of kLaTets
// consecutive (domain-sorted) tets, one tet per thread; the block's corner
// terms go to shared memory, then every free vertex the block touches sums
// its corners there in increasing (tet, corner) order.  A vertex whose
// corners all lie in one block ("owned") is finished there:
//   RHS form:      b_v = by0_v + sum_c f_c
//   residual form: r_v = (m_v/dt^2)(y_v - x_v) + sum_c f_c  (= b_v - (K x)_v)
// A vertex shared by several blocks gets the block's partial sum in its
// slot (slots ordered by block); k_assemble_shared adds base + the slots in
// slot order (deterministic, no atomics).
constexpr int kLaTets = PDG_LA_TETS;
#ifndef PDG_LA_MINB
#define PDG_LA_MINB 8
#endif

template <bool RESID>
__device__ __forceinline__ float4 assembly_base(const LocalAsmArgs& A, int v) {
    if (RESID) {
        const float m = A.mh2[v];
        const float4 y = A.y[v], xv = A.x[v];
        return make_float4(m * (y.x - xv.x), m * (y.y - xv.y), m * (y.z - xv.z), 0.f);
    }
    return A.by0[v];
}

// One block of the fused kernel: tets [blk kLaTets, (blk + 1) kLaTets) of the mesh in A.
template <bool RESID, bool FAST>
__device__ __forceinline__ void local_assemble_block(const LocalAsmArgs& A, int blk) {
    __shared__ float fx[4 * kLaTets], fy[4 * kLaTets], fz[4 * kLaTets];
    pdl_trigger();
    const int e = blk * kLaTets + threadIdx.x;
    const bool live = e < A.n_t;
    const int ec = live ? e : A.n_t - 1;
    LocalIn L;
    const int4 tv = __ldg(&A.tets[ec]);
    L.r1 = __ldg(&A.geo[ec]);
    L.r2 = __ldg(&A.geo[A.n_t + ec]);
    L.r3 = __ldg(&A.geo[2 * (int64_t)A.n_t + ec]);
    const int j0 = __ldg(&A.vptr[blk]), j1 = __ldg(&A.vptr[blk + 1]);
    pdl_wait();   // x comes from the previous solve
    L.x0 = A.x[tv.x];
    L.x1 = A.x[tv.y];
    L.x2 = A.x[tv.z];
    L.x3 = A.x[tv.w];
    float f[4][3];
    local_corners<RESID, FAST>(L, f);
    if (live) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            fx[4 * threadIdx.x + c] = f[c][0];
            fy[4 * threadIdx.x + c] = f[c][1];
            fz[4 * threadIdx.x + c] = f[c][2];
        }
    }
    __syncthreads();
    for (int j = j0 + threadIdx.x; j < j1; j += kLaTets) {
        const int k0 = __ldg(&A.cptr[j]), k1 = __ldg(&A.cptr[j + 1]);
        float ax = 0.f, ay = 0.f, az = 0.f;
        for (int k = k0; k < k1; ++k) {
            const int q = __ldg(&A.corner[k]);
            ax += fx[q];
            ay += fy[q];
            az += fz[q];
        }
        const int slot = __ldg(&A.slot[j]);
        if (slot >= 0) {
            A.part[slot] = make_float4(ax, ay, az, 0.f);
        } else {
            const int v = __ldg(&A.vert[j]);
            const float4 base = assembly_base<RESID>(A, v);
            A.b[v] = make_float4(base.x + ax, base.y + ay, base.z + az, 0.f);
        }
    }
}

template <bool RESID, bool FAST>
__global__ void __launch_bounds__(kLaTets, PDG_LA_MINB) k_local_assemble(LocalAsmArgs A) {
    local_assemble_block<RESID, FAST>(A, blockIdx.x);
}

// shared vertices: b_v = base + the blocks' partial sums in block order
template <bool RESID>
__device__ __forceinline__ void assemble_shared_block(const LocalAsmArgs& A, int n_shared, int blk) {
    pdl_trigger();
    const int j = blk * 256 + threadIdx.x;
    const bool live = j < n_shared;
    const int v = live ? __ldg(&A.sh_vert[j]) : 0;
    const int s0 = live ? __ldg(&A.sh_ptr[j]) : 0, s1 = live ? __ldg(&A.sh_ptr[j + 1]) : 0;
    pdl_wait();   // the partial sums come from k_local_assemble
    if (!live) return;
    float4 acc = assembly_base<RESID>(A, v);
    for (int q = s0; q < s1; ++q) {
        const float4 p = A.part[q];
        acc.x += p.x;
        acc.y += p.y;
        acc.z += p.z;
    }
    A.b[v] = make_float4(acc.x, acc.y, acc.z, 0.f);
}

template <bool RESID>
__global__ void __launch_bounds__(256) k_assemble_shared(LocalAsmArgs A, int n_shared) {
    assemble_shared_block<RESID>(A, n_shared, blockIdx.x);
}

// Serving: the same two kernels over every resident request of a batch (RHS
// form); a block finds its request from the per-kernel block offsets, so each
// request's values come from exactly the arithmetic and order above.
__device__ __forceinline__ LocalAsmArgs batch_args(const BatchSlot& S) {
    LocalAsmArgs A{};
    A.n_t = S.n_t;
    A.tets = S.tets;
    A.geo = S.geo;
    A.x = S.x;
    A.by0 = S.by0;
    A.b = S.b;
    A.vptr = S.la_vptr;
    A.vert = S.la_vert;
    A.slot = S.la_slot;
    A.cptr = S.la_cptr;
    A.corner = S.la_corner;
    A.sh_ptr = S.la_sh_ptr;
    A.sh_vert = S.la_sh_vert;
    A.part = S.la_part;
    return A;
}

__global__ void __launch_bounds__(kLaTets, PDG_LA_MINB) k_b_local_assemble(const BatchSlot* __restrict__ slots,
                                                                         const int* __restrict__ off, int n_slots) {
    const int s = batch_find_slot(off, n_slots, blockIdx.x);
    local_assemble_block<false, true>(batch_args(slots[s]), blockIdx.x - off[s]);
}

__global__ void __launch_bounds__(256) k_b_assemble_shared(const BatchSlot* __restrict__ slots,
                                                         const int* __restrict__ off, int n_slots) {
    const int s = batch_find_slot(off, n_slots, blockIdx.x);
    const BatchSlot& S = slots[s];
    assemble_shared_block<false>(batch_args(S), S.la_shared, blockIdx.x - off[s]);
}

}  // namespace

// Assembly plan of the fused kernel from the tet -> (sorted) vertex table and
// the free-vertex incidence lists (increasing 4 t + c).
void build_local_plan(pd_mesh* m, const std::vector<int32_t>& inc_ptr, const std::vector<int32_t>& inc,
                      cudaStream_t s) {
    const int32_t n_t = m->n_t, n_free = m->n_free;
    const int32_t n_blk = std::max(1, (n_t + kLaTets - 1) / kLaTets);
    // per free vertex: the blocks its corners fall in (ascending, since inc is ascending)
    std::vector<int32_t> sh_of(n_free, -1), sh_ptr(1, 0), sh_vert;
    std::vector<int32_t> cnt_entries(n_blk, 0);
    for (int32_t v = 0; v < n_free; ++v) {
        int32_t nb = 0, last = -1;
        for (int32_t k = inc_ptr[v]; k < inc_ptr[v + 1]; ++k) {
            const int32_t b = (inc[k] / 4) / kLaTets;
            if (b != last) {
                ++nb;
                ++cnt_entries[b];
                last = b;
            }
        }
        if (nb > 1) {
            sh_of[v] = (int32_t)sh_vert.size();
            sh_vert.push_back(v);
            sh_ptr.push_back(sh_ptr.back() + nb);
        }
    }
    std::vector<int32_t> vptr(n_blk + 1, 0);
    for (int32_t b = 0; b < n_blk; ++b) vptr[b + 1] = vptr[b] + cnt_entries[b];
    const int32_t n_ent = vptr[n_blk];
    std::vector<int32_t> vert(n_ent), sidx(n_ent), slot(n_ent), ccount(n_ent, 0), fill(vptr.begin(), vptr.end() - 1);
    // entries in vertex order within each block; corner counts
    for (int32_t v = 0; v < n_free; ++v) {
        int32_t last = -1, rank = 0, j = -1;
        for (int32_t k = inc_ptr[v]; k < inc_ptr[v + 1]; ++k) {
            const int32_t b = (inc[k] / 4) / kLaTets;
            if (b != last) {
                j = fill[b]++;
                vert[j] = v;
                sidx[j] = sh_of[v];
                slot[j] = sh_of[v] < 0 ? -1 : sh_ptr[sh_of[v]] + rank;
                ++rank;
                last = b;
            }
            ++ccount[j];
        }
    }
    std::vector<int32_t> cptr(n_ent + 1, 0);
    for (int32_t j = 0; j < n_ent; ++j) cptr[j + 1] = cptr[j] + ccount[j];
    std::vector<uint16_t> corner(std::max<int32_t>(cptr[n_ent], 1));
    std::fill(ccount.begin(), ccount.end(), 0);
    std::fill(fill.begin(), fill.end(), 0);
    std::copy(vptr.begin(), vptr.end() - 1, fill.begin());
    for (int32_t v = 0; v < n_free; ++v) {
        int32_t last = -1, j = -1;
        for (int32_t k = inc_ptr[v]; k < inc_ptr[v + 1]; ++k) {
            const int32_t b = (inc[k] / 4) / kLaTets;
            if (b != last) {
                j = fill[b]++;
                last = b;
            }
            corner[cptr[j] + ccount[j]++] = (uint16_t)(inc[k] - 4 * b * kLaTets);
        }
    }
    (void)sidx;
    upload(m->d_la_vptr, vptr, s);
    upload(m->d_la_vert, vert, s);
    upload(m->d_la_slot, slot, s);
    upload(m->d_la_cptr, cptr, s);
    upload(m->d_la_corner, corner, s);
    upload(m->d_la_sh_ptr, sh_ptr, s);
    upload(m->d_la_sh_vert, sh_vert, s);
    m->d_la_part.alloc(std::max<size_t>(sh_ptr.back(), 1));
    m->la_blocks = n_blk;
    m->la_entries = n_ent;
    m->la_corners = cptr[n_ent];
    m->la_slots = sh_ptr.back();
    m->la_shared = (int32_t)sh_vert.size();
    PDG_CUDA(cudaStreamSynchronize(s));   // the host vectors are released on return
}

void launch_local_assemble(const pd_mesh* m, const float4* x, const float4* by0, const float4* y, float4* b,
                           bool residual, bool fast, cudaStream_t s) {
    if (m->n_t <= 0) return;
    LocalAsmArgs A{};
    A.n_t = m->n_t;
    A.tets = m->d_tets.p;
    A.geo = m->d_geo.p;
    A.x = x;
    A.by0 = by0;
    A.y = y;
    A.mh2 = m->d_mh2.p;
    A.b = b;
    A.vptr = m->d_la_vptr.p;
    A.vert = m->d_la_vert.p;
    A.slot = m->d_la_slot.p;
    A.cptr = m->d_la_cptr.p;
    A.corner = m->d_la_corner.p;
    A.sh_ptr = m->d_la_sh_ptr.p;
    A.sh_vert = m->d_la_sh_vert.p;
    A.part = m->d_la_part.p;
    const int nsb = (m->la_shared + 255) / 256;
    const dim3 grid(m->la_blocks), block(kLaTets);
    if (residual) launch_pdl(k_local_assemble<true, true>, grid, block, 0, s, A);
    else if (fast) launch_pdl(k_local_assemble<false, true>, grid, block, 0, s, A);
    else launch_pdl(k_local_assemble<false, false>, grid, block, 0, s, A);
    if (nsb > 0) {
        if (residual) launch_pdl(k_assemble_shared<true>, dim3(nsb), dim3(256), 0, s, A, m->la_shared);
        else launch_pdl(k_assemble_shared<false>, dim3(nsb), dim3(256), 0, s, A, m->la_shared);
    }
    PDG_CHECK_LAUNCH();
}

void launch_b_local_assemble(const BatchSlot* slots, const int* off, int n_slots, int blocks, cudaStream_t s) {
    if (blocks <= 0) return;
    launch_pdl(k_b_local_assemble, dim3(blocks), dim3(kLaTets), 0, s, slots, off, n_slots);
    PDG_CHECK_LAUNCH();
}

void launch_b_assemble_shared(const BatchSlot* slots, const int* off, int n_slots, int blocks, cudaStream_t s) {
    if (blocks <= 0) return;
    launch_pdl(k_b_assemble_shared, dim3(blocks), dim3(256), 0, s, slots, off, n_slots);
    PDG_CHECK_LAUNCH();
}

void launch_project(const float* F, int n, float* R, float* V, float* sig, cudaStream_t s) {
    if (n <= 0) return;
    k_project<<<(n + kProjThreads - 1) / kProjThreads, kProjThreads, 0, s>>>(F, n, R, V, sig);
    PDG_CHECK_LAUNCH();
}

}  // namespace pdg
