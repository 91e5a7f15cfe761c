// Learned k-step surrogate of the particle loop: a message-passing network
// over the SPH neighbour graph (edges |r_ij| < 2h), BF16 operands on the
// tensor cores (umma.cuh) with FP32 accumulation, hand-written forward and
// backward kernels, Adam, and the C ABI declared in include/sph_surrogate.h.
//
// The network and its parameter format are those of surrogate_layout.py:
// encoder, two rounds of [edge MLP on (h_i, h_j, e_ij), sum over j scaled by
// 1/k_ref, residual node MLP on (h, M)], decoder.  Every dense layer is one
// tcgen05 contraction over all nodes.  The edge MLP's first layer is split
// by blocks (W1 h_i + b1 and W2 h_j are node contractions, W3 e_ij is formed
// per edge) and its second layer, being linear, is applied after the sum
// (We2 S_i + deg_i / k_ref be2), so the per-edge work is one gather, the
// SiLU and the sum.  Nodes are the particles in the simulation's sorted
// order; the edges are the entries of its neighbour list closer than 2h.
#include "sph_internal.h"
#include "sph_kernels.cuh"
#include "sph_surrogate.h"
#include "umma.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

using namespace sphgb;
using bf16 = __nv_bfloat16;

namespace {

constexpr int H = 128;        // hidden width
constexpr int FIN = 16;       // padded node input width
constexpr int FOUT = 16;      // padded output width
constexpr int BWD_LAYERS = 12;   // dense layers with a weight gradient
constexpr int W3_SUMS = H * (2 * 3 + 3 + 1);   // edge weights and biases of a round, in 3-D
constexpr int SUMS = 2 * W3_SUMS + 10 * H;     // and the biases of ten layers

#define CUR(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) return set_error(SPH_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// Offsets of the parameter tensors in the flat vector, in the order of
// surrogate_layout.layout().
struct Layout {
    int dim = 0, nin = 0, ne = 0, nout = 0;
    int enc1w, enc1b, enc2w, enc2b;
    int w1[2], b1[2], w2[2], w3[2], we2[2], be2[2], n1[2], n1b[2], n2[2], n2b[2];
    int dec1w, dec1b, dec2w, dec2b;
    int total = 0;
};

Layout make_layout(int dim)
{
    Layout L;
    L.dim = dim;
    L.nin = 2 * dim + 4;
    L.ne = 2 * dim + 3;
    L.nout = 2 * dim + 1;
    int o = 0;
    auto take = [&](int k) {
        const int r = o;
        o += k;
        return r;
    };
    L.enc1w = take(H * L.nin);
    L.enc1b = take(H);
    L.enc2w = take(H * H);
    L.enc2b = take(H);
    for (int r = 0; r < 2; ++r) {
        L.w1[r] = take(H * H);
        L.b1[r] = take(H);
        L.w2[r] = take(H * H);
        L.w3[r] = take(H * L.ne);
        L.we2[r] = take(H * H);
        L.be2[r] = take(H);
        L.n1[r] = take(H * 2 * H);
        L.n1b[r] = take(H);
        L.n2[r] = take(H * H);
        L.n2b[r] = take(H);
    }
    L.dec1w = take(H * H);
    L.dec1b = take(H);
    L.dec2w = take(L.nout * H);
    L.dec2b = take(L.nout);
    L.total = o;
    return L;
}

// What differs from one training step to the next, read by its kernels from
// device memory so that the step's launches can be replayed: the targets and the
// update's step size and regulariser.
struct StepArgs {
    const double *x1, *u1, *rho1;
    float lr_t, eps_t;
};

struct Surrogate {
    int dim = 0, n = 0, npad = 0, sms = 0;
    Layout L;
    float k_ref = 1.f, t_jump = 0.f, sd_edge_u = 1.f, sd_edge_rho = 1.f;
    double t_jump64 = 0.0;       // the jump's time span (the device clock advances by it)
    std::vector<float> norm;     // mu_in, sd_in, mu_out, sd_out
    float *norm_d = nullptr;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    long long adam_t = 0;
    // packed BF16 weights: forward (B operands) and transposed (backward)
    bf16 *Wenc1, *Wenc2, *Wpq[2], *We2[2], *Wn1[2], *Wn2[2], *Wd1, *Wd2;
    bf16 *Wd2T, *Wd1T, *Wn2T[2], *Wn1T[2], *We2T[2], *WpqT[2], *Wenc2T;
    float *bpq[2], *bd2;
    // forward activations (rows: nodes in sorted order, padded to npad, zero beyond n)
    bf16 *X16, *A0, *A1[2], *S[2], *G1[2], *hLb, *A2;
    __half *PQ[2];               // [P | Q] node terms of the edge MLP's first layer, FP16
    __half *PQf = nullptr;       // the same with the state-difference channels folded in (forward)
    float *Z0, *h[3], *degs, *Z1[2], *Z2, *Y;
    float4 *NF;                  // per node: u / sd_edge_u (xyz), density deviation / sd_edge_rho
    // backward; a layer's weight and bias gradients are taken beside the chain of data
    // gradients (side streams), so what they read has a buffer per layer
    float *dYf, *dZf[4], *dA[2], *dh[3], *dS = nullptr;
    bf16 *dYb, *dZb[4], *dAb[2], *dhb[3], *dPQ[2];
    cudaStream_t side[2] = {nullptr, nullptr};   // weight gradients, bias gradients
    std::vector<cudaEvent_t> fork;               // one a layer
    cudaEvent_t join[2] = {nullptr, nullptr};
    double *sums;                // FP64 sums over blocks: dW3 and db1 of both rounds, layer biases
    double *loss_d = nullptr;
    double *loss_h = nullptr;    // pinned: where the loss and the gradient are read back
    float *grad_h = nullptr;
    StepArgs *args = nullptr, *args_h = nullptr;   // of the current training step (device, pinned)
    // a training step's launches as a graph, without and with the update (from the second call on)
    cudaGraphExec_t step_graph[2] = {nullptr, nullptr};
    int64_t step_calls[2] = {0, 0};

    void drop_graphs()
    {
        for (cudaGraphExec_t &g : step_graph) {
            if (g) cudaGraphExecDestroy(g);
            g = nullptr;
        }
        step_calls[0] = step_calls[1] = 0;
    }
    unsigned *err = nullptr;
    // judge snapshots (original order)
    double *sx = nullptr, *su = nullptr, *sr = nullptr;
    double *vx = nullptr, *vu = nullptr, *vr = nullptr;   // last verified state
    // judge: oil occupancy bitmaps of the jump and of the plain steps, the
    // interface tolerance (0: not used to reject) and the last run's maxima
    unsigned *occ_a = nullptr, *occ_b = nullptr;
    double itol = 0.0, max_cerr = 0.0, max_ierr = 0.0;
    std::vector<void *> allocs;

    ~Surrogate()
    {
        for (cudaStream_t t : side)
            if (t) cudaStreamSynchronize(t);
        for (void *p : allocs) cudaFree(p);
        if (loss_h) cudaFreeHost(loss_h);
        drop_graphs();
        for (cudaEvent_t e : fork)
            if (e) cudaEventDestroy(e);
        for (cudaEvent_t e : join)
            if (e) cudaEventDestroy(e);
        for (cudaStream_t t : side)
            if (t) cudaStreamDestroy(t);
    }
};

void free_surrogate(void *p) { delete static_cast<Surrogate *>(p); }

template <class T>
int dalloc(Surrogate &S, T **p, size_t count)
{
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) return set_error(SPH_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    S.allocs.push_back(q);
    cudaMemset(q, 0, std::max<size_t>(count, 1) * sizeof(T));
    *p = static_cast<T *>(q);
    return SPH_OK;
}

// ---------------------------------------------------------------------------
// Kernels

// The weights as the contractions read them, one launch for all tensors
// (27 launches of 3 us each before): job y copies W (rows x cols of theta at
// off) to BF16 dst[(row_off + r) * ld + c], transposed dst[c * ld + row_off +
// r], or (FP32 vectors, biases) dstf[c].
struct PackJob {
    bf16 *dst;
    float *dstf;
    int off, rows, cols, ld, row_off, transpose;
};
constexpr int PACK_JOBS = 3 + 2 * 11 + 4 + 1;
struct PackTable {
    PackJob job[PACK_JOBS];
};

__global__ void k_pack(const float *theta, const __grid_constant__ PackTable t)
{
    const PackJob &p = t.job[blockIdx.y];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= p.rows * p.cols) return;
    const int r = k / p.cols, c = k % p.cols;
    const float w = theta[p.off + k];
    if (p.dstf) {
        p.dstf[k] = w;
        return;
    }
    const bf16 v = __float2bfloat16_rn(w);
    if (p.transpose) p.dst[(size_t)c * p.ld + p.row_off + r] = v;
    else p.dst[(size_t)(p.row_off + r) * p.ld + c] = v;
}

// Normalised node inputs [u, (rho - rho0)/rho0, oil, wall, T a,
// T (Drho/Dt)/rho0] (sorted order; the rates are those of the evaluation at
// the current state), and the per-node terms of the edge state differences.
template <int DIM>
__global__ void k_features(Dev d, const float *norm, float T, float inv_su, float inv_sr, bf16 *X, float4 *NF)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    constexpr int NIN = 2 * DIM + 4;
    const uint8_t tg = d.tag[k];
    const Inst &I = d.inst[d.iid[k]];
    const float inv_rho0 = by_phase(tg & 1, I.inv_rho0);
    const float4 a = d.acc[k];
    float raw[NIN];
#pragma unroll
    for (int c = 0; c < DIM; ++c) raw[c] = (float)d.u[(size_t)c * d.n + k];
    raw[DIM] = d.drho[k] * inv_rho0;
    raw[DIM + 1] = (float)(tg & 1);
    raw[DIM + 2] = (float)((tg >> 1) & 1);
    raw[DIM + 3] = T * a.x;
    raw[DIM + 4] = T * a.y;
    if (DIM == 3) raw[DIM + 5] = T * a.z;
    raw[2 * DIM + 3] = T * a.w * inv_rho0;
    __align__(16) bf16 out[FIN];
#pragma unroll
    for (int c = 0; c < FIN; ++c) out[c] = __float2bfloat16_rn(c < NIN ? (raw[c] - norm[c]) / norm[NIN + c] : 0.f);
#pragma unroll
    for (int c = 0; c < FIN; c += 8) *(uint4 *)(X + (size_t)k * FIN + c) = *(const uint4 *)(out + c);
    NF[k] = make_float4(raw[0] * inv_su, raw[1] * inv_su, DIM == 3 ? raw[2] * inv_su : 0.f, raw[DIM] * inv_sr);
}

// Edge features of the pair (i, j): r_ij / 2h (DIM), |r_ij| / 2h,
// phase_i != phase_j, (u_i - u_j) / sd_edge_u (DIM), density deviation
// difference / sd_edge_rho.
template <int DIM>
__device__ __forceinline__ bool edge_features(const Dev &d, const Grid &g, float R2, float inv2h, const float4 &oi,
                                              int phi, const float4 &nfi, const float4 *NF, unsigned e, int &j,
                                              float (&ef)[2 * DIM + 3])
{
    j = (int)(e & NBR_IDX_MASK);
    if (!SPH_IN_RANGE(d.flags, j, d.n)) return false;
    const float4 oj = d.pos[j];
    float rx, ry, rz;
    const float r2 = pair_vec<DIM>(oi, oj, entry_shift(e, 0, g.Es), entry_shift(e, 1, g.Es),
                                   DIM == 3 ? entry_shift(e, 2, g.Es) : 0.f, rx, ry, rz);
    if (!(r2 < R2)) return false;
    ef[0] = rx * inv2h;
    ef[1] = ry * inv2h;
    if (DIM == 3) ef[2] = rz * inv2h;
    ef[DIM] = sqrtf(r2) * inv2h;
    ef[DIM + 1] = rec_phase(oj.w) != phi ? 1.f : 0.f;
    const float4 nfj = NF[j];
    ef[DIM + 2] = nfi.x - nfj.x;
    ef[DIM + 3] = nfi.y - nfj.y;
    if (DIM == 3) ef[DIM + 4] = nfi.z - nfj.z;
    ef[2 * DIM + 2] = nfi.w - nfj.w;
    return true;
}

// The pair-only part of the edge features: r_ij / 2h (DIM), |r_ij| / 2h,
// phase_i != phase_j.  The state-difference channels of edge_features are
// linear in node quantities, so the forward pass folds them into the node
// terms (the epilogue of the P, Q layer: with f_i the node's scaled (u, delta)
// channels and W3d their columns of W3, W3d (f_i - f_j) = W3d f_i - W3d f_j, so
// P'_i = P_i + W3d f_i and Q'_j = Q_j - W3d f_j give the same pre-activation
// P'_i + Q'_j + W3g e_ij) and the edge phase needs only these.
template <int DIM>
__device__ __forceinline__ bool edge_geom(const Dev &d, const Grid &g, float R2, float inv2h, const float4 &oi,
                                          int phi, unsigned e, int &j, float (&ef)[DIM + 2])
{
    j = (int)(e & NBR_IDX_MASK);
    if (!SPH_IN_RANGE(d.flags, j, d.n)) return false;
    const float4 oj = d.pos[j];
    float rx, ry, rz;
    const float r2 = pair_vec<DIM>(oi, oj, entry_shift(e, 0, g.Es), entry_shift(e, 1, g.Es),
                                   DIM == 3 ? entry_shift(e, 2, g.Es) : 0.f, rx, ry, rz);
    if (!(r2 < R2)) return false;
    ef[0] = rx * inv2h;
    ef[1] = ry * inv2h;
    if (DIM == 3) ef[2] = rz * inv2h;
    ef[DIM] = sqrtf(r2) * inv2h;
    ef[DIM + 1] = rec_phase(oj.w) != phi ? 1.f : 0.f;
    return true;
}

__device__ __forceinline__ void store4(bf16 *p, const float (&v)[4])
{
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    uint2 raw;
    raw.x = *(const unsigned *)&a;
    raw.y = *(const unsigned *)&b;
    *(uint2 *)p = raw;
}


__device__ __forceinline__ __half2 tanh_h2(__half2 x)
{
    uint32_t r;
    asm("tanh.approx.f16x2 %0, %1;" : "=r"(r) : "r"(*(const uint32_t *)&x));
    return *(const __half2 *)&r;
}

// Forward edge phase: half a warp per receiver i, eight features per lane.
// S_i = (1/k_ref) sum_j SiLU(P'_i + Q'_j + W3g e_ij) over list entries with
// |r_ij| < 2h (the folded node terms and the pair features); degs_i = deg_i /
// k_ref.  The pre-activation and SiLU run on feature pairs in FP16 (packed FMA,
// and SiLU(z) = h + h tanh(h) with h = z/2); the sum of each 32 list entries is
// added to an FP32 accumulator.
//
// Bound by instruction issue and the tanh unit (DRAM a few per cent): per edge
// and 64 feature pairs, 10 packed operations a pair.  What is done per edge and
// not per feature (the slot and sender-row reads, addresses, the loop) is
// shared by a warp's two receivers and its eight features a lane: 58 warp
// instructions an edge with a warp per receiver and four features a lane, about
// 28 so.  The two receivers' next 32 entries are decoded lane-parallel (their
// list columns are adjacent words) into 16-byte slots, the valid ones
// compacted in list order: the pair features and a mask in FP16 (packed
// arithmetic takes either half of a register as both) and the sender.  The
// shorter of the two is padded with its last valid slot at mask 0 (a term that
// is finite whenever the sum is), so the warp runs one uniform loop; sender rows
// come straight from L1/L2, EDGE_U edges' loads issued before the first is
// used.  Blocks are persistent: W3 stays in registers.
// 656 600 particles, one round (GB300, profiler): 3.60 -> 2.40 ms; on 193 496,
// 1.05 -> 0.69 ms with 463 M warp instructions instead of 762 M, the FP16 half of
// the FMA pipe 65 % busy.  Five blocks an SM (96 registers) and four edges in
// flight measured best (jump 6.7 ms; six blocks 7.5, eight 7.3, eight edges 6.8).
constexpr int EDGE_U = 4, EDGE_BLOCKS = 5;
constexpr int EWF = 128;   // threads of the forward edge kernel (4 warps, two receivers each)

template <int DIM>
__global__ void __launch_bounds__(EWF, EDGE_BLOCKS)
    k_edge_fwd(Dev d, Grid g, float R2, float inv2h, const __half *__restrict__ PQ, const float *W3, float inv_kref,
               bf16 *S, float *degs)
{
    constexpr int NE = 2 * DIM + 3;   // columns of W3 (the pair features are its first NG)
    constexpr int NG = DIM + 2;
    constexpr int U = EDGE_U;
    constexpr int CAP = (32 + U - 1) / U * U;
    __shared__ __align__(16) uint4 slots[EWF / 32][2][CAP];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = lane >> 4, f0 = (lane & 15) * 8;
    __half2 w2[NG][4];   // W3 column c for the features (f0, f0 + 1), ...
#pragma unroll
    for (int c = 0; c < NG; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            w2[c][q] = __floats2half2_rn(W3[(f0 + 2 * q) * NE + c], W3[(f0 + 2 * q + 1) * NE + c]);
    const __half2 half2c = __float2half2_rn(0.5f);
    uint4(*const slot)[CAP] = slots[wid];
    const uint4 *const mine = slot[half];
    const __half *const Q = PQ + H + f0;
    const int n = d.n;
    const int stride = gridDim.x * (EWF / 32) * 2;
    for (int base = (blockIdx.x * (EWF / 32) + wid) * 2; base < n; base += stride) {
        // decoding: lane l takes receiver base + (l & 1) and entry l >> 1 of 16
        const int di = min(base + (lane & 1), n - 1);
        const float4 oi = d.pos[di];
        const int phi = rec_phase(oi.w);
        const int dcnt = base + (lane & 1) < n ? d.ncnt[di] : 0;
        const int most = max(dcnt, __shfl_xor_sync(0xffffffffu, dcnt, 1));
        // summing: this half's receiver
        const int i = min(base + half, n - 1);
        const uint4 praw = *(const uint4 *)(PQ + (size_t)i * 2 * H + f0);
        const __half2 P[4] = {*(const __half2 *)&praw.x, *(const __half2 *)&praw.y, *(const __half2 *)&praw.z,
                              *(const __half2 *)&praw.w};
        float acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = 0.f;
        int deg = 0;
        for (int k0 = 0; k0 < most; k0 += 32) {
            int have0 = 0, have1 = 0;
            __syncwarp();
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
                const int k = k0 + pass * 16 + (lane >> 1);
                bool valid = false;
                int j = 0;
                float ef[NG];
                if (k < dcnt)
                    valid = edge_geom<DIM>(d, g, R2, inv2h, oi, phi, d.nbr[(size_t)k * n + di], j, ef);
                const unsigned m = __ballot_sync(0xffffffffu, valid);
                if (valid) {
                    const unsigned own = m & (0x55555555u << (lane & 1));
                    const __half2 a = __floats2half2_rn(ef[0], ef[1]), b = __floats2half2_rn(ef[2], ef[3]);
                    const __half2 c = __floats2half2_rn(ef[NG - 1], 1.f);   // (2-D: the first half is not used)
                    slot[lane & 1][((lane & 1) ? have1 : have0) + __popc(own & ((1u << lane) - 1u))] =
                        make_uint4(*(const uint32_t *)&a, *(const uint32_t *)&b, *(const uint32_t *)&c, (uint32_t)j);
                }
                have0 += __popc(m & 0x55555555u);
                have1 += __popc(m & 0xaaaaaaaau);
            }
            __syncwarp();
            const int cnt = half ? have1 : have0;
            const int full = (max(have0, have1) + U - 1) / U * U;
            // padding: the last valid slot (or, with none, the receiver itself) at mask 0
            if (cnt < full) {
                uint4 pad = make_uint4(0u, 0u, 0u, (uint32_t)i);
                if (cnt > 0) {
                    pad = mine[cnt - 1];
                    pad.z &= 0xffffu;
                }
                for (int q = cnt + (lane & 15); q < full; q += 16) slot[half][q] = pad;
            }
            __syncwarp();
            deg += cnt;
            __half2 s[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = __float2half2_rn(0.f);
            for (int e0 = 0; e0 < full; e0 += U) {
                uint4 sl[U], row[U];
#pragma unroll
                for (int t = 0; t < U; ++t) sl[t] = mine[e0 + t];
#pragma unroll
                for (int t = 0; t < U; ++t) row[t] = *(const uint4 *)(Q + (size_t)sl[t].w * (2 * H));
#pragma unroll
                for (int t = 0; t < U; ++t) {
                    const __half2 q2[4] = {*(const __half2 *)&row[t].x, *(const __half2 *)&row[t].y,
                                           *(const __half2 *)&row[t].z, *(const __half2 *)&row[t].w};
                    const __half2 eab = *(const __half2 *)&sl[t].x, ecd = *(const __half2 *)&sl[t].y;
                    const __half2 eem = *(const __half2 *)&sl[t].z;
                    const __half2 ec[5] = {__low2half2(eab), __high2half2(eab), __low2half2(ecd), __high2half2(ecd),
                                           __low2half2(eem)};
                    const __half2 mask = __high2half2(eem);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        __half2 z = __hadd2(P[q], q2[q]);
#pragma unroll
                        for (int c = 0; c < NG; ++c) z = __hfma2(w2[c][q], ec[c], z);
                        const __half2 h = __hmul2(z, half2c);
                        // mask 1: the rounded sum s + x; mask 0: s
                        s[q] = __hfma2(__hfma2(h, tanh_h2(h), h), mask, s[q]);
                    }
                }
            }
            if (cnt > 0)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 a = __half22float2(s[q]);
                    acc[2 * q] += a.x;
                    acc[2 * q + 1] += a.y;
                }
        }
        if (base + half < n) {
            uint4 o;
            uint32_t ow[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const __nv_bfloat162 v = __floats2bfloat162_rn(acc[2 * q] * inv_kref, acc[2 * q + 1] * inv_kref);
                ow[q] = *(const uint32_t *)&v;
            }
            o = make_uint4(ow[0], ow[1], ow[2], ow[3]);
            *(uint4 *)(S + (size_t)i * H + f0) = o;
            if ((lane & 15) == 0) degs[i] = deg * inv_kref;
        }
    }
}

// Two FP32 values in one 64-bit register, and the packed arithmetic on them
// (each half rounds like the scalar operation).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// SiLU'(z) of a pair, which may be held negated, with the fast reciprocal
// (relative error about 1e-6, far below the BF16 rounding of the network's
// operands).  Scalar but for the last product: packed sums here made the training
// step 5 % slower (the packed pipe is the busy one).
template <bool NEGATED>
__device__ __forceinline__ f32x2 dsilu2(f32x2 z)
{
    float a, b;
    unpack2(z, a, b);
    const float sa = __fdividef(1.f, 1.f + __expf(NEGATED ? a : -a)), sb = __fdividef(1.f, 1.f + __expf(NEGATED ? b : -b));
    const float ua = fmaf(NEGATED ? -a : a, 1.f - sa, 1.f), ub = fmaf(NEGATED ? -b : b, 1.f - sb, 1.f);
    return mul2(pack2(sa, sb), pack2(ua, ub));
}

// Two FP16 pairs (four features) as two FP32 pairs.
__device__ __forceinline__ void half4(uint2 raw, f32x2 (&v)[2])
{
    const float2 a = __half22float2(*(const __half2 *)&raw.x), b = __half22float2(*(const __half2 *)&raw.y);
    v[0] = pack2(a.x, a.y);
    v[1] = pack2(b.x, b.y);
}

// Backward edge phase: one warp per node i, four features (two FP32 pairs) a
// lane.  With dZ_ij = dS_i SiLU'(z_ij) / k_ref: dP_i = sum_j dZ_ij, dQ_i = sum_j
// dZ_ji (the neighbour relation is symmetric, so node i gathers its own sender
// terms), dW3 += dZ_ij e_ij and db1 += dP_i.
//
// Bound by the FP32 pipe and, with the few warps its registers allow, by latency:
// per edge and feature two nine-term dot products, two SiLU' and a nine-term
// outer product, in FP32.  The arithmetic is on packed pairs (half the
// instructions; z_ji is summed negated, so that the channels that change sign
// with the direction use the same pair features); two edges at a time share
// each read of W3 from shared memory (four wavefronts a channel) and the next
// two's rows are on their way meanwhile; the edge features lie in the slots as
// pairs (e, e).  Blocks are persistent: the weight gradient stays in registers over
// all nodes of a warp and is reduced over the block once (once per eight nodes
// before: 160 atomics a node on 1 280 addresses); the blocks' sums meet in FP64
// (w3_sum: dW3 then db1, zeroed before), which k_sums_out rounds into the gradient.
// Measured (GB300): a training step on 193 496 particles 13.76 -> 12.51 ms (two
// launches of 4.86 ms with scalar arithmetic and a block reduction per eight
// nodes).  Not kept: three blocks of 128 (12 warps instead of 8, 168 registers:
// the same), two features a lane (half the registers, two or three times the
// warps, but the per-edge work shared by half as many features: 3 to 19 %
// longer), the dot or the outer products scalar (2 to 8 % longer).
constexpr int EWB = 256;     // threads (8 warps, one node each at a time)
constexpr int EWB_BLOCKS = 1;

// Slots of the backward edge phase: the 2 DIM + 3 features twice each, then
// the sender, padded to whole 16-byte vectors.
template <int DIM>
__host__ __device__ constexpr int bwd_slot_width() { return (2 * (2 * DIM + 3) + 1 + 3) / 4 * 4; }

// What an edge reads of its sender: P_j, Q_j and dS_j (four features).
struct SenderRow {
    uint2 p, q;
    ulonglong2 s;
};

template <int DIM>
__global__ void __launch_bounds__(EWB, EWB_BLOCKS)
    k_edge_bwd(Dev d, Grid g, float R2, float inv2h, const float4 *NF, const __half *__restrict__ PQ, const float *W3,
               float inv_kref, const float *__restrict__ dS, bf16 *dPQ, double *w3_sum)
{
    constexpr int NE = 2 * DIM + 3;
    constexpr int SWD = bwd_slot_width<DIM>();
    constexpr int WARPS = EWB / 32;
    __shared__ __align__(16) float slots[WARPS][32][SWD];
    __shared__ __align__(16) float4 sw[NE][32];
    __shared__ float red[H * (NE + 1)];
    for (int t = threadIdx.x; t < NE * 32; t += EWB) {
        const int c = t / 32, l = t % 32;
        sw[c][l] = make_float4(W3[(4 * l) * NE + c], W3[(4 * l + 1) * NE + c], W3[(4 * l + 2) * NE + c],
                               W3[(4 * l + 3) * NE + c]);
    }
    for (int t = threadIdx.x; t < H * (NE + 1); t += EWB) red[t] = 0.f;
    __syncthreads();
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, f0 = lane * 4;
    const int n = d.n;
    float(*const slot)[SWD] = slots[wid];
    const f32x2 ik2 = pack2(inv_kref, inv_kref), minus = pack2(-1.f, -1.f);
    f32x2 gw[NE][2], gb[2] = {0ull, 0ull};
#pragma unroll
    for (int c = 0; c < NE; ++c) gw[c][0] = gw[c][1] = 0ull;
    for (int i = blockIdx.x * WARPS + wid; i < n; i += gridDim.x * WARPS) {
        f32x2 Pi[2], Qn[2], dSi[2], dP[2] = {0ull, 0ull}, dQ[2] = {0ull, 0ull};
        half4(*(const uint2 *)(PQ + (size_t)i * 2 * H + f0), Pi);
        half4(*(const uint2 *)(PQ + (size_t)i * 2 * H + H + f0), Qn);
#pragma unroll
        for (int q = 0; q < 2; ++q) Qn[q] = mul2(Qn[q], minus);
        {
            const ulonglong2 t = *(const ulonglong2 *)(dS + (size_t)i * H + f0);
            dSi[0] = mul2(t.x, ik2);
            dSi[1] = mul2(t.y, ik2);
        }
        const float4 oi = d.pos[i];
        const float4 nfi = NF[i];
        const int phi = rec_phase(oi.w);
        const int cnt = d.ncnt[i];
        auto fetch = [&](int e) {
            const size_t j = (size_t)__float_as_int(slot[e][2 * NE]);
            SenderRow r;
            r.p = *(const uint2 *)(PQ + j * 2 * H + f0);
            r.q = *(const uint2 *)(PQ + j * 2 * H + H + f0);
            r.s = *(const ulonglong2 *)(dS + j * H + f0);
            return r;
        };
        // M edges of the batch from slot e on, their rows given
        auto edges = [&](int e, const SenderRow *row, auto count) {
            constexpr int M = decltype(count)::value;
            f32x2 zi[M][2], zj[M][2];   // z_ij, -z_ji
#pragma unroll
            for (int t = 0; t < M; ++t) {
                f32x2 Pj[2], Qj[2];
                half4(row[t].p, Pj);
                half4(row[t].q, Qj);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    zi[t][q] = add2(Pi[q], Qj[q]);
                    zj[t][q] = fma2(Pj[q], minus, Qn[q]);
                }
            }
#pragma unroll
            for (int c = 0; c < NE; ++c) {
                const ulonglong2 w = *(const ulonglong2 *)&sw[c][lane];
#pragma unroll
                for (int t = 0; t < M; ++t) {
                    const f32x2 ec = *(const f32x2 *)&slot[e + t][2 * c];
                    // e_ji: the relative position and the state differences change
                    // sign, the distance and the phase flag do not
                    const f32x2 en = c < DIM || c >= DIM + 2 ? ec : mul2(ec, minus);
                    zi[t][0] = fma2(w.x, ec, zi[t][0]);
                    zi[t][1] = fma2(w.y, ec, zi[t][1]);
                    zj[t][0] = fma2(w.x, en, zj[t][0]);
                    zj[t][1] = fma2(w.y, en, zj[t][1]);
                }
            }
#pragma unroll
            for (int t = 0; t < M; ++t) {
                f32x2 di[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    di[q] = mul2(dSi[q], dsilu2<false>(zi[t][q]));
                    dP[q] = add2(dP[q], di[q]);
                    dQ[q] = fma2(mul2(q ? row[t].s.y : row[t].s.x, ik2), dsilu2<true>(zj[t][q]), dQ[q]);
                }
#pragma unroll
                for (int c = 0; c < NE; ++c) {
                    const f32x2 ec = *(const f32x2 *)&slot[e + t][2 * c];
                    gw[c][0] = fma2(di[0], ec, gw[c][0]);
                    gw[c][1] = fma2(di[1], ec, gw[c][1]);
                }
            }
        };
        for (int k0 = 0; k0 < cnt; k0 += 32) {
            // decoding: the valid ones of 32 entries to the slots, in list order
            __syncwarp();
            int j = 0;
            float ef[NE];
            bool valid = false;
            if (k0 + lane < cnt)
                valid = edge_features<DIM>(d, g, R2, inv2h, oi, phi, nfi, NF, d.nbr[(size_t)(k0 + lane) * n + i], j, ef);
            const unsigned m = __ballot_sync(0xffffffffu, valid);
            if (valid) {
                float *const s = slot[__popc(m & ((1u << lane) - 1u))];
#pragma unroll
                for (int c = 0; c < NE; ++c) *(f32x2 *)(s + 2 * c) = pack2(ef[c], ef[c]);
                s[2 * NE] = __int_as_float(j);
            }
            __syncwarp();
            const int have = __popc(m);
            if (have == 0) continue;
            SenderRow row[2] = {fetch(0), fetch(min(1, have - 1))};
            int e = 0;
            for (; e + 2 <= have; e += 2) {
                const SenderRow next[2] = {fetch(min(e + 2, have - 1)), fetch(min(e + 3, have - 1))};
                edges(e, row, std::integral_constant<int, 2>());
                row[0] = next[0];
                row[1] = next[1];
            }
            if (e < have) edges(e, row, std::integral_constant<int, 1>());
        }
        float p[4], q[4];
        unpack2(dP[0], p[0], p[1]);
        unpack2(dP[1], p[2], p[3]);
        unpack2(dQ[0], q[0], q[1]);
        unpack2(dQ[1], q[2], q[3]);
        store4(dPQ + (size_t)i * 2 * H + f0, p);
        store4(dPQ + (size_t)i * 2 * H + H + f0, q);
        gb[0] = add2(gb[0], dP[0]);
        gb[1] = add2(gb[1], dP[1]);
    }
    // block sums of dW3 and db1, warp after warp
    for (int w = 0; w < WARPS; ++w) {
        if (wid == w) {
            float v[4];
#pragma unroll
            for (int c = 0; c < NE; ++c) {
                unpack2(gw[c][0], v[0], v[1]);
                unpack2(gw[c][1], v[2], v[3]);
#pragma unroll
                for (int q = 0; q < 4; ++q) red[(f0 + q) * NE + c] += v[q];
            }
            unpack2(gb[0], v[0], v[1]);
            unpack2(gb[1], v[2], v[3]);
#pragma unroll
            for (int q = 0; q < 4; ++q) red[H * NE + f0 + q] += v[q];
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < H * (NE + 1); t += EWB) {
        const float s = red[t];
        if (s != 0.f) atomicAdd(w3_sum + t, (double)s);
    }
}

// The FP64 sums (edge weights and biases, biases of the layers) into the gradient.
struct SumTable {
    int count, from[14], to[14], len[14];
};
__global__ void k_sums_out(const double *sum, float *grad, const __grid_constant__ SumTable t)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (k < t.len[j]) grad[t.to[j] + k] = (float)sum[t.from[j] + k];
}

// Column sums over n rows of src (ld), optionally weighted per row, added to
// dst: a thread per column and block of rows; the blocks' FP32 sums meet in FP64
// (atomics), so the order they finish in shows in the last bits of an FP64 sum only,
// and after the rounding to FP32 in one unit of the last place at most.
__global__ void k_colsum(const float *src, int ld, int cols, int n, const float *roww, double *dst)
{
    const int c = threadIdx.x;
    const int rows_per = (n + gridDim.x - 1) / gridDim.x;
    const int r0 = blockIdx.x * rows_per, r1 = min(n, r0 + rows_per);
    if (c >= cols) return;
    float s = 0.f;
    for (int r = r0; r < r1; ++r) s += (roww ? roww[r] : 1.f) * src[(size_t)r * ld + c];
    if (s != 0.f) atomicAdd(dst + c, (double)s);
}

// Targets from the state after k plain steps (original order, instance
// frame) against the current state (sorted), masked squared error, dL/dy.
template <int DIM>
__global__ void k_loss(Dev d, const float *norm, float T, const float *Y, const StepArgs *args, float inv_count,
                       float *dYf, bf16 *dYb, double *loss)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const double *const x1 = args->x1, *const u1 = args->u1, *const rho1 = args->rho1;
    double l = 0.0;
    if (k < d.n) {
        constexpr int NIN = 2 * DIM + 4, NOUT = 2 * DIM + 1;
        const float *mu_out = norm + 2 * NIN, *sd_out = norm + 2 * NIN + NOUT;
        const int p = d.pid[k];
        const uint8_t tg = d.tag[k];
        const Inst &I = d.inst[d.iid[k]];
        const bool wall = tg & 2;
        const float4 a = d.acc[k];
        const float av[3] = {a.x, a.y, a.z};
        float delta[NOUT];
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            const double u0c = d.u[(size_t)c * d.n + k], u1c = u1[(size_t)p * DIM + c];
            const double dxc = x1[(size_t)p * DIM + c] - (d.x[(size_t)c * d.n + k] - I.offset[c]);
            delta[c] = (float)(dxc - (double)T * 0.5 * (u0c + u1c));
            delta[DIM + c] = (float)(u1c - u0c - (double)T * av[c]);
        }
        const double rho0 = (double)by_phase(tg & 1, I.rho0);
        delta[2 * DIM] = (float)((rho1[p] - (rho0 + (double)d.drho[k])) / rho0 - (double)T * a.w / rho0);
        float dy[FOUT];
#pragma unroll
        for (int c = 0; c < FOUT; ++c) dy[c] = 0.f;
#pragma unroll
        for (int c = 0; c < NOUT; ++c) {
            if (wall && c < 2 * DIM) continue;
            const float t = (delta[c] - mu_out[c]) / sd_out[c];
            const float e = Y[(size_t)k * FOUT + c] - t;
            l += (double)e * e;
            dy[c] = 2.f * e * inv_count;
        }
#pragma unroll
        for (int c = 0; c < FOUT; ++c) {
            dYf[(size_t)k * FOUT + c] = dy[c];
            dYb[(size_t)k * FOUT + c] = __float2bfloat16_rn(dy[c]);
        }
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0 && l != 0.0) atomicAdd(loss, l);
}

// Applies the de-normalised increments: x += dx, u += du on fluid particles,
// rho += drho on all; nothing when the list build behind them gave up (stopped).
template <int DIM>
__global__ void k_apply(Dev d, const float *norm, float T, const float *Y)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n || stopped(d)) return;
    constexpr int NIN = 2 * DIM + 4, NOUT = 2 * DIM + 1;
    const float *mu_out = norm + 2 * NIN, *sd_out = norm + 2 * NIN + NOUT;
    const uint8_t tg = d.tag[k];
    const Inst &I = d.inst[d.iid[k]];
    const float4 a = d.acc[k];
    const float av[3] = {a.x, a.y, a.z};
    float D[NOUT];
#pragma unroll
    for (int c = 0; c < NOUT; ++c) D[c] = Y[(size_t)k * FOUT + c] * sd_out[c] + mu_out[c];
    bool finite = true;
    if (!(tg & 2)) {
#pragma unroll
        for (int c = 0; c < DIM; ++c) {
            const double u0 = d.u[(size_t)c * d.n + k], du = (double)T * av[c] + (double)D[DIM + c];
            const double x = d.x[(size_t)c * d.n + k] + ((double)T * (u0 + 0.5 * du) + (double)D[c]);
            const double u = u0 + du;
            d.x[(size_t)c * d.n + k] = x;
            d.u[(size_t)c * d.n + k] = u;
            finite = finite && isfinite(x) && isfinite(u);
        }
    }
    const float dr = d.drho[k] + (T * a.w + D[2 * DIM] * by_phase(tg & 1, I.rho0));
    d.drho[k] = dr;
    if (!finite || !isfinite(dr)) atomicOr(d.flags, FLAG_NONFINITE);
}

// De-normalised increments in original order: out[p * NOUT + c].
template <int DIM>
__global__ void k_predict_out(Dev d, const float *norm, float T, const float *Y, double *out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.n) return;
    constexpr int NIN = 2 * DIM + 4, NOUT = 2 * DIM + 1;
    const float *mu_out = norm + 2 * NIN, *sd_out = norm + 2 * NIN + NOUT;
    const int p = d.pid[k];
    const uint8_t tg = d.tag[k];
    const Inst &I = d.inst[d.iid[k]];
    const float4 a = d.acc[k];
    const float av[3] = {a.x, a.y, a.z};
    float D[NOUT];
#pragma unroll
    for (int c = 0; c < NOUT; ++c) D[c] = Y[(size_t)k * FOUT + c] * sd_out[c] + mu_out[c];
#pragma unroll
    for (int c = 0; c < DIM; ++c) {
        const double u0 = d.u[(size_t)c * d.n + k], du = (double)T * av[c] + (double)D[DIM + c];
        out[(size_t)p * NOUT + c] = (tg & 2) ? 0.0 : (double)T * (u0 + 0.5 * du) + (double)D[c];
        out[(size_t)p * NOUT + DIM + c] = (tg & 2) ? 0.0 : du;
    }
    out[(size_t)p * NOUT + 2 * DIM] = (double)(T * a.w + D[2 * DIM] * by_phase(tg & 1, I.rho0));
}

// Adam (Kingma & Ba 2015) with bias correction folded into the step size; the weights
// stay when the list build behind the gradient gave up (stopped).
__global__ void k_adam(Dev d, float *theta, const float *g, float *m, float *v, int count, const StepArgs *args,
                       float b1, float b2)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= count || stopped(d)) return;
    const float lr_t = args->lr_t, eps_t = args->eps_t;
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.f - b1) * gk;
    const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    theta[k] -= lr_t * mk / (sqrtf(vk) + eps_t);
}

// ---------------------------------------------------------------------------
// Host side

inline int nb(int work, int t = 256) { return (work + t - 1) / t; }

struct Epi {
    float *Cf = nullptr;
    int ldcf = 0;
    bf16 *Cb = nullptr;
    int ldcb = 0;
    const float *bias = nullptr;
    const float *row_scale = nullptr, *row_bias = nullptr;
    float *Z = nullptr;
    int ldz = 0;
    const float *residual = nullptr;
    int ldr = 0;
    const float *residual2 = nullptr;
    int ldr2 = 0;
    int act = 0;
    const float *dact = nullptr;
    int lddact = 0;
    // the P, Q layer: folded node terms (see umma::GemmArgs)
    const float4 *fold_f = nullptr;
    const float *fold_w = nullptr;
    int dim = 0;
    __half *fold_out = nullptr;
};

int mm(Surrogate &S, cudaStream_t st, const bf16 *A, int lda, const bf16 *B, int ldb, int M, int N, int K,
       const Epi &e)
{
    umma::GemmArgs g{};
    g.A = A;
    g.lda = lda;
    g.B = B;
    g.ldb = ldb;
    g.M = M;
    g.N = N;
    g.K = K;
    g.k_split = ((K + umma::BK - 1) / umma::BK) * umma::BK;
    g.Cf = e.Cf;
    g.ldcf = e.ldcf;
    g.Cb = e.Cb;
    g.ldcb = e.ldcb;
    g.bias = e.bias;
    g.row_scale = e.row_scale;
    g.row_bias = e.row_bias;
    g.Z = e.Z;
    g.ldz = e.ldz;
    g.residual = e.residual;
    g.ldr = e.ldr;
    g.residual2 = e.residual2;
    g.ldr2 = e.ldr2;
    g.act = e.act;
    g.dact = e.dact;
    g.lddact = e.lddact;
    g.err = S.err;
    if (e.fold_out) {
        g.fold_f = e.fold_f;
        g.fold_w = e.fold_w;
        g.fold_ldw = 2 * e.dim + 3;
        g.fold_v = e.dim + 2;
        g.fold_s = 2 * e.dim + 2;
        g.fold_dim = e.dim;
        g.fold_out = e.fold_out;
        g.fold_ld = N;
    }
    // every layer of the network is k_layer's, which alone has its epilogues
    const umma::LayerLaunch launch = umma::layer_for(g);
    cudaError_t err = launch ? launch(g, st) : cudaErrorInvalidValue;
    if (err != cudaSuccess) return set_error(SPH_ECUDA, std::string("gemm: ") + cudaGetErrorString(err));
    return SPH_OK;
}

// dW (rows x cols, ld cols, in the flat gradient) += dY^T X over the nodes: dY with fy
// features (the first `rows` of them, or with dW2 both halves of 256), X with fx.  4096
// nodes a block.
int wgrad(Surrogate &S, cudaStream_t st, const bf16 *dY, int ldy, int fy, const bf16 *X, int ldx, int fx, float *dW,
          int rows, int cols, float *dW2 = nullptr)
{
    cudaError_t err = umma::wgrad(dY, ldy, fy, X, ldx, fx, S.n, dW, dW2, cols, rows, cols, 4096, S.err, st);
    if (err != cudaSuccess) return set_error(SPH_ECUDA, std::string("wgrad: ") + cudaGetErrorString(err));
    return SPH_OK;
}

int pack_weights(Surrogate &S, cudaStream_t st)
{
    const Layout &L = S.L;
    PackTable t{};
    int jobs = 0, most = 0;
    auto pk = [&](int off, int rows, int cols, bf16 *dst, int ld, int row_off, int tr) {
        t.job[jobs++] = {dst, nullptr, off, rows, cols, ld, row_off, tr};
        most = std::max(most, rows * cols);
    };
    auto copy = [&](int off, int count, float *dst) { t.job[jobs++] = {nullptr, dst, off, 1, count, 0, 0, 0}; };
    pk(L.enc1w, H, L.nin, S.Wenc1, FIN, 0, 0);
    pk(L.enc2w, H, H, S.Wenc2, H, 0, 0);
    pk(L.enc2w, H, H, S.Wenc2T, H, 0, 1);
    for (int r = 0; r < 2; ++r) {
        pk(L.w1[r], H, H, S.Wpq[r], H, 0, 0);
        pk(L.w2[r], H, H, S.Wpq[r], H, H, 0);
        pk(L.w1[r], H, H, S.WpqT[r], 2 * H, 0, 1);
        pk(L.w2[r], H, H, S.WpqT[r], 2 * H, H, 1);
        pk(L.we2[r], H, H, S.We2[r], H, 0, 0);
        pk(L.we2[r], H, H, S.We2T[r], H, 0, 1);
        pk(L.n1[r], H, 2 * H, S.Wn1[r], 2 * H, 0, 0);
        pk(L.n1[r], H, 2 * H, S.Wn1T[r], H, 0, 1);
        pk(L.n2[r], H, H, S.Wn2[r], H, 0, 0);
        pk(L.n2[r], H, H, S.Wn2T[r], H, 0, 1);
        copy(L.b1[r], H, S.bpq[r]);
    }
    pk(L.dec1w, H, H, S.Wd1, H, 0, 0);
    pk(L.dec1w, H, H, S.Wd1T, H, 0, 1);
    pk(L.dec2w, L.nout, H, S.Wd2, H, 0, 0);
    pk(L.dec2w, L.nout, H, S.Wd2T, FOUT, 0, 1);
    copy(L.dec2b, L.nout, S.bd2);
    k_pack<<<dim3(nb(most), jobs), 256, 0, st>>>(S.theta, t);
    CUR(cudaGetLastError());
    return SPH_OK;
}

int alloc_surrogate(Surrogate &S)
{
    const size_t P = (size_t)S.npad;
    const size_t nt = (size_t)S.L.total;
    int e = 0;
    e |= dalloc(S, &S.theta, nt);
    e |= dalloc(S, &S.grad, nt);
    e |= dalloc(S, &S.m, nt);
    e |= dalloc(S, &S.v, nt);
    e |= dalloc(S, &S.norm_d, 64);
    e |= dalloc(S, &S.Wenc1, H * FIN);
    e |= dalloc(S, &S.Wenc2, H * H);
    e |= dalloc(S, &S.Wenc2T, H * H);
    for (int r = 0; r < 2; ++r) {
        e |= dalloc(S, &S.Wpq[r], 2 * H * H);
        e |= dalloc(S, &S.WpqT[r], 2 * H * H);
        e |= dalloc(S, &S.We2[r], H * H);
        e |= dalloc(S, &S.We2T[r], H * H);
        e |= dalloc(S, &S.Wn1[r], 2 * H * H);
        e |= dalloc(S, &S.Wn1T[r], 2 * H * H);
        e |= dalloc(S, &S.Wn2[r], H * H);
        e |= dalloc(S, &S.Wn2T[r], H * H);
        e |= dalloc(S, &S.bpq[r], 2 * H);
        e |= dalloc(S, &S.A1[r], P * 2 * H);
        e |= dalloc(S, &S.PQ[r], P * 2 * H);
        if (r == 0) e |= dalloc(S, &S.PQf, P * 2 * H);
        e |= dalloc(S, &S.S[r], P * H);
        e |= dalloc(S, &S.G1[r], P * H);
        e |= dalloc(S, &S.Z1[r], P * H);
    }
    e |= dalloc(S, &S.Wd1, H * H);
    e |= dalloc(S, &S.Wd1T, H * H);
    e |= dalloc(S, &S.Wd2, FOUT * H);
    e |= dalloc(S, &S.Wd2T, H * FOUT);
    e |= dalloc(S, &S.bd2, FOUT);
    e |= dalloc(S, &S.X16, P * FIN);
    e |= dalloc(S, &S.A0, P * H);
    e |= dalloc(S, &S.Z0, P * H);
    for (int k = 0; k < 3; ++k) e |= dalloc(S, &S.h[k], P * H);
    e |= dalloc(S, &S.degs, P);
    e |= dalloc(S, &S.hLb, P * H);
    e |= dalloc(S, &S.Z2, P * H);
    e |= dalloc(S, &S.A2, P * H);
    e |= dalloc(S, &S.Y, P * FOUT);
    e |= dalloc(S, &S.NF, P);
    e |= dalloc(S, &S.loss_d, 1);
    e |= dalloc(S, &S.err, 1);
    if (e) return SPH_ENOMEM;
    CUR(cudaDeviceSynchronize());   // the zero fills precede any use on the simulation's stream
    return SPH_OK;
}

// Particles up to which the backward pass keeps a buffer per layer and takes the weight and
// bias gradients beside the data gradients; beyond, or where that much memory is not there, the
// layers share one set of buffers and one stream (10.1 against 4.2 KB a particle).  A training step
// with one set against a set per layer (GB300): 3 220 particles 857 against 583 us, 46 556 1846
// against 1490, 77 976 5474 against 5177, 193 496 12.18 against 11.95 ms, 335 000 19.91 against 19.78,
// 656 600 38.91 against 38.77: beyond a million the 5.9 KB a particle buy next to nothing.
constexpr int SIDE_MAX = 1 << 20;

// The device buffers of the backward pass; all of them or none.
int alloc_backward_set(Surrogate &S, bool own, float **dS)
{
    const size_t P = (size_t)S.npad, mark = S.allocs.size();
    int e = 0;
    auto layers = [&](auto *p, int count, size_t width) {
        for (int k = 0; k < count && !e; ++k) {
            if (k == 0 || own) e |= dalloc(S, &p[k], P * width);
            else p[k] = p[0];
        }
    };
    layers(&S.dYf, 1, FOUT);
    layers(&S.dYb, 1, FOUT);
    layers(S.dZf, 4, H);
    layers(S.dZb, 4, H);
    layers(S.dA, 2, 2 * H);
    layers(S.dAb, 2, 2 * H);
    layers(S.dh, 3, H);
    layers(S.dhb, 3, H);
    layers(S.dPQ, 2, 2 * H);
    layers(dS, 1, H);
    if (!e) e = dalloc(S, &S.sums, SUMS);
    if (!e) e = dalloc(S, &S.args, 1);
    if (e) {
        for (; S.allocs.size() > mark; S.allocs.pop_back()) cudaFree(S.allocs.back());
        cudaGetLastError();   // the refused allocation is not an error of what follows
        return SPH_ENOMEM;
    }
    return SPH_OK;
}

int alloc_backward(Surrogate &S)
{
    if (S.dS) return SPH_OK;
    if (!S.loss_h) {
        void *q = nullptr;
        const cudaError_t ce = cudaMallocHost(&q, sizeof(double) + sizeof(StepArgs) + sizeof(float) * S.L.total);
        if (ce != cudaSuccess) return set_error(SPH_ENOMEM, std::string("cudaMallocHost: ") + cudaGetErrorString(ce));
        S.loss_h = static_cast<double *>(q);
        S.args_h = reinterpret_cast<StepArgs *>(S.loss_h + 1);
        S.grad_h = reinterpret_cast<float *>(S.args_h + 1);
    }
    bool own = S.n <= SIDE_MAX;
    float *dS = nullptr;
    int rc = alloc_backward_set(S, own, &dS);
    if (rc && own) rc = alloc_backward_set(S, own = false, &dS);
    if (rc) return rc;
    if (own) {
        S.fork.resize(BWD_LAYERS, nullptr);
        for (cudaEvent_t &ev : S.fork)
            if (!ev) CUR(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        for (cudaEvent_t &ev : S.join)
            if (!ev) CUR(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        for (cudaStream_t &t : S.side)
            if (!t) CUR(cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking));
    }
    CUR(cudaDeviceSynchronize());
    S.dS = dS;
    return SPH_OK;
}

// Forward pass at the simulation's current state (rates evaluated by the
// caller); the pre-activations the backward pass needs are stored only when
// training.
int forward(Surrogate &S, const SimView &v, bool training)
{
    const Layout &L = S.L;
    const float *T = S.theta;
    cudaStream_t st = v.stream;
    const int n = v.n;
    int rc = 0;
    const float isu = 1.f / S.sd_edge_u, isr = 1.f / S.sd_edge_rho;
    if (v.dim == 2) k_features<2><<<nb(n), 256, 0, st>>>(v.d, S.norm_d, S.t_jump, isu, isr, S.X16, S.NF);
    else k_features<3><<<nb(n), 256, 0, st>>>(v.d, S.norm_d, S.t_jump, isu, isr, S.X16, S.NF);
    CUR(cudaGetLastError());
    {
        Epi e;
        e.bias = T + L.enc1b;
        e.act = 1;
        e.Z = training ? S.Z0 : nullptr;
        e.ldz = H;
        e.Cb = S.A0;
        e.ldcb = H;
        if ((rc = mm(S, st, S.X16, FIN, S.Wenc1, FIN, n, H, FIN, e))) return rc;
    }
    {
        Epi e;
        e.bias = T + L.enc2b;
        e.Cf = S.h[0];
        e.ldcf = H;
        e.Cb = S.A1[0];
        e.ldcb = 2 * H;
        if ((rc = mm(S, st, S.A0, H, S.Wenc2, H, n, H, H, e))) return rc;
    }
    const float R2 = (float)(4.0 * v.h * v.h), inv2h = (float)(0.5 / v.h), invk = 1.f / S.k_ref;
    for (int r = 0; r < 2; ++r) {
        {
            Epi e;
            e.bias = S.bpq[r];
            // the backward pass reads the unfolded terms
            e.Cb = training ? (bf16 *)S.PQ[r] : nullptr;
            e.ldcb = 2 * H;
            e.fold_f = S.NF;
            e.fold_w = T + L.w3[r];
            e.dim = v.dim;
            e.fold_out = S.PQf;
            if ((rc = mm(S, st, S.A1[r], 2 * H, S.Wpq[r], H, n, 2 * H, H, e))) return rc;
        }
        const int eb = std::min(nb(n, EWF / 16), S.sms * EDGE_BLOCKS);
        if (v.dim == 2)
            k_edge_fwd<2><<<eb, EWF, 0, st>>>(v.d, v.g, R2, inv2h, S.PQf, T + L.w3[r], invk, S.S[r],
                                                           S.degs);
        else
            k_edge_fwd<3><<<eb, EWF, 0, st>>>(v.d, v.g, R2, inv2h, S.PQf, T + L.w3[r], invk, S.S[r],
                                                           S.degs);
        CUR(cudaGetLastError());
        {
            Epi e;
            e.row_scale = S.degs;
            e.row_bias = T + L.be2[r];
            e.Cb = S.A1[r] + H;
            e.ldcb = 2 * H;
            if ((rc = mm(S, st, S.S[r], H, S.We2[r], H, n, H, H, e))) return rc;
        }
        {
            Epi e;
            e.bias = T + L.n1b[r];
            e.act = 1;
            e.Z = training ? S.Z1[r] : nullptr;
            e.ldz = H;
            e.Cb = S.G1[r];
            e.ldcb = H;
            if ((rc = mm(S, st, S.A1[r], 2 * H, S.Wn1[r], 2 * H, n, H, 2 * H, e))) return rc;
        }
        {
            Epi e;
            e.bias = T + L.n2b[r];
            e.residual = S.h[r];
            e.ldr = H;
            e.Cf = S.h[r + 1];
            e.ldcf = H;
            e.Cb = r == 0 ? S.A1[1] : S.hLb;
            e.ldcb = r == 0 ? 2 * H : H;
            if ((rc = mm(S, st, S.G1[r], H, S.Wn2[r], H, n, H, H, e))) return rc;
        }
    }
    {
        Epi e;
        e.bias = T + L.dec1b;
        e.act = 1;
        e.Z = training ? S.Z2 : nullptr;
        e.ldz = H;
        e.Cb = S.A2;
        e.ldcb = H;
        if ((rc = mm(S, st, S.hLb, H, S.Wd1, H, n, H, H, e))) return rc;
    }
    {
        Epi e;
        e.bias = S.bd2;
        e.Cf = S.Y;
        e.ldcf = FOUT;
        if ((rc = mm(S, st, S.A2, H, S.Wd2, H, n, FOUT, H, e))) return rc;
    }
    return SPH_OK;
}

// Backward pass from dY (S.dYf / S.dYb) into S.grad (zeroed here).  The chain
// of data gradients runs on the simulation's stream; each layer's weight
// gradient and column sums, which nothing waits for before the update, run on
// two streams of the surrogate's own from the moment their inputs are there
// (a layer's launch fills a fraction of the chip: 26 tiles of 152 SMs on 3 220
// particles), and the simulation's stream waits for both at the end.  A training
// step on 3 220 particles 1.12 -> 0.80 ms, on 193 496 12.51 -> 12.37 ms.
int backward(Surrogate &S, const SimView &v)
{
    const Layout &L = S.L;
    const float *T = S.theta;
    float *G = S.grad;
    cudaStream_t st = v.stream;
    const int n = v.n;
    const int cs_blocks = std::max(1, std::min(1024, nb(n, 512)));
    int rc = 0, layer = 0;
    cudaStream_t sw = S.side[0] ? S.side[0] : st, sb = S.side[1] ? S.side[1] : st;
    // the side streams see everything queued on the simulation's stream so far
    auto fork = [&]() -> int {
        if (!S.side[0]) return SPH_OK;
        const cudaEvent_t ev = S.fork[layer++];
        CUR(cudaEventRecord(ev, st));
        CUR(cudaStreamWaitEvent(sw, ev, 0));
        CUR(cudaStreamWaitEvent(sb, ev, 0));
        return SPH_OK;
    };
    CUR(cudaMemsetAsync(G, 0, sizeof(float) * L.total, st));
    CUR(cudaMemsetAsync(S.sums, 0, sizeof(double) * SUMS, st));
    // the FP64 sums: the edge phase's of both rounds, then H for each bias of a layer
    SumTable out{};
    int next = 2 * W3_SUMS;
    auto sum_of = [&](int from, int to, int len) {
        out.from[out.count] = from;
        out.to[out.count] = to;
        out.len[out.count++] = len;
    };
    auto bias_sum = [&](int to, int len) {
        sum_of(next, to, len);
        next += H;
        return S.sums + next - H;
    };
    for (int r = 0; r < 2; ++r) {
        sum_of(r * W3_SUMS, L.w3[r], H * L.ne);
        sum_of(r * W3_SUMS + H * L.ne, L.b1[r], H);
    }
    // decoder, layer 2
    if ((rc = fork())) return rc;
    if ((rc = wgrad(S, sw, S.dYb, FOUT, FOUT, S.A2, H, H, G + L.dec2w, L.nout, H))) return rc;
    k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dYf, FOUT, L.nout, n, nullptr, bias_sum(L.dec2b, L.nout));
    {
        Epi e;
        e.act = 2;
        e.dact = S.Z2;
        e.lddact = H;
        e.Cf = S.dZf[0];
        e.ldcf = H;
        e.Cb = S.dZb[0];
        e.ldcb = H;
        if ((rc = mm(S, st, S.dYb, FOUT, S.Wd2T, FOUT, n, H, FOUT, e))) return rc;
    }
    // decoder, layer 1
    if ((rc = fork())) return rc;
    if ((rc = wgrad(S, sw, S.dZb[0], H, H, S.hLb, H, H, G + L.dec1w, H, H))) return rc;
    k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dZf[0], H, H, n, nullptr, bias_sum(L.dec1b, H));
    {
        Epi e;
        e.Cf = S.dh[0];
        e.ldcf = H;
        e.Cb = S.dhb[0];
        e.ldcb = H;
        if ((rc = mm(S, st, S.dZb[0], H, S.Wd1T, H, n, H, H, e))) return rc;
    }
    const float R2 = (float)(4.0 * v.h * v.h), inv2h = (float)(0.5 / v.h), invk = 1.f / S.k_ref;
    for (int r = 1; r >= 0; --r) {
        const int q = 1 - r;                           // dh comes in as dh[q] and leaves as dh[q + 1]
        const bf16 *hb = r == 0 ? S.A1[0] : S.A1[1];   // h_r in BF16: left half of [h, M]
        // node MLP, layer 2 (residual: dh passes through)
        if ((rc = fork())) return rc;
        if ((rc = wgrad(S, sw, S.dhb[q], H, H, S.G1[r], H, H, G + L.n2[r], H, H))) return rc;
        k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dh[q], H, H, n, nullptr, bias_sum(L.n2b[r], H));
        {
            Epi e;
            e.act = 2;
            e.dact = S.Z1[r];
            e.lddact = H;
            e.Cf = S.dZf[1 + q];
            e.ldcf = H;
            e.Cb = S.dZb[1 + q];
            e.ldcb = H;
            if ((rc = mm(S, st, S.dhb[q], H, S.Wn2T[r], H, n, H, H, e))) return rc;
        }
        // node MLP, layer 1 on [h, M]
        if ((rc = fork())) return rc;
        if ((rc = wgrad(S, sw, S.dZb[1 + q], H, H, S.A1[r], 2 * H, 2 * H, G + L.n1[r], H, 2 * H))) return rc;
        k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dZf[1 + q], H, H, n, nullptr, bias_sum(L.n1b[r], H));
        {
            Epi e;
            e.Cf = S.dA[q];
            e.ldcf = 2 * H;
            e.Cb = S.dAb[q];
            e.ldcb = 2 * H;
            if ((rc = mm(S, st, S.dZb[1 + q], H, S.Wn1T[r], H, n, 2 * H, H, e))) return rc;
        }
        // second edge layer, applied after the sum: M = S We2^T + degs be2
        if ((rc = fork())) return rc;
        if ((rc = wgrad(S, sw, S.dAb[q] + H, 2 * H, H, S.S[r], H, H, G + L.we2[r], H, H))) return rc;
        k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dA[q] + H, 2 * H, H, n, S.degs, bias_sum(L.be2[r], H));
        {
            Epi e;
            e.Cf = S.dS;
            e.ldcf = H;
            if ((rc = mm(S, st, S.dAb[q] + H, 2 * H, S.We2T[r], H, n, H, H, e))) return rc;
        }
        // edge phase
        const int wb = std::min(nb(n, EWB / 32), S.sms * EWB_BLOCKS);
        if (v.dim == 2)
            k_edge_bwd<2><<<wb, EWB, 0, st>>>(v.d, v.g, R2, inv2h, S.NF, S.PQ[r], T + L.w3[r], invk,
                                                         S.dS, S.dPQ[q], S.sums + r * W3_SUMS);
        else
            k_edge_bwd<3><<<wb, EWB, 0, st>>>(v.d, v.g, R2, inv2h, S.NF, S.PQ[r], T + L.w3[r], invk,
                                                         S.dS, S.dPQ[q], S.sums + r * W3_SUMS);
        CUR(cudaGetLastError());
        // first edge layer, node parts: P = h W1^T + b1, Q = h W2^T
        if ((rc = fork())) return rc;
        if ((rc = wgrad(S, sw, S.dPQ[q], 2 * H, 2 * H, hb, 2 * H, H, G + L.w1[r], H, H, G + L.w2[r]))) return rc;
        // dh_r = dh_{r+1} + d[h part of n1 input] + dP W1 + dQ W2
        {
            Epi e;
            e.residual = S.dh[q];   // may be the output: a row's elements are read before they are written
            e.ldr = H;
            e.residual2 = S.dA[q];
            e.ldr2 = 2 * H;
            e.Cf = S.dh[q + 1];
            e.ldcf = H;
            e.Cb = S.dhb[q + 1];
            e.ldcb = H;
            if ((rc = mm(S, st, S.dPQ[q], 2 * H, S.WpqT[r], 2 * H, n, H, 2 * H, e))) return rc;
        }
    }
    // encoder, layer 2
    if ((rc = fork())) return rc;
    if ((rc = wgrad(S, sw, S.dhb[2], H, H, S.A0, H, H, G + L.enc2w, H, H))) return rc;
    k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dh[2], H, H, n, nullptr, bias_sum(L.enc2b, H));
    {
        Epi e;
        e.act = 2;
        e.dact = S.Z0;
        e.lddact = H;
        e.Cf = S.dZf[3];
        e.ldcf = H;
        e.Cb = S.dZb[3];
        e.ldcb = H;
        if ((rc = mm(S, st, S.dhb[2], H, S.Wenc2T, H, n, H, H, e))) return rc;
    }
    // encoder, layer 1
    if ((rc = fork())) return rc;
    if ((rc = wgrad(S, sw, S.dZb[3], H, H, S.X16, FIN, FIN, G + L.enc1w, H, L.nin))) return rc;
    k_colsum<<<cs_blocks, 256, 0, sb>>>(S.dZf[3], H, H, n, nullptr, bias_sum(L.enc1b, H));
    CUR(cudaGetLastError());
    for (int k = 0; k < 2 && S.side[k]; ++k) {
        CUR(cudaEventRecord(S.join[k], S.side[k]));
        CUR(cudaStreamWaitEvent(st, S.join[k], 0));
    }
    k_sums_out<<<dim3(nb(W3_SUMS), out.count), 256, 0, st>>>(S.sums, G, out);
    CUR(cudaGetLastError());
    return SPH_OK;
}

Surrogate *get(sph_handle h)
{
    return h ? static_cast<Surrogate *>(sim_ext(h)) : nullptr;
}

constexpr double ADAM_B1 = 0.9, ADAM_B2 = 0.999;

// (node, channel) terms of the loss: every channel of fluid nodes, the density channel of walls.
double loss_terms(const Surrogate &S, const SimView &v)
{
    return (double)(v.n - v.nwall) * S.L.nout + (double)v.nwall;
}

// Queues one training step: rates, forward, loss, backward and, with update,
// Adam and the repacking of the weights.  What changes from step to step is in
// S.args, so the launches can be captured once and replayed: launched one by
// one, about 75 kernels of a few microseconds keep the stream waiting for the host
// and for the events between the streams.  Replayed, a step of 3 220 particles took 566
// instead of 662 us, of 193 496 particles 11.92 instead of 12.16 ms.
int enqueue_train_step(sph_handle h, Surrogate &S, bool update)
{
    int rc = sph_eval_rates(h);
    if (rc) return rc;
    const SimView v = sim_view(h);
    if ((rc = forward(S, v, true))) return rc;
    CUR(cudaMemsetAsync(S.loss_d, 0, sizeof(double), v.stream));
    const float inv_count = (float)(1.0 / loss_terms(S, v));
    if (v.dim == 2)
        k_loss<2><<<nb(v.n), 256, 0, v.stream>>>(v.d, S.norm_d, S.t_jump, S.Y, S.args, inv_count, S.dYf, S.dYb,
                                                 S.loss_d);
    else
        k_loss<3><<<nb(v.n), 256, 0, v.stream>>>(v.d, S.norm_d, S.t_jump, S.Y, S.args, inv_count, S.dYf, S.dYb,
                                                 S.loss_d);
    CUR(cudaGetLastError());
    if ((rc = backward(S, v))) return rc;
    if (!update) return SPH_OK;
    k_adam<<<nb(S.L.total), 256, 0, v.stream>>>(v.d, S.theta, S.grad, S.m, S.v, S.L.total, S.args, (float)ADAM_B1,
                                                (float)ADAM_B2);
    CUR(cudaGetLastError());
    return pack_weights(S, v.stream);
}

// The step's launches as a graph; NULL where the stream does not allow it (nothing has been
// launched then).
cudaGraphExec_t capture_train_step(sph_handle h, Surrogate &S, bool update, cudaStream_t st)
{
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        const int rc = enqueue_train_step(h, S, update);
        const cudaError_t e = cudaStreamEndCapture(st, &g);
        if (!rc && e == cudaSuccess && cudaGraphInstantiate(&exec, g, 0) != cudaSuccess) exec = nullptr;
        if (g) cudaGraphDestroy(g);
    }
    cudaGetLastError();   // a refusal is not an error of the step
    return exec;
}

int check_err(Surrogate &S, cudaStream_t st)
{
    unsigned e = 0;
    CUR(cudaMemcpyAsync(&e, S.err, sizeof(e), cudaMemcpyDeviceToHost, st));
    CUR(cudaStreamSynchronize(st));
    if (e) {
        CUR(cudaMemsetAsync(S.err, 0, sizeof(unsigned), st));
        return set_error(SPH_ETIMEOUT, "a tensor-core wait of the surrogate exceeded one second");
    }
    return SPH_OK;
}

}  // namespace

extern "C" {

int sph_mm_bf16(const void *A, int lda, const void *B, int ldb, float *C, int ldc, int M, int N, int K, int k_split,
                int accumulate, void *stream, unsigned *err_dev)
{
    if (!A || !B || !C || !err_dev) return set_error(SPH_EINVAL, "NULL argument");
    if (M < 0 || K < 0 || (N != 16 && N != 32 && N != 64 && N != 128 && N != 256))
        return set_error(SPH_EINVAL, "N must be 16, 32, 64, 128 or 256 and M, K >= 0");
    if (K % 16 != 0 || lda % 8 != 0 || ldb % 8 != 0 || lda < K || ldb < K || ldc < N)
        return set_error(SPH_EINVAL, "K must be a multiple of 16, lda and ldb multiples of 8 and >= K");
    if (k_split <= 0) k_split = ((K + umma::BK - 1) / umma::BK) * umma::BK;
    if (k_split % umma::BK != 0) return set_error(SPH_EINVAL, "k_split must be a multiple of 64");
    if (K > k_split && !accumulate) return set_error(SPH_EINVAL, "a split K needs accumulate");
    if ((uintptr_t)A % 16 || (uintptr_t)B % 16) return set_error(SPH_EINVAL, "A and B must be 16-byte aligned");
    umma::GemmArgs g{};
    g.A = (const bf16 *)A;
    g.lda = lda;
    g.B = (const bf16 *)B;
    g.ldb = ldb;
    g.M = M;
    g.N = N;
    g.K = K;
    g.k_split = k_split;
    g.Cf = C;
    g.ldcf = ldc;
    g.atomic = accumulate ? 1 : 0;
    g.err = err_dev;
    cudaError_t e = umma::gemm(g, (cudaStream_t)stream);
    if (e != cudaSuccess) return set_error(SPH_ECUDA, std::string("gemm launch: ") + cudaGetErrorString(e));
    return SPH_OK;
}

int sph_surrogate_init(sph_handle h, const double *weights, int64_t nweights, const double *norm, int64_t nnorm)
{
    if (!h || !weights || !norm) return set_error(SPH_EINVAL, "NULL argument");
    const SimView v = sim_view(h);
    if (v.ninst != 1) return set_error(SPH_EINVAL, "the surrogate runs on single-instance handles");
    if (v.npiston > 0) return set_error(SPH_EINVAL, "the surrogate does not move piston particles");
    const Layout L = make_layout(v.dim);
    if (nweights != L.total) return set_error(SPH_EINVAL, "weights: wrong number of parameters for this dim");
    if (nnorm != 2 * L.nin + 2 * L.nout + 4) return set_error(SPH_EINVAL, "norm: wrong length for this dim");
    for (int64_t k = 0; k < nnorm; ++k)
        if (!std::isfinite(norm[k])) return set_error(SPH_EINVAL, "norm must be finite");
    for (int c = 0; c < L.nin; ++c)
        if (!(norm[L.nin + c] > 0)) return set_error(SPH_EINVAL, "sd_in must be positive");
    for (int c = 0; c < L.nout; ++c)
        if (!(norm[2 * L.nin + L.nout + c] > 0)) return set_error(SPH_EINVAL, "sd_out must be positive");
    const int o = 2 * L.nin + 2 * L.nout;
    if (!(norm[o] > 0) || !(norm[o + 1] >= 0) || !(norm[o + 2] > 0) || !(norm[o + 3] > 0))
        return set_error(SPH_EINVAL, "k_ref, sd_edge_u and sd_edge_rho must be positive and T >= 0");
    for (int64_t k = 0; k < nweights; ++k)
        if (!std::isfinite(weights[k])) return set_error(SPH_EINVAL, "weights must be finite");
    Surrogate *S = get(h);
    if (!S || S->dim != v.dim || S->n != v.n) {
        S = new Surrogate();
        S->dim = v.dim;
        S->n = v.n;
        S->npad = std::max(128, ((v.n + 127) / 128) * 128);
        S->L = L;
        int dev = 0;
        cudaError_t ce = cudaGetDevice(&dev);
        if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&S->sms, cudaDevAttrMultiProcessorCount, dev);
        if (ce != cudaSuccess) {
            delete S;
            return set_error(SPH_ECUDA, cudaGetErrorString(ce));
        }
        int rc = alloc_surrogate(*S);
        if (rc) {
            delete S;
            return rc;
        }
        sim_set_ext(h, S, free_surrogate);
    }
    S->drop_graphs();   // their launches hold the normalisation
    S->k_ref = (float)norm[o];
    S->t_jump = (float)norm[o + 1];
    S->t_jump64 = norm[o + 1];
    S->sd_edge_u = (float)norm[o + 2];
    S->sd_edge_rho = (float)norm[o + 3];
    S->norm.assign(norm, norm + o);
    std::vector<float> tf(weights, weights + nweights);
    CUR(cudaMemcpyAsync(S->theta, tf.data(), sizeof(float) * nweights, cudaMemcpyHostToDevice, v.stream));
    CUR(cudaMemcpyAsync(S->norm_d, S->norm.data(), sizeof(float) * S->norm.size(), cudaMemcpyHostToDevice, v.stream));
    CUR(cudaMemsetAsync(S->m, 0, sizeof(float) * nweights, v.stream));
    CUR(cudaMemsetAsync(S->v, 0, sizeof(float) * nweights, v.stream));
    S->adam_t = 0;
    int rc = pack_weights(*S, v.stream);
    if (rc) return rc;
    CUR(cudaStreamSynchronize(v.stream));
    return SPH_OK;
}

int sph_surrogate_get_weights(sph_handle h, double *weights, int64_t nweights)
{
    Surrogate *S = get(h);
    if (!S || !weights) return set_error(SPH_EINVAL, "no surrogate on this handle, or NULL argument");
    if (nweights != S->L.total) return set_error(SPH_EINVAL, "weights: wrong length");
    const SimView v = sim_view(h);
    std::vector<float> tf(nweights);
    CUR(cudaMemcpyAsync(tf.data(), S->theta, sizeof(float) * nweights, cudaMemcpyDeviceToHost, v.stream));
    CUR(cudaStreamSynchronize(v.stream));
    for (int64_t k = 0; k < nweights; ++k) weights[k] = tf[k];
    return SPH_OK;
}

int sph_surrogate_predict(sph_handle h, double *out, int64_t bytes)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    const SimView v0 = sim_view(h);
    const size_t need = (size_t)v0.n * S->L.nout * sizeof(double);
    if (!out || bytes < (int64_t)need) return set_error(SPH_EINVAL, "output buffer too small");
    if (v0.n == 0) return SPH_OK;
    int rc0 = sph_eval_rates(h);
    if (rc0) return rc0;
    const SimView v = sim_view(h);
    int rc = forward(*S, v, false);
    if (rc) return rc;
    double *dout = nullptr;
    CUR(cudaMallocAsync((void **)&dout, need, v.stream));
    if (v.dim == 2) k_predict_out<2><<<nb(v.n), 256, 0, v.stream>>>(v.d, S->norm_d, S->t_jump, S->Y, dout);
    else k_predict_out<3><<<nb(v.n), 256, 0, v.stream>>>(v.d, S->norm_d, S->t_jump, S->Y, dout);
    CUR(cudaGetLastError());
    CUR(cudaMemcpyAsync(out, dout, need, cudaMemcpyDeviceToHost, v.stream));
    CUR(cudaFreeAsync(dout, v.stream));
    if ((rc = check_err(*S, v.stream))) return rc;
    return sim_check(h);
}

int sph_surrogate_advance(sph_handle h, int k_steps)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (k_steps < 1) return set_error(SPH_EINVAL, "k_steps must be >= 1");
    const SimView v0 = sim_view(h);
    if (v0.n == 0) return sim_moved(h, k_steps, S->t_jump64);
    int rc0 = sph_eval_rates(h);
    if (rc0) return rc0;
    const SimView v = sim_view(h);
    int rc = forward(*S, v, false);
    if (rc) return rc;
    if (v.dim == 2) k_apply<2><<<nb(v.n), 256, 0, v.stream>>>(v.d, S->norm_d, S->t_jump, S->Y);
    else k_apply<3><<<nb(v.n), 256, 0, v.stream>>>(v.d, S->norm_d, S->t_jump, S->Y);
    CUR(cudaGetLastError());
    return sim_moved(h, k_steps, S->t_jump64);
}

int sph_surrogate_train_step(sph_handle h, const double *x1, const double *u1, const double *rho1, double lr,
                             int update, double *loss_out, double *grad_out, int64_t ngrad)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (!x1 || !u1 || !rho1) return set_error(SPH_EINVAL, "target arrays are NULL");
    if (update && !(lr > 0)) return set_error(SPH_EINVAL, "lr must be positive");
    if (grad_out && ngrad != S->L.total) return set_error(SPH_EINVAL, "grad_out: wrong length");
    const SimView v0 = sim_view(h);
    if (v0.n == 0) return set_error(SPH_EINVAL, "no particles");
    int rc = alloc_backward(*S);
    if (rc) return rc;
    *S->args_h = {x1, u1, rho1, 0.f, 0.f};
    const int64_t t = S->adam_t + 1;
    if (update) {
        const double b1 = ADAM_B1, b2 = ADAM_B2, eps = 1e-8;
        // theta -= lr mhat / (sqrt(vhat) + eps) with mhat = m / c1, vhat = v / c2
        const double c1 = 1.0 - std::pow(b1, (double)t), c2 = 1.0 - std::pow(b2, (double)t);
        S->args_h->lr_t = (float)(lr * std::sqrt(c2) / c1);
        S->args_h->eps_t = (float)(eps * std::sqrt(c2));
    }
    CUR(cudaMemcpyAsync(S->args, S->args_h, sizeof(StepArgs), cudaMemcpyHostToDevice, v0.stream));
    // the first step of each kind launches kernel by kernel, later ones replay its graph, but
    // where there is none (cudaStreamLegacy cannot be captured)
    cudaGraphExec_t &graph = S->step_graph[update ? 1 : 0];
    if (S->step_calls[update ? 1 : 0]++ > 0 && !v0.timing && !graph)
        graph = capture_train_step(h, *S, update != 0, v0.stream);
    if (graph && !v0.timing) {
        CUR(cudaGraphLaunch(graph, v0.stream));
        sim_evaluated(h);
    } else if ((rc = enqueue_train_step(h, *S, update != 0))) {
        return rc;
    }
    if (update) S->adam_t = t;
    const SimView v = v0;
    const double count = loss_terms(*S, v);
    // the loss and the gradient come back behind everything else, with one wait (check_err's)
    CUR(cudaMemcpyAsync(S->loss_h, S->loss_d, sizeof(double), cudaMemcpyDeviceToHost, v.stream));
    if (grad_out) CUR(cudaMemcpyAsync(S->grad_h, S->grad, sizeof(float) * ngrad, cudaMemcpyDeviceToHost, v.stream));
    if ((rc = check_err(*S, v.stream))) return rc;
    if (grad_out)
        for (int64_t k = 0; k < ngrad; ++k) grad_out[k] = S->grad_h[k];
    if (loss_out) *loss_out = *S->loss_h / count;
    rc = sim_check(h);
    if (update && rc == SPH_ETIMEOUT) S->adam_t = t - 1;   // no update was made
    return rc;
}

int sph_snapshot(sph_handle h, double *x_dev, double *u_dev, double *rho_dev)
{
    if (!h || !x_dev || !u_dev || !rho_dev) return set_error(SPH_EINVAL, "NULL argument");
    return sim_snapshot_device(h, x_dev, u_dev, rho_dev);
}

int sph_load_snapshot(sph_handle h, const double *x_dev, const double *u_dev, const double *rho_dev)
{
    if (!h || !x_dev || !u_dev || !rho_dev) return set_error(SPH_EINVAL, "NULL argument");
    return sim_load_device(h, x_dev, u_dev, rho_dev);
}

namespace {

// Errors that mean "the jump produced an unusable state" rather than a
// failure of the library.
bool state_error(int rc)
{
    return rc == SPH_ENONFINITE || rc == SPH_EDOMAIN || rc == SPH_ECAPACITY || rc == SPH_ECFL;
}

// The plain steps that judge or replace a jump must span the time the network
// jumps (its normalisation block's t_jump): k_steps * dt = t_jump, up to the
// rounding of either.
int check_jump_span(const Surrogate &S, double dt, int k_steps)
{
    const double span = (double)k_steps * dt;
    if (!(std::fabs(span - S.t_jump64) <= 1e-9 * S.t_jump64)) {
        char m[200];
        snprintf(m, sizeof m, "k_steps * dt = %.9g s differs from the network's jump span t_jump = %.9g s", span,
                 S.t_jump64);
        return set_error(SPH_EINVAL, m);
    }
    return SPH_OK;
}

// Snapshot buffers of the judged run (allocated once per surrogate).
int judge_buffers(Surrogate &S, const SimView &v, sph_handle h)
{
    if (S.sx) return SPH_OK;
    const size_t nd = (size_t)v.n * v.dim;
    const size_t words = (size_t)sim_occupancy_words(h);
    int e = dalloc(S, &S.sx, nd) | dalloc(S, &S.su, nd) | dalloc(S, &S.sr, (size_t)v.n) |
            dalloc(S, &S.vx, nd) | dalloc(S, &S.vu, nd) | dalloc(S, &S.vr, (size_t)v.n) |
            dalloc(S, &S.occ_a, words) | dalloc(S, &S.occ_b, words);
    if (e) return SPH_ENOMEM;
    CUR(cudaDeviceSynchronize());
    return SPH_OK;
}

// One judged macro-step: the surrogate jump and k plain steps from the same
// state; the plain result is kept.  *err = |c_jump - c_plain| / d_ref for the
// oil centroids, *ierr = |O_jump xor O_plain| / |O_plain| for the oil
// occupancies (both 1e30 when the jump broke the state).  Updates the
// surrogate's maxima; *reject tells whether either tolerance is exceeded.
int judged_jump(sph_handle h, Surrogate &S, const SimView &v, double dt, int k_steps, double d_ref, double tol,
                double *err, bool *reject)
{
    int rc;
    if ((rc = sim_snapshot_device(h, S.sx, S.su, S.sr))) return rc;
    if ((rc = sph_surrogate_advance(h, k_steps))) return rc;
    double cs[3] = {0, 0, 0}, cp[3];
    const int crc = sim_centroid(h, cs);
    if (crc && !state_error(crc)) return crc;
    if (!crc && (rc = sim_occupancy(h, S.occ_a))) return rc;
    if ((rc = sim_load_device(h, S.sx, S.su, S.sr))) return rc;
    if ((rc = sim_moved(h, -k_steps, -S.t_jump64))) return rc;
    if ((rc = sph_run(h, dt, k_steps, 1))) return rc;
    if ((rc = sim_centroid(h, cp))) return rc;
    double ierr = 1.0e30;
    if (!crc) {
        if ((rc = sim_occupancy(h, S.occ_b))) return rc;
        if ((rc = sim_occupancy_error(h, S.occ_a, S.occ_b, &ierr))) return rc;
    }
    double e2 = 0.0;
    for (int c = 0; c < v.dim; ++c) e2 += (cs[c] - cp[c]) * (cs[c] - cp[c]);
    *err = crc ? 1.0e30 : std::sqrt(e2) / d_ref;
    S.max_cerr = std::max(S.max_cerr, *err);
    S.max_ierr = std::max(S.max_ierr, ierr);
    *reject = *err > tol || (S.itol > 0 && ierr > S.itol);
    return SPH_OK;
}

}  // namespace

int sph_surrogate_advance_judged(sph_handle h, double dt, int k_steps, double tol, double d_ref, double *err)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (!(dt > 0) || k_steps < 1 || !(tol > 0) || !(d_ref > 0))
        return set_error(SPH_EINVAL, "bad dt, k_steps, tol or d_ref");
    if (int e = check_jump_span(*S, dt, k_steps)) return e;
    const SimView v = sim_view(h);
    int rc = judge_buffers(*S, v, h);
    if (rc) return rc;
    double e = 0.0;
    bool reject = false;
    S->max_cerr = S->max_ierr = 0.0;
    if ((rc = judged_jump(h, *S, v, dt, k_steps, d_ref, tol, &e, &reject))) return rc;
    if (err) *err = e;
    if ((rc = check_err(*S, v.stream))) return rc;
    if ((rc = sim_check(h))) return rc;
    return reject ? set_error(SPH_EFALLBACK, "the judge rejected the surrogate jump; the state holds the plain steps")
                  : SPH_OK;
}

int sph_surrogate_set_interface_tol(sph_handle h, double tol)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (!(tol >= 0) || !std::isfinite(tol)) return set_error(SPH_EINVAL, "tol must be >= 0");
    S->itol = tol;
    return SPH_OK;
}

int sph_surrogate_judge_stats(sph_handle h, double *max_centroid_err, double *max_interface_err)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (max_centroid_err) *max_centroid_err = S->max_cerr;
    if (max_interface_err) *max_interface_err = S->max_ierr;
    return SPH_OK;
}

int sph_surrogate_run(sph_handle h, double dt, int k_steps, int64_t n_macro, int judge_every, double tol,
                      double d_ref, int64_t *n_judged, int64_t *n_rejected, double *max_err)
{
    Surrogate *S = get(h);
    if (!S) return set_error(SPH_EINVAL, "no surrogate on this handle");
    if (!(dt > 0) || k_steps < 1 || n_macro < 0 || judge_every < 0 || !(tol > 0) || !(d_ref > 0))
        return set_error(SPH_EINVAL, "bad dt, k_steps, n_macro, judge_every, tol or d_ref");
    if (int e = check_jump_span(*S, dt, k_steps)) return e;
    const SimView v = sim_view(h);
    if (int e = judge_buffers(*S, v, h)) return e;
    S->max_cerr = S->max_ierr = 0.0;
    // a state the plain method produced or accepted, and the macro-step it belongs to
    auto verify = [&](int64_t m, int64_t &mv) {
        mv = m;
        return sim_snapshot_device(h, S->vx, S->vu, S->vr);
    };
    int64_t judged = 0, rejected = 0, mv = 0;
    double worst = 0.0;
    bool fallback = false;
    int rc = verify(0, mv);
    if (rc) return rc;
    for (int64_t mstep = 0; mstep < n_macro; ++mstep) {
        const bool judge = judge_every > 0 && (mstep % judge_every) == 0;
        if (judge) {
            // surrogate jump and plain steps from the same state; the plain result is kept
            double err = 0.0;
            bool reject = false;
            rc = judged_jump(h, *S, v, dt, k_steps, d_ref, tol, &err, &reject);
            if (rc && !state_error(rc)) return rc;
            if (rc) {
                // the plain steps failed from the state the unjudged jumps left: back to
                // the last verified state, plain steps from there
                const int64_t redo = (mstep + 1 - mv) * k_steps;
                if ((rc = sim_load_device(h, S->vx, S->vu, S->vr))) return rc;
                if ((rc = sim_moved(h, -redo, -(double)(mstep + 1 - mv) * S->t_jump64))) return rc;
                if ((rc = sph_run(h, dt, redo, 1))) return rc;
                err = 1.0e30;
                reject = true;
                S->max_cerr = std::max(S->max_cerr, err);
            }
            worst = std::max(worst, err);
            ++judged;
            fallback = reject;
            rejected += fallback ? 1 : 0;
            if ((rc = verify(mstep + 1, mv))) return rc;
        } else if (fallback) {
            if ((rc = sph_run(h, dt, k_steps, 1))) return rc;
        } else {
            if ((rc = sph_surrogate_advance(h, k_steps))) return rc;
            const int crc = sim_check(h);
            if (crc && !state_error(crc)) return crc;
            if (crc) {
                // the jump broke the state: back to the last verified state, plain steps from there
                const int64_t redo = (mstep + 1 - mv) * k_steps;
                if ((rc = sim_load_device(h, S->vx, S->vu, S->vr))) return rc;
                if ((rc = sim_moved(h, -redo, -(double)(mstep + 1 - mv) * S->t_jump64))) return rc;
                if ((rc = sph_run(h, dt, redo, 1))) return rc;
                ++rejected;
                fallback = true;
                if ((rc = verify(mstep + 1, mv))) return rc;
            }
        }
    }
    if ((rc = check_err(*S, v.stream))) return rc;
    if (n_judged) *n_judged = judged;
    if (n_rejected) *n_rejected = rejected;
    if (max_err) *max_err = worst;
    return sim_check(h);
}

}  // extern "C"
