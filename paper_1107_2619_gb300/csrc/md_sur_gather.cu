// Neighbour gathers of the learned per-atom surrogate: descriptors, forces, and the
// descriptor tangent used by the force term of the training loss.  One warp per atom, lane k
// = radial-basis channel k (32 channels = 32 lanes).  The lanes first evaluate the geometry of
// 32 list entries at once (lane q: entry q), stage it in shared memory, and then all lanes walk
// the entries inside the descriptor cutoff two at a time (packed FP32 operations), each adding its
// own channel.  The per-channel quantities of neighbour j (its gradient row g_j) are then one
// coalesced 128-byte row read.
//
//   descriptors  G_ik = sum_j b_k(r_ij)
//   forces       F_i  = sum_j [ sum_k (g_ik + g_jk) b_k'(r_ij) ] (r_j - r_i) / r_ij
//   tangent      u_ik = sum_j b_k'(r_ij) (r_j - r_i) / r_ij . (phi_j - phi_i),  phi = dL/dF
// with g = dE/dG.  The pair coefficient is symmetric in (i, j), so the forces are central pair
// forces and the virial has the pair form.  FP32 arithmetic; FP64 kick and partial sums.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "md_eam_common.cuh"
#include "md_pack2.cuh"
#include "md_phases.cuh"

namespace mdk {

namespace {

constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float mi(float d, float L, float iL) { return d - L * rintf(d * iL); }

using namespace pk;   // the packed operations of the channel loops (the halves: consecutive pairs of the row)

__device__ __forceinline__ float both(F2 x) {
    float a, b;
    unpack(x, a, b);
    return a + b;
}

// 2^x (PTX ex2.approx.ftz: relative error < 2^-22).
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ F2 ex2_2(F2 x) {
    float a, b;
    unpack(x, a, b);
    return pack(ex2(a), ex2(b));
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// The warp sums of four values with six shuffles instead of twenty: each of the first two rounds
// halves the values a lane carries; lane l ends with the sum of value l & 3.
__device__ __forceinline__ float warp_sum4(float a, float b, float c, float d) {
    const int lane = threadIdx.x & 31;
    const bool o1 = lane & 1, o2 = lane & 2;
    float x = o1 ? b : a, y = o1 ? d : c;
    x += __shfl_xor_sync(kFull, o1 ? a : b, 1);
    y += __shfl_xor_sync(kFull, o1 ? c : d, 1);
    float z = o2 ? y : x;
    z += __shfl_xor_sync(kFull, o2 ? x : y, 2);
    z += __shfl_xor_sync(kFull, z, 4);
    z += __shfl_xor_sync(kFull, z, 8);
    z += __shfl_xor_sync(kFull, z, 16);
    return z;
}

// Per-pair constants of one chunk of 32 list entries, compacted: the pairs inside rd take slots
// 0 .. n-1 in list order, two slots to a block whose words lie in the order the packed loops read
// them (value f of slot s at word (s / 2) kBlk + 2 f + (s & 1); kBlk = 4 (2 m + 1) words keeps the
// 16-byte reads aligned and the scattered stores two to a bank).  An odd n is filled up with a
// slot of zeros.
template <int NF>
struct Stage {
    static constexpr int kBlk = (NF + 1) / 2 * 4 % 8 ? (NF + 1) / 2 * 4 : (NF + 1) / 2 * 4 + 4;
    float4 w[16 * kBlk / 4];
    __device__ __forceinline__ void put(int s, int f, float v) {
        reinterpret_cast<float *>(w)[(s >> 1) * kBlk + 2 * f + (s & 1)] = v;
    }
    // values f and f + 1 (f even) of block b, each as its two slots
    __device__ __forceinline__ void get2(int b, int f, F2 &x, F2 &y) const {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(&w[(b * kBlk + 2 * f) / 4]);
        x.v = q.x;
        y.v = q.y;
    }
};

// Geometry of list entries [base, base + 32) of an atom at pi: lane q takes entry base + q; inside
// rd, fn(slot, r, 1/r, d, j) with the compacted slot.  Returns the number of pairs inside.
template <typename Fn>
__device__ __forceinline__ int stage_chunk(const Atoms &A, const SurNet &S, const float4 &pi, const Box &B,
                                           const NbrRow &row, int cnt, int base, int lane, Fn &&fn) {
    const int q = base + lane;
    const bool valid = q < cnt;
    const int j = valid ? __ldg(row.ptr(q)) : 0;
    const float4 pj = __ldg(A.posf + j);
    const float dx = mi(pj.x - pi.x, B.Lf[0], B.invLf[0]);
    const float dy = mi(pj.y - pi.y, B.Lf[1], B.invLf[1]);
    const float dz = mi(pj.z - pi.z, B.Lf[2], B.invLf[2]);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const bool inside = valid && r2 < S.rd2 && r2 > 0.f;
    const unsigned m = __ballot_sync(kFull, inside);
    if (inside) {
        const float rinv = rsqrtf(r2);
        fn(__popc(m & ((1u << lane) - 1u)), r2 * rinv, rinv, dx, dy, dz, j);
    }
    return __popc(m);
}
// The cutoff function fc = (cos(pi r / rd) + 1) / 2 and its derivative.
__device__ __forceinline__ void cutoff(const SurNet &S, float r, float &fc, float &dfc) {
    float sn, cs;
    __sincosf(S.pi_rd * r, &sn, &cs);
    fc = 0.5f * (cs + 1.f);
    dfc = -0.5f * S.pi_rd * sn;
}

// A block's atoms: a contiguous range (its warps' neighbourhoods overlap, so the gathered rows stay
// in L1), dealt to the warps in turn.
__device__ __forceinline__ void block_range(int a0, int a1, int &b0, int &b1) {
    const long long n = a1 - a0;
    b0 = a0 + (int)(n * blockIdx.x / gridDim.x);
    b1 = a0 + (int)(n * (blockIdx.x + 1) / gridDim.x);
}

// ---------------------------------------------------------------- descriptors
// FP32 rows G[i][k] (S.G), or, for the tensor-core network, the standardised input
// x = (G - gmu) ginv rounded to bf16 in the 128-atom tile layout the MMA reads (S.Gt):
// tile t = i / 128, row r = i % 128, column k at byte t*8192 + (r/8)*512 + (k/8)*128 + (r%8)*16 + (k%8)*2.
__global__ void __launch_bounds__(kThreads) k_sur_desc(Atoms A, SurNet S, int a0, int a1, int bf16) {
    if (eam::timed_out(A.flags)) return;
    __shared__ Stage<2> stage[kWarps];   // r, fc
    __shared__ __align__(16) __nv_bfloat16 out[kWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Stage<2> &st = stage[w];
    const float mu = S.mu0 + S.dmu * (float)lane;
    const float kx = -S.inv2w2 * kLog2e;   // b = 2^(kx a^2) fc
    const F2 nmu = pack(-mu, -mu), kx2 = pack(kx, kx);
    const float gm = S.gmu[lane], gi = S.ginv[lane];
    int b0, b1;
    block_range(a0, a1, b0, b1);
    for (int i = b0 + w; i < b1; i += kWarps) {
        const Box &B = A.boxes[ph::replica_of(A, i)];
        const float4 pi = A.posf[i];
        const int cnt = min(A.count[i], A.k_max);
        const NbrRow row = nbr_row(A, i);
        F2 G = pack(0.f, 0.f);
        for (int base = 0; base < cnt; base += 32) {
            const int np = stage_chunk(A, S, pi, B, row, cnt, base, lane,
                                       [&](int s, float r, float, float, float, float, int) {
                float fc, dfc;
                cutoff(S, r, fc, dfc);
                st.put(s, 0, r);
                st.put(s, 1, fc);
            });
            if (lane < 2 && (np & 1)) st.put(np, lane, 0.f);
            __syncwarp();
#pragma unroll 4
            for (int b = 0; b < (np + 1) >> 1; b++) {
                F2 r, fc;
                st.get2(b, 0, r, fc);
                const F2 a = add2(r, nmu);
                G = fma2(ex2_2(mul2(mul2(kx2, a), a)), fc, G);
            }
            __syncwarp();
        }
        const float g = both(G);
        if (bf16) {
            out[w][lane] = __float2bfloat16_rn((g - gm) * gi);
            __syncwarp();
            if (lane < 4) {
                const int r = i & (kSurTile - 1);
                const size_t off = (size_t)(i / kSurTile) * kSurTileBytes + (r >> 3) * 512 + lane * 128 + (r & 7) * 16;
                *reinterpret_cast<uint4 *>(S.Gt + off) = reinterpret_cast<const uint4 *>(out[w])[lane];
            }
            __syncwarp();
        } else {
            S.G[(size_t)i * kSurNb + lane] = g;
        }
    }
}

// ---------------------------------------------------------------- forces (+ kick, partials)
// Eight lanes take one pair, four channels a lane, so that a warp walks four staged pairs at a time:
// with a lane per channel the pair's seven constants went to all 32 lanes of every pair, and
// returning them from shared memory (128 bytes a cycle) bounded the kernel (83 % of the L1's
// throughput, 0.35 ms for 524,288 bcc Fe atoms); here one read serves four pairs, and four rows g_j
// come with one 16-byte load a lane.
// phi_scale > 0 (training): also phi_i = phi_scale (F_i - Fref_i) and part[0] = sum |F_i - Fref_i|^2.
// What follows an atom's force is FP64 work, which takes the FP64 pipe the same time for one active
// lane as for 32 (md_bits.cuh): a warp keeps the forces of up to 32 atoms, one per lane, and then
// finishes them together.
template <bool ENERGY, bool TRAIN>
__global__ void __launch_bounds__(kThreads, 8) k_sur_force(Atoms A, SurNet S, int a0, int a1, int kick, double half_dt,
                                                           float phi_scale) {
    if (eam::timed_out(A.flags)) return;
    constexpr bool VIRIAL = ENERGY && !TRAIN;
    __shared__ float4 P0[kWarps][32], P1[kWarps][32];   // (r, fc', -fc/w^2, u_x), (u_y, u_z, j bits, 0)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k0 = 4 * (lane & 7), grp = lane >> 3;   // this lane's channels k0 .. k0 + 3, its pair of the four
    const float mu = S.mu0 + S.dmu * (float)k0;
    const F2 nmu01 = pack(-mu, -(S.mu0 + S.dmu * (float)(k0 + 1)));
    const F2 nmu23 = pack(-(S.mu0 + S.dmu * (float)(k0 + 2)), -(S.mu0 + S.dmu * (float)(k0 + 3)));
    const float kx = -S.inv2w2 * kLog2e;
    const F2 kx2 = pack(kx, kx);
    double part[kPartials];
#pragma unroll
    for (int q = 0; q < kPartials; q++) part[q] = 0.0;
    int b0, b1;
    block_range(a0, a1, b0, b1);
    for (int i0 = b0 + w; i0 < b1; i0 += kWarps * 32) {   // up to 32 atoms i0 + kWarps q, q = 0 .. 31
        float fx = 0.f, fy = 0.f, fz = 0.f;
        float wv[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const int na = min(32, (b1 - i0 + kWarps - 1) / kWarps);
        for (int q = 0; q < na; q++) {
            const int i = i0 + kWarps * q;
            const Box &B = A.boxes[ph::replica_of(A, i)];
            const float4 pi = A.posf[i];
            const int cnt = min(A.count[i], A.k_max);
            const NbrRow row = nbr_row(A, i);
            const float4 g = __ldg(reinterpret_cast<const float4 *>(S.g + (size_t)i * kSurNb + k0));
            const F2 gi01 = pack(g.x, g.y), gi23 = pack(g.z, g.w);
            float sx = 0.f, sy = 0.f, sz = 0.f;
            float sw[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int base = 0; base < cnt; base += 32) {
                const int np = stage_chunk(A, S, pi, B, row, cnt, base, lane,
                                           [&](int s, float r, float rinv, float dx, float dy, float dz, int j) {
                    float fc, dfc;
                    cutoff(S, r, fc, dfc);
                    P0[w][s] = make_float4(r, dfc, -fc * S.invw2, dx * rinv);
                    P1[w][s] = make_float4(dy * rinv, dz * rinv, __int_as_float(j), 0.f);
                });
                const int ng = (np + 3) >> 2;
                if (lane >= np && lane < 4 * ng) {   // fill the last four up with nothing
                    P0[w][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
                    P1[w][lane] = make_float4(0.f, 0.f, __int_as_float(i), 0.f);
                }
                __syncwarp();
                // c = sum over this lane's channels of (g_ik + g_jk) b_k'(r); f += c u; the g_j rows
                // of kBatch fours are loaded before any of them is used
                constexpr int kBatch = 4;
                for (int q0 = 0; q0 < ng; q0 += kBatch) {
                    float4 gj[kBatch];
#pragma unroll
                    for (int u = 0; u < kBatch; u++) {
                        const int j = __float_as_int(P1[w][4 * min(q0 + u, ng - 1) + grp].z);
                        gj[u] = __ldg(reinterpret_cast<const float4 *>(S.g + (size_t)j * kSurNb + k0));
                    }
#pragma unroll
                    for (int u = 0; u < kBatch; u++) {
                        if (q0 + u < ng) {
                            const float4 p0 = P0[w][4 * (q0 + u) + grp], p1 = P1[w][4 * (q0 + u) + grp];
                            const F2 r = pack(p0.x, p0.x), dfc = pack(p0.y, p0.y), nw = pack(p0.z, p0.z);
                            const F2 a01 = add2(r, nmu01), a23 = add2(r, nmu23);
                            const F2 b01 = mul2(ex2_2(mul2(mul2(kx2, a01), a01)), fma2(a01, nw, dfc));   // b_k'(r)
                            const F2 b23 = mul2(ex2_2(mul2(mul2(kx2, a23), a23)), fma2(a23, nw, dfc));
                            const F2 g01 = add2(gi01, pack(gj[u].x, gj[u].y)), g23 = add2(gi23, pack(gj[u].z, gj[u].w));
                            const float c = both(fma2(g01, b01, mul2(g23, b23)));
                            sx = fmaf(c, p0.w, sx);
                            sy = fmaf(c, p1.x, sy);
                            sz = fmaf(c, p1.y, sz);
                            if constexpr (VIRIAL) {   // -1/2 c r u (x) u
                                const float h = -0.5f * c * p0.x, hx = h * p0.w, hy = h * p1.x;
                                sw[0] = fmaf(hx, p0.w, sw[0]);
                                sw[1] = fmaf(hy, p1.x, sw[1]);
                                sw[2] = fmaf(h * p1.y, p1.y, sw[2]);
                                sw[3] = fmaf(hy, p1.y, sw[3]);
                                sw[4] = fmaf(hx, p1.y, sw[4]);
                                sw[5] = fmaf(hx, p1.x, sw[5]);
                            }
                        }
                    }
                }
                __syncwarp();
            }
            const float t = warp_sum4(sx, sy, sz, VIRIAL ? sw[0] : 0.f);   // lanes 0, 1, 2, 3: x, y, z, xx
            const float tx = __shfl_sync(kFull, t, 0), ty = __shfl_sync(kFull, t, 1), tz = __shfl_sync(kFull, t, 2);
            if (lane == q) {
                fx = tx;
                fy = ty;
                fz = tz;
            }
            if constexpr (VIRIAL) {
                const float t1 = warp_sum4(sw[1], sw[2], sw[3], sw[4]), t2 = warp_sum(sw[5]);
                const float x0 = __shfl_sync(kFull, t, 3);
                if (lane == q) {
                    wv[0] = x0;
                    wv[5] = t2;
                }
#pragma unroll
                for (int v = 0; v < 4; v++) {
                    const float x = __shfl_sync(kFull, t1, v);
                    if (lane == q) wv[1 + v] = x;
                }
            }
        }
        if (lane < na) {
            const int i = i0 + kWarps * lane;
            const double dx = fx, dy = fy, dz = fz;
            A.force[i] = make_double4_32a(dx, dy, dz, 0.0);
            if (!isfinite(fx + fy + fz)) atomicOr(&A.flags->error, FLAG_NONFINITE);
            if (TRAIN) {
                const double4_32a fr = S.fref[i];
                const float ex = fx - (float)fr.x, ey = fy - (float)fr.y, ez = fz - (float)fr.z;
                S.phi[i] = make_float4(phi_scale * ex, phi_scale * ey, phi_scale * ez, 0.f);
                part[0] += (double)ex * ex + (double)ey * ey + (double)ez * ez;
            } else {
                double4_32a v = A.vel[i];
                eam::kick_and_partials(v, dx, dy, dz, half_dt, kick != 0);
                if (kick) A.vel[i] = v;
                if (ENERGY) {
                    const double m = 1.0 / (kMvv2e * v.w);
                    part[0] += A.e_atom[i];
                    part[1] += m * fma(v.x, v.x, fma(v.y, v.y, v.z * v.z));
#pragma unroll
                    for (int q = 0; q < 6; q++) part[2 + q] += wv[q];
                    part[8] += m * v.x; part[9] += m * v.y; part[10] += m * v.z;
                }
            }
        }
    }
    if (ENERGY || TRAIN) eam::block_partials(part, A.partials, A.part_stride);
}

// ---------------------------------------------------------------- tangent of the descriptors
// u_ik (standardised: times ginv_k) for the force term of the loss gradient.  The pair's projection
// t = u_ij . (phi_j - phi_i) is the same for every channel: the staging lane folds it into b'.
__global__ void __launch_bounds__(kThreads) k_sur_u(Atoms A, SurNet S, int a0, int a1) {
    __shared__ Stage<4> stage[kWarps];   // r, t fc', -t fc/w^2
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Stage<4> &st = stage[w];
    const float mu = S.mu0 + S.dmu * (float)lane;
    const float kx = -S.inv2w2 * kLog2e;
    const F2 nmu = pack(-mu, -mu), kx2 = pack(kx, kx);
    const float gi = S.ginv[lane];
    int b0, b1;
    block_range(a0, a1, b0, b1);
    for (int i = b0 + w; i < b1; i += kWarps) {
        const Box &B = A.boxes[ph::replica_of(A, i)];
        const float4 pi = A.posf[i];
        const float4 fi = S.phi[i];
        const int cnt = min(A.count[i], A.k_max);
        const NbrRow row = nbr_row(A, i);
        F2 u = pack(0.f, 0.f);
        for (int base = 0; base < cnt; base += 32) {
            const int np = stage_chunk(A, S, pi, B, row, cnt, base, lane,
                                       [&](int s, float r, float rinv, float dx, float dy, float dz, int j) {
                float fc, dfc;
                cutoff(S, r, fc, dfc);
                const float4 fj = __ldg(S.phi + j);
                const float t = dx * rinv * (fj.x - fi.x) + dy * rinv * (fj.y - fi.y) + dz * rinv * (fj.z - fi.z);
                st.put(s, 0, r);
                st.put(s, 1, t * dfc);
                st.put(s, 2, -t * (fc * S.invw2));
            });
            if (lane < 3 && (np & 1)) st.put(np, lane, 0.f);
            __syncwarp();
#pragma unroll 4
            for (int b = 0; b < (np + 1) >> 1; b++) {
                F2 r, td, tw, unused;
                st.get2(b, 0, r, td);
                st.get2(b, 2, tw, unused);
                const F2 a = add2(r, nmu);
                u = fma2(ex2_2(mul2(mul2(kx2, a), a)), fma2(a, tw, td), u);
            }
            __syncwarp();
        }
        S.u[(size_t)i * kSurNb + lane] = both(u) * gi;
    }
}

// ---------------------------------------------------------------- per-replica energy terms
// One block per replica r of [r0, r1): E_r = sum of its per-atom energies (fixed order);
// ce[2r] = 2 w_e (E_r - Eref_r) / (S N_r^2), ce[2r+1] = w_e/S ((E_r - Eref_r)/N_r)^2, S = r1 - r0.
__global__ void k_sur_frames(Atoms A, SurNet S, const int32_t *rep_off, int r0, int r1, double w_e) {
    __shared__ double sh[kThreads / 32];
    const int r = r0 + blockIdx.x;
    const int b = rep_off[r], e = rep_off[r + 1];
    double x = 0.0;
    for (int i = b + threadIdx.x; i < e; i += blockDim.x) x += A.e_atom[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        double E = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) E += sh[k];
        const double nr = (double)(e - b), ns = (double)(r1 - r0);
        const double d = E - S.eref[r];
        S.ce[2 * r] = nr > 0 ? 2.0 * w_e * d / (ns * nr * nr) : 0.0;
        S.ce[2 * r + 1] = nr > 0 ? w_e / ns * (d / nr) * (d / nr) : 0.0;
    }
}

// ---------------------------------------------------------------- descriptor statistics
// Per-block sums of G_k and G_k^2 over all atoms: part[b][k], part[b][32 + k].
__global__ void k_sur_stats(Atoms A, SurNet S, double *part) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __shared__ double sh[kWarps][2 * kSurNb];
    double s1 = 0.0, s2 = 0.0;
    for (long long i = (long long)blockIdx.x * kWarps + w; i < A.n; i += (long long)gridDim.x * kWarps) {
        const double g = S.G[i * kSurNb + lane];
        s1 += g;
        s2 += g * g;
    }
    sh[w][lane] = s1;
    sh[w][kSurNb + lane] = s2;
    __syncthreads();
    if (threadIdx.x < 2 * kSurNb) {
        double t = 0.0;
        for (int k = 0; k < kWarps; k++) t += sh[k][threadIdx.x];
        part[(size_t)blockIdx.x * 2 * kSurNb + threadIdx.x] = t;
    }
}

__global__ void k_sur_kick_drift(Atoms A, double half_dt, double dt, SkinLimit lim) {
    if (eam::timed_out(A.flags)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.n) return;
    ph::kick_drift(A, A.boxes, i, half_dt, dt, 1.0, false, lim);
}

// Rows of 32 floats from cell order back to the caller's order.
__global__ void k_sur_unsort_rows(Atoms A, const float *src, float *dst) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)A.n * kSurNb) return;
    const int i = (int)(t / kSurNb), k = (int)(t % kSurNb);
    dst[(size_t)A.id[i] * kSurNb + k] = src[t];
}

// Blocks of a gather: as many as stay resident at once (SurNet::gather, fewer for few atoms), so that
// each warp has the most atoms to finish together; at most one block per kWarps atoms.
int gather_blocks(const SurNet &S, int kernel, int n_atoms) {
    return std::max(1, std::min(blocks_for(n_atoms, kWarps), S.gather[kernel]));
}
cudaError_t resident_blocks(const void *kernel, int n_sm, int &out) {
    int per_sm = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1 || n_sm < 1) return cudaErrorInvalidConfiguration;
    out = std::min(8192, n_sm * per_sm);
    return cudaSuccess;
}

template <bool ENERGY, bool TRAIN>
cudaError_t force_t(const Atoms &A, const SurNet &S, int a0, int a1, int kick, double half_dt, float phi_scale,
                    int *rows_out, cudaStream_t s) {
    const int nb = gather_blocks(S, TRAIN ? kGatherTrain : (ENERGY ? kGatherEnergy : kGatherForce), a1 - a0);
    if (rows_out) *rows_out = nb;
    if (a1 <= a0) return cudaSuccess;
    k_sur_force<ENERGY, TRAIN><<<nb, kThreads, 0, s>>>(A, S, a0, a1, kick, half_dt, phi_scale);
    return cudaGetLastError();
}

}  // namespace

cudaError_t sur_gather_grids(SurNet &S) {
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = resident_blocks((const void *)k_sur_desc, n_sm, S.gather[kGatherDesc]);
    if (e == cudaSuccess) e = resident_blocks((const void *)k_sur_force<false, false>, n_sm, S.gather[kGatherForce]);
    if (e == cudaSuccess) e = resident_blocks((const void *)k_sur_force<true, false>, n_sm, S.gather[kGatherEnergy]);
    if (e == cudaSuccess) e = resident_blocks((const void *)k_sur_force<true, true>, n_sm, S.gather[kGatherTrain]);
    if (e == cudaSuccess) e = resident_blocks((const void *)k_sur_u, n_sm, S.gather[kGatherU]);
    return e;
}

cudaError_t launch_sur_kick_drift(const Atoms &A, double half_dt, double dt, SkinLimit lim, cudaStream_t s) {
    if (A.n == 0) return cudaSuccess;
    k_sur_kick_drift<<<blocks_for(A.n, kThreads), kThreads, 0, s>>>(A, half_dt, dt, lim);
    return cudaGetLastError();
}

cudaError_t launch_sur_descriptors(const Atoms &A, const SurNet &S, int a0, int a1, cudaStream_t s) {
    if (a1 <= a0) return cudaSuccess;
    k_sur_desc<<<gather_blocks(S, kGatherDesc, a1 - a0), kThreads, 0, s>>>(A, S, a0, a1, S.bf16);
    return cudaGetLastError();
}

cudaError_t launch_sur_force(const Atoms &A, const SurNet &S, int a0, int a1, bool kick, bool energy,
                             double half_dt, double phi_scale, int *rows_out, cudaStream_t s) {
    if (phi_scale > 0.0) return force_t<true, true>(A, S, a0, a1, 0, 0.0, (float)phi_scale, rows_out, s);
    return energy ? force_t<true, false>(A, S, a0, a1, kick, half_dt, 0.f, rows_out, s)
                  : force_t<false, false>(A, S, a0, a1, kick, half_dt, 0.f, rows_out, s);
}

cudaError_t launch_sur_u(const Atoms &A, const SurNet &S, int a0, int a1, cudaStream_t s) {
    if (a1 <= a0) return cudaSuccess;
    k_sur_u<<<gather_blocks(S, kGatherU, a1 - a0), kThreads, 0, s>>>(A, S, a0, a1);
    return cudaGetLastError();
}

cudaError_t launch_sur_frame_terms(const Atoms &A, const SurNet &S, const int32_t *rep_off, int r0, int r1,
                                   double w_e, cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    k_sur_frames<<<r1 - r0, 256, 0, s>>>(A, S, rep_off, r0, r1, w_e);
    return cudaGetLastError();
}

cudaError_t launch_sur_stats(const Atoms &A, const SurNet &S, double *part, int blocks, cudaStream_t s) {
    k_sur_stats<<<blocks, kThreads, 0, s>>>(A, S, part);
    return cudaGetLastError();
}

cudaError_t launch_sur_unsort_rows(const Atoms &A, const float *src, float *dst, cudaStream_t s) {
    if (A.n == 0) return cudaSuccess;
    k_sur_unsort_rows<<<blocks_for((long long)A.n * kSurNb, 256), 256, 0, s>>>(A, src, dst);
    return cudaGetLastError();
}

}  // namespace mdk
