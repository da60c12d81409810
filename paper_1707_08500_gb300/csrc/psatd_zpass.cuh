#pragma once
// FP32 z stage of the push (pass B of Sec. 3.2 of arXiv:1707.08500): the z
// transforms of every field, Eq. 1a/1b per mode and the inverse z transforms
// of E and B, for z lengths n = 4 N with N in {8, 12, 16, 20, 24}.
//
// A work item is a chunk of M consecutive (ky, kx) modes of one box, all z.
// Three steps, with a block barrier between them:
//
//   1  a thread takes N values at stride 4 of one pencil, does the N-point DFT
//      in registers and multiplies by the twiddles;
//   2  a thread owns a block of four z positions (frequencies k1 + N k2) of one
//      mode, all fields: the 4-point DFTs, Eq. 1 on the four modes and the
//      4-point inverse DFTs of E and B, in registers from its nine loads of
//      four values to its six stores of four;
//   3  a thread takes N values at stride 4, does the N-point inverse DFT and
//      writes the valid z planes to global memory.
//
// The next item's E and B are copied into a second buffer while the current
// item is worked on, its J and rho into their own place once step 2 is done
// with the current ones.
//
// Bound: instruction issue (54% of cycles with the 12 warps that two items and
// their second buffers leave room for; 168 registers a thread), then HBM (40%).
// A value passes through shared memory five times: in, out of and into step 1,
// out of and into step 2, out into step 3; with two balanced factors and Eq. 1
// by itself (k_pass_b) it is nine times.  64 boxes of 96^3, nine fields, a 2.9
// GB pass: 0.96 ms against 1.05 ms there.  Measured and not taken: values read
// from global memory straight into step 1 (1.28 ms: its latency is not
// covered), 128 registers (1.27 ms), coefficients pinned before step 1 (0.98
// ms), packed FP32 pairs of modes (1.3 ms: a third of the instructions then
// move registers into pairs).
#include "psatd_kernels.cuh"

namespace psatd {

// Decode work item `it` of stage B into *sd by one warp (lane: its lane
// index): the descriptor of its subdomain, range-checked.
template <typename T>
__device__ __forceinline__ void decode_b_warp(const Args<T>& a, int64_t it, SubDesc* sd, int lane) {
    int s = 0;
    if (a.per_sub[1] > 0) s = int(it / a.per_sub[1]);
    else if (lane == 0) s = find_sub<1>(a.subs, a.nsub, it);
    s = __shfl_sync(0xffffffffu, s, 0);
    const int* src = reinterpret_cast<const int*>(a.subs + s);
    int* dst = reinterpret_cast<int*>(sd);
    for (int i = lane; i < int(sizeof(SubDesc) / 4); i += 32) dst[i] = __ldg(src + i);
    __syncwarp();
    if (lane == 0) {
        const int64_t rel = it - sd->itemB;
        if (rel < 0 || (a.per_sub[1] > 0 && rel >= a.per_sub[1])) atomicOr(a.err, 1u);
    }
}

// The Eq. 1 coefficients of a mode (TAB_* order).
struct EqCoef { float C, S, Sk, omC, omCk, Dk, inv; };
__device__ __forceinline__ EqCoef ld_eq(const float* tb, int o, int NM) {
    EqCoef e;
    e.C = __ldg(tb + o);
    e.S = __ldg(tb + (o + NM));
    e.Sk = __ldg(tb + (o + 2 * NM));
    e.omC = __ldg(tb + (o + 3 * NM));
    e.omCk = __ldg(tb + (o + 4 * NM));
    e.Dk = __ldg(tb + (o + 5 * NM));
    e.inv = __ldg(tb + (o + 6 * NM));
    return e;
}

// Eq. 1a/1b on one mode in place, v = (Ex Ey Ez Bx By Bz Jx Jy Jz), element i of
// every field's NI; (sx, sy) = [k].E' for the Gauss sums.
//   E' = C E + i S khat x B - S/k J + khat [(1-C) khat.E + (S/k - dt) khat.J]
//   B' = C B - i S khat x E + i (1-C)/k khat x J
template <bool STAG, int NI>
__device__ __forceinline__ void eq1_z(const EqCoef& e, cpx<float> (*v)[NI], int i, float kx, float ky, float kz, cpx<float> px,
                                      cpx<float> py, cpx<float> pz, float& sx, float& sy) {
    using c = cpx<float>;
    const float hx = kx * e.inv, hy = ky * e.inv, hz = kz * e.inv;
    const float Sx = e.S * hx, Sy = e.S * hy, Sz = e.S * hz;
    const float Kx = e.omCk * hx, Ky = e.omCk * hy, Kz = e.omCk * hz;
    c E0 = v[0][i], E1 = v[1][i], E2 = v[2][i], B0 = v[3][i], B1 = v[4][i], B2 = v[5][i];
    c J0 = v[6][i], J1 = v[7][i], J2 = v[8][i];
    c pyz, pxz, pxy;
    if constexpr (STAG) {
        pyz = cmul(py, pz); pxz = cmul(px, pz); pxy = cmul(px, py);
        E0 = cmul(E0, px); E1 = cmul(E1, py); E2 = cmul(E2, pz);
        J0 = cmul(J0, px); J1 = cmul(J1, py); J2 = cmul(J2, pz);
        B0 = cmul(B0, pyz); B1 = cmul(B1, pxz); B2 = cmul(B2, pxy);
    }
    auto dot = [&](float a0, float a1, float a2) { return fmaf(a0, hx, fmaf(a1, hy, a2 * hz)); };
    const float lx = fmaf(e.omC, dot(E0.x, E1.x, E2.x), e.Dk * dot(J0.x, J1.x, J2.x));
    const float ly = fmaf(e.omC, dot(E0.y, E1.y, E2.y), e.Dk * dot(J0.y, J1.y, J2.y));
    // component a of E' and B' from the cyclic neighbours b, c of a:
    // (khat x F)_a = h_b F_c - h_c F_b
    auto new_e = [&](c Ea, c Bb, c Bc, c Ja, float h, float Sb, float Sc) {
        return mk(fmaf(e.C, Ea.x, fmaf(-Sb, Bc.y, fmaf(Sc, Bb.y, fmaf(-e.Sk, Ja.x, h * lx)))),
                  fmaf(e.C, Ea.y, fmaf(Sb, Bc.x, fmaf(-Sc, Bb.x, fmaf(-e.Sk, Ja.y, h * ly)))));
    };
    auto new_b = [&](c Ba, c Eb, c Ec, c Jb, c Jc, float Sb, float Sc, float Kb, float Kc) {
        return mk(fmaf(e.C, Ba.x, fmaf(Sb, Ec.y, fmaf(-Sc, Eb.y, fmaf(-Kb, Jc.y, Kc * Jb.y)))),
                  fmaf(e.C, Ba.y, fmaf(-Sb, Ec.x, fmaf(Sc, Eb.x, fmaf(Kb, Jc.x, -Kc * Jb.x)))));
    };
    c F0 = new_e(E0, B1, B2, J0, hx, Sy, Sz), F1 = new_e(E1, B2, B0, J1, hy, Sz, Sx), F2 = new_e(E2, B0, B1, J2, hz, Sx, Sy);
    c G0 = new_b(B0, E1, E2, J1, J2, Sy, Sz, Ky, Kz);
    c G1 = new_b(B1, E2, E0, J2, J0, Sz, Sx, Kz, Kx);
    c G2 = new_b(B2, E0, E1, J0, J1, Sx, Sy, Kx, Ky);
    sx = fmaf(kx, F0.x, fmaf(ky, F1.x, kz * F2.x));
    sy = fmaf(kx, F0.y, fmaf(ky, F1.y, kz * F2.y));
    if constexpr (STAG) {
        F0 = cmulc(F0, px); F1 = cmulc(F1, py); F2 = cmulc(F2, pz);
        G0 = cmulc(G0, pyz); G1 = cmulc(G1, pxz); G2 = cmulc(G2, pxy);
    }
    v[0][i] = F0; v[1][i] = F1; v[2][i] = F2;
    v[3][i] = G0; v[4][i] = G1; v[5][i] = G2;
}

// f(integral_constant<int, N>) for the first factor N: a compile-time one, or
// one of the five chosen per item (CN = 0).
template <int CN, class F>
__device__ __forceinline__ void with_n(int N, F&& f) {
    if constexpr (CN > 0) {
        f(std::integral_constant<int, CN>{});
    } else {
        if (N == 24) f(std::integral_constant<int, 24>{});
        else if (N == 20) f(std::integral_constant<int, 20>{});
        else if (N == 16) f(std::integral_constant<int, 16>{});
        else if (N == 12) f(std::integral_constant<int, 12>{});
        else f(std::integral_constant<int, 8>{});
    }
}

// Shared-memory index of element (block k1, position i of 4, mode m) of a
// pencil chunk: odd blocks swap neighbouring positions, so that the lanes of
// step 2 (M modes of consecutive blocks) fall on different banks.
template <int M>
__device__ __forceinline__ int zidx(int k1, int i, int m) { return (4 * k1 + (i ^ (k1 & 1))) * M + m; }

// Copy the chunk's pencils of `nfld` fields from field f0 on to shared memory
// (dst, field stride fs, element (k1, i) of zidx = z plane 4 k1 + i), zero past
// the ragged end of the plane; asynchronous.  LZ: the z length (0: lz).  One
// pointer step a row: a flattened loop's index arithmetic was a seventh of the
// kernel's instructions.
template <int M, int NT, int LZ>
__device__ __forceinline__ void copy_pencils(const cpx<float>* __restrict__ spec, int Q, int lz, int q0, int f0, int nfld,
                                             cpx<float>* dst, int fs) {
    constexpr int W = M / 2, R = NT / W;
    static_assert(R % 8 == 0, "rows R apart share the swap of zidx");
    const int Lz = LZ ? LZ : lz;
    const int z0 = int(threadIdx.x) / W, m = 2 * (int(threadIdx.x) % W), left = min(max(Q - q0 - m, 0), 2);
    const bool al = (Q & 1) == 0;
    cpx<float>* p0 = dst + (z0 ^ ((z0 >> 2) & 1)) * M + m;
    const cpx<float>* row = spec + (int64_t(f0) * Lz + z0) * Q + q0 + (left ? m : 0);
    const int64_t step = int64_t(R) * Q, plane = int64_t(Lz) * Q;
#pragma unroll 1
    for (int f = 0; f < nfld; ++f, p0 += fs, row += plane) {
        const cpx<float>* src = row;
        cpx<float>* p = p0;
        if (al) {
#pragma unroll
            for (int z = z0; z < Lz; z += R, src += step, p += R * M) cp_async16(p, src, 8 * left);
        } else {
#pragma unroll 1
            for (int z = z0; z < Lz; z += R, src += step, p += R * M) {
                cp_async8z(p, src, left > 0 ? 8 : 0);
                cp_async8z(p + 1, src + (left > 1 ? 1 : 0), left > 1 ? 8 : 0);
            }
        }
    }
}

// Table position of frequency k of an axis whose first factor is f1 (a
// compile-time value, or one of the three of kRegY).
template <int F1C>
__device__ __forceinline__ int z_pos(int k, int f1, int f2) {
    if constexpr (F1C > 0) return (k % F1C) * f2 + k / F1C;
    if (f1 == 12) return (k % 12) * f2 + k / 12;
    if (f1 == 10) return (k % 10) * f2 + k / 10;
    return (k % 8) * f2 + k / 8;
}

// ---- the kernel --------------------------------------------------------------
// CN: first factor N of every box (0: per item, at most 24).  NW warps: a
// thread per (k1, mode) of the longest axis, N M of them.
template <int CN, int M, bool HEAT, bool STAG, int NW, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) k_pass_z(Args<float> a) {
    constexpr int NT = NW * 32;
    constexpr int NO = HEAT ? 1 : 6;       // fields advanced (the others are sources)
    static_assert(HEAT || NT >= (CN ? CN : 24) * M, "step 2 takes one round");
    extern __shared__ __align__(16) unsigned char smraw[];
    cpx<float>* const sm = reinterpret_cast<cpx<float>*>(smraw);
    __shared__ SubDesc s_d[3];             // descriptors of the current item and the next two
    __shared__ int64_t s_it[3];            // their numbers, -1 past the last
    __shared__ float red[2 * NW];
    __shared__ tw_t<float> s_tw[CN ? 4 * CN : 96];   // w^(j r) at j N + r, j < 4, r < N
    const int warp = int(threadIdx.x) >> 5, lane = int(threadIdx.x) & 31;
    const TicketDraw<float> draw{a};
    wait_for_previous_launch();
    if (threadIdx.x == 0) {
        s_it[0] = draw.first();
        s_it[1] = s_it[0] >= 0 ? draw.next() : -1;
    }
    __syncthreads();
    if (warp < 2 && s_it[warp] >= 0) decode_b_warp(a, s_it[warp], &s_d[warp], lane);
    __syncthreads();
    int cur = 0, buf = 0, tw_of = -1;
    int64_t it = s_it[0];
    if (it >= 0) {
        const SubDesc& d = s_d[0];
        const int q0 = int(it - d.itemB) * M;
        copy_pencils<M, NT, 4 * CN>(a.spec + d.spec_off, d.q, d.L[2], q0, 0, NO, sm, d.fsB);
        copy_pencils<M, NT, 4 * CN>(a.spec + d.spec_off, d.q, d.L[2], q0, NO, a.nf - NO, sm + 2 * NO * d.fsB, d.fsB);
    }
    while (it >= 0) {
        const SubDesc& d = s_d[cur];
        const int nx = cur == 2 ? 0 : cur + 1, n2 = nx == 2 ? 0 : nx + 1;
        const int Lz = CN ? 4 * CN : d.L[2], N1 = CN ? CN : d.L[2] >> 2, Q = d.q;
        const int q0 = int(it - d.itemB) * M;
        const int mc = min(M, Q - q0);
        const int nf = a.nf, fs = d.fsB;
        cpx<float>* const X = sm + buf * NO * fs;      // E and B
        cpx<float>* const Y = sm + 2 * NO * fs;        // the sources

        // the Eq. 1 coefficients of this thread's four modes (offsets inside a
        // box's tables and spectra fit 32 bits: kZMaxElems)
        const int m2 = int(threadIdx.x) % M, k1 = int(threadIdx.x) / M;
        const bool on = k1 < N1 && m2 < mc;
        const int NM = Lz * Q;
        const int f1 = d.az.f1, f2 = d.az.f2;
        EqCoef e[4];
        float kx = 0.f, ky = 0.f, kz[4], wgt = 0.f;
        cpx<float> px, py, pz[4];
        if (!HEAT && on) {
            const int lxh = d.lxh, Ly = d.L[1], q = q0 + m2;
            const float* const tb = a.tab + d.tab_coef;
            const float* const tk = a.tab + d.tab_k;
            const int yp = q / lxh, xp = q - yp * lxh;
            kx = __ldg(tk + xp);
            ky = __ldg(tk + lxh + yp);
            wgt = xp == 0 || xp == lxh - 1 ? 1.f : 2.f;
            if constexpr (STAG) {
                px = ldg_c(a.tabc + d.tab_ph + xp);
                py = ldg_c(a.tabc + d.tab_ph + lxh + yp);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = k1 + N1 * i;             // its frequency, at table position zp
                const int zp = z_pos<CN ? split_first(4 * CN) : 0>(k, f1, f2);
                e[i] = ld_eq(tb, zp * Q + q, NM);
                kz[i] = __ldg(tk + lxh + Ly + zp);
                if constexpr (STAG) pz[i] = ldg_c(a.tabc + d.tab_ph + lxh + Ly + zp);
            }
        }
        cp_async_wait_all();
        __syncthreads();                               // this item's pencils are here; the last item's step 3 is done
        const int64_t nxt = s_it[nx];
        const SubDesc& dn = s_d[nx];
        const int qn = nxt >= 0 ? int(nxt - dn.itemB) * M : 0;
        if (nxt >= 0) copy_pencils<M, NT, 4 * CN>(a.spec + dn.spec_off, dn.q, dn.L[2], qn, 0, NO, sm + (buf ^ 1) * NO * fs, fs);
        if (threadIdx.x == 0) s_it[n2] = nxt >= 0 ? draw.next() : -1;
        if (tw_of != d.az.tw) {                        // another z length than the last item's
            tw_of = d.az.tw;
            for (int i = int(threadIdx.x); i < 4 * N1; i += NT) s_tw[i] = ld_tw(a.tw + tw_of + (i / N1) * (i % N1));
            __syncthreads();
        }

        // ---- step 1: N-point DFTs at stride 4
        with_n<CN>(N1, [&](auto nc) {
            constexpr int N = decltype(nc)::value;
            const int n1 = nf * 4 * M;
#pragma unroll 1
            for (int t = int(threadIdx.x); t < n1; t += NT) {
                const int m = t % M, j = (t / M) & 3, f = t / (4 * M);
                cpx<float>* s = f < NO ? X + f * fs : Y + (f - NO) * fs;
                cpx<float> v[N];
#pragma unroll
                for (int r = 0; r < N; ++r) v[r] = s[zidx<M>(r, j, m)];
                Dft<N, false>::run(v);
                s[zidx<M>(0, j, m)] = v[0];
#pragma unroll
                for (int r = 1; r < N; ++r) s[zidx<M>(r, j, m)] = mul_tw(v[r], s_tw[j * N + r]);
            }
        });
        __syncthreads();
        if (warp == NW - 1 && s_it[n2] >= 0) decode_b_warp(a, s_it[n2], &s_d[n2], lane);

        // ---- step 2: a block of four positions of one mode, all fields
        float g_res = 0.f, g_rho = 0.f;
        if constexpr (HEAT) {
            const float* const tb = a.tab + d.tab_coef + q0;
#pragma unroll 1
            for (int t = int(threadIdx.x); t < N1 * M; t += NT) {
                const int m = t % M, kk = t / M;
                if (m >= mc) continue;
                cpx<float> v[4], w[4];
                float c[4], g[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = kk + N1 * i, o = z_pos<CN ? split_first(4 * CN) : 0>(k, f1, f2) * Q + m;
                    c[i] = __ldg(tb + o);
                    if (nf > 1) g[i] = __ldg(tb + (o + NM));
                    v[i] = X[zidx<M>(kk, i, m)];
                }
                Dft<4, false>::run(v);
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = scale(v[i], c[i]);
                if (nf > 1) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = Y[zidx<M>(kk, i, m)];
                    Dft<4, false>::run(w);
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = mk(fmaf(w[i].x, g[i], v[i].x), fmaf(w[i].y, g[i], v[i].y));
                }
                Dft<4, true>::run(v);
                X[zidx<M>(kk, 0, m)] = v[0];
#pragma unroll
                for (int r = 1; r < 4; ++r) X[zidx<M>(kk, r, m)] = mul_tw_conj(v[r], s_tw[r * N1 + kk]);
            }
        } else {
            if (on) {
                int at[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) at[i] = zidx<M>(k1, i, m2);
                cpx<float> v[9][4];
#pragma unroll
                for (int f = 0; f < 9; ++f) {
                    const cpx<float>* s = f < 6 ? X + f * fs : Y + (f - 6) * fs;
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[f][i] = s[at[i]];
                    Dft<4, false>::run(v[f]);
                }
                float sx[4], sy[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) eq1_z<STAG>(e[i], v, i, kx, ky, kz[i], px, py, pz[i], sx[i], sy[i]);
                if (nf > 9) {
                    // |i[k].E' N - rho|^2 = (N sy + rho_x)^2 + (rho_y - N sx)^2
                    // with s = [k].E', weighted by the half-spectrum multiplicity
                    cpx<float> rho[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) rho[i] = Y[3 * fs + at[i]];
                    Dft<4, false>::run(rho);
                    const float Nfull = float(d.L[0] * d.L[1]) * float(Lz);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float rx = fmaf(sy[i], Nfull, rho[i].x), ry = fmaf(-sx[i], Nfull, rho[i].y);
                        g_res = fmaf(wgt, fmaf(rx, rx, ry * ry), g_res);
                        g_rho = fmaf(wgt, fmaf(rho[i].x, rho[i].x, rho[i].y * rho[i].y), g_rho);
                    }
                }
                const tw_t<float> w1 = s_tw[N1 + k1], w2 = s_tw[2 * N1 + k1], w3 = s_tw[3 * N1 + k1];
#pragma unroll
                for (int f = 0; f < 6; ++f) {
                    Dft<4, true>::run(v[f]);
                    cpx<float>* s = X + f * fs;
                    s[at[0]] = v[f][0];
                    s[at[1]] = mul_tw_conj(v[f][1], w1);
                    s[at[2]] = mul_tw_conj(v[f][2], w2);
                    s[at[3]] = mul_tw_conj(v[f][3], w3);
                }
            }
        }
        if constexpr (!HEAT) {
            if (nf > 9) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    g_res += __shfl_down_sync(0xffffffffu, g_res, o);
                    g_rho += __shfl_down_sync(0xffffffffu, g_rho, o);
                }
                if (lane == 0) {
                    red[warp] = g_res;
                    red[NW + warp] = g_rho;
                }
            }
        }
        __syncthreads();

        // ---- step 3: inverse DFTs, valid z planes to global memory, while the
        // next item's sources arrive
        if (nxt >= 0) copy_pencils<M, NT, 4 * CN>(a.spec + dn.spec_off, dn.q, dn.L[2], qn, NO, nf - NO, Y, fs);
        with_n<CN>(N1, [&](auto nc) {
            constexpr int N = decltype(nc)::value;
            cpx<float>* const spec = a.spec + d.spec_off + q0;
            const int n3 = NO * 4 * M;
#pragma unroll 1
            for (int t = int(threadIdx.x); t < n3; t += NT) {
                const int m = t % M, j = (t / M) & 3, f = t / (4 * M);
                if (m >= mc) continue;
                const cpx<float>* s = X + f * fs;
                cpx<float> v[N];
#pragma unroll
                for (int r = 0; r < N; ++r) v[r] = s[zidx<M>(r, j, m)];
                Dft<N, true>::run(v);
                // plane z = j + 4 r is valid for lo <= r < hi
                const int lo = (d.ngz - j + 3) >> 2, hi = (d.ngz + d.nv[2] - j + 3) >> 2;
                const int o = (f * Lz + j) * Q + m, step = 4 * Q;
#pragma unroll
                for (int r = 0; r < N; ++r)
                    if (r >= lo && r < hi) stcs_c(spec + (o + r * step), v[r]);
            }
        });
        if constexpr (!HEAT) {
            if (nf > 9 && threadIdx.x == 0) {
                float s1 = 0.f, s2 = 0.f;
                for (int i = 0; i < NW; ++i) s1 += red[i];
                for (int i = 0; i < NW; ++i) s2 += red[NW + i];
                a.gauss_part[2 * it] = s1;
                a.gauss_part[2 * it + 1] = s2;
            }
        }
        cur = nx;
        buf ^= 1;
        it = nxt;
    }
}

// ---- boxes one cell deep (2D problems): Eq. 1 alone -----------------------------
// No z transform: a thread takes its mode of all nine (ten) fields from global
// memory to registers, and back.  Bound by HBM.  k_pass_b staged the same
// values in shared memory between three block barriers: 0.236 ms on 1024 boxes
// of 96^2 with the Gauss sums (616 MB), 0.133 ms (4.6 TB/s) here.
template <bool STAG>
__global__ void __launch_bounds__(kThreads, 4) k_pass_b_flat(Args<float> a) {
    __shared__ SubDesc d;
    __shared__ float red[2 * (kThreads / 32)];
    __shared__ int64_t s_ticket[2];
    Tickets<float> tk(a, s_ticket);
    for (int64_t it = tk.current(); it >= 0; tk.advance(), it = tk.current()) {
        tk.prefetch();
        decode_item<1>(a, it, &d);
        const int M = d.chunkB, Q = d.q, lxh = d.lxh, Ly = d.L[1], nf = a.nf;
        const int q0 = int(it - d.itemB) * M, qe = min(q0 + M, Q);
        cpx<float>* const spec = a.spec + d.spec_off;
        const float* const tb = a.tab + d.tab_coef;
        const float* const k = a.tab + d.tab_k;
        const cpx<float>* const ph = a.tabc + d.tab_ph;
        const float kz = __ldg(k + lxh + Ly), Nfull = float(d.L[0] * Ly);
        float g_res = 0.f, g_rho = 0.f;
        for (int q = q0 + int(threadIdx.x); q < qe; q += kThreads) {
            cpx<float> v[9][1], rho = mk(0.f, 0.f), px, py, pz;
#pragma unroll
            for (int f = 0; f < 9; ++f) {
                const float2 w = __ldcs(reinterpret_cast<const float2*>(spec + int64_t(f) * Q + q));
                v[f][0] = mk(w.x, w.y);
            }
            if (nf > 9) {
                const float2 w = __ldcs(reinterpret_cast<const float2*>(spec + 9 * int64_t(Q) + q));
                rho = mk(w.x, w.y);
            }
            const EqCoef e = ld_eq(tb, q, Q);
            const int yp = q / lxh, xp = q - yp * lxh;
            const float kx = __ldg(k + xp), ky = __ldg(k + lxh + yp);
            if constexpr (STAG) {
                px = ldg_c(ph + xp);
                py = ldg_c(ph + lxh + yp);
                pz = ldg_c(ph + lxh + Ly);
            }
            float sx, sy;
            eq1_z<STAG>(e, v, 0, kx, ky, kz, px, py, pz, sx, sy);
#pragma unroll
            for (int f = 0; f < 6; ++f) stcs_c(spec + int64_t(f) * Q + q, v[f][0]);
            const float rx = fmaf(sy, Nfull, rho.x), ry = fmaf(-sx, Nfull, rho.y);
            const float wgt = xp == 0 || xp == lxh - 1 ? 1.f : 2.f;
            g_res = fmaf(wgt, fmaf(rx, rx, ry * ry), g_res);
            g_rho = fmaf(wgt, fmaf(rho.x, rho.x, rho.y * rho.y), g_rho);
        }
        if (nf > 9) {
            block_sum2(g_res, g_rho, red);
            if (threadIdx.x == 0) {
                a.gauss_part[2 * it] = g_res;
                a.gauss_part[2 * it + 1] = g_rho;
            }
        }
        __syncthreads();
    }
}

}  // namespace psatd
