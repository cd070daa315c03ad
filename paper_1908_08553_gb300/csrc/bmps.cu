// Boundary-MPS approximate contraction (the environment approximation the
// paper names as the way past the exact method's memory limit, Sec. 7):
// the top row of the double-layer network is a matrix product state whose
// physical legs are the rows' down legs; every further row is applied to it as
// a matrix product operator, and the grown state is compressed back to bond
// chi before the next row:
//   right to left, tensor c (a x p x b) is made right-orthonormal: the one-
//     sided Jacobi SVD of its transpose gives M = (V Sigma) U^T; U^T (numerical
//     rank k rows) stays, V Sigma is absorbed into tensor c - 1;
//   left to right, tensor c viewed as (a p) x b is cut by its SVD, the chi
//     largest singular values kept: U stays, Sigma V^T is absorbed into c + 1.
// The last row closes the state into a scalar.  Every tensor is rescaled to
// max |entry| in [1/2, 1) by an exact power of two after each row, the powers
// summed in an integer exponent.  One block contracts one network (the norm,
// or the norm with one or two Pauli operators inserted), in FP64 or FP32
// throughout (an approximation whose truncation error is far above FP32
// rounding; GB300 runs FP32 at 64 times its FP64 rate); its tensors live in a
// global-memory workspace of its own.
#include <cstdint>

#include "jacobi.cuh"
#include "tn_kernels.h"

namespace tn {

namespace {

constexpr int kBmpsThreads = 512;     // 16 warps: two column pairs of a 64-column SVD each; two blocks fit an SM
constexpr int kBmpsMaxBond = 512;     // columns of any SVD (host-checked)

template <typename T>
__device__ __forceinline__ T bmps_block_max(T v, T* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    T r = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) r = fmax(r, red[k]);
    __syncthreads();
    return r;
}

// Scale x[0..n) by 2^-e with e the frexp exponent of max |x|; returns e.
template <typename T>
__device__ int bmps_rescale(T* x, long long n, T* red) {
    T m = 0;
    for (long long k = threadIdx.x; k < n; k += blockDim.x) m = fmax(m, fabs(x[k]));
    m = bmps_block_max(m, red);
    if (!(m > T(0)) || !isfinite(m)) return 0;
    int e;
    frexp(m, &e);
    const T f = (T)ldexp(1.0, -e);
    for (long long k = threadIdx.x; k < n; k += blockDim.x) x[k] *= f;
    __syncthreads();
    return e;
}

// Singular values (column norms) of the n columns of S after block_jacobi,
// ordered: sel[0..k) = the columns with the k largest norms (ties: lower
// index), k = min(kmax, numerical rank: sigma > 1e-14 sigma_max in FP64,
// 3e-6 sigma_max in FP32).  Returns k.
template <typename T>
__device__ int bmps_select(const T* S, int m, int n, long long lds, int kmax, T* sig, int* sel, T* red) {
    // FP32 keeps values above a few units of its rounding of the largest
    const T floor_rel = sizeof(T) == 8 ? T(1e-14) : T(3e-6);
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        T s2 = 0;
        const T* cc = S + c * lds;
        for (int r = 0; r < m; ++r) s2 += cc[r] * cc[r];
        sig[c] = sqrt(s2);
    }
    __syncthreads();
    T mx = 0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) mx = fmax(mx, sig[c]);
    mx = bmps_block_max(mx, red);
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        int rank = 0;
        for (int q = 0; q < n; ++q) rank += (sig[q] > sig[c]) || (sig[q] == sig[c] && q < c);
        sel[rank] = c;
    }
    __syncthreads();
    int k = 0;
    for (int r = 0; r < n && r < kmax; ++r)
        if (sig[sel[r]] > floor_rel * mx) ++k;
    return k > 0 ? k : 1;     // a zero tensor keeps one (zero) column
}

// Double-layer tensor of site (r, c): T[(u u')(l l')(dn dn')(rt rt')] =
// sum_{p,q} A[p,u,l,dn,rt] O[p][q] A[q,u',l',dn',rt'] (O = I, X or Z).
template <typename T>
__device__ void bmps_site(const double* A, const int* d5, int op, T* Tout) {
    const int u = d5[1], l = d5[2], dn = d5[3], rt = d5[4];
    const long long half = (long long)u * l * dn * rt;
    const int U = u * u, Lg = l * l, Dn = dn * dn, R = rt * rt;
    const long long n = (long long)U * Lg * Dn * R;
    double o00 = 1, o01 = 0, o10 = 0, o11 = 1;
    if (op == 1) { o00 = 0; o01 = 1; o10 = 1; o11 = 0; }
    else if (op == 2) { o00 = -1; o01 = 0; o10 = 0; o11 = 1; }
    for (long long idx = threadIdx.x; idx < n; idx += blockDim.x) {
        long long k = idx;
        const int rr = (int)(k % R); k /= R;
        const int dd = (int)(k % Dn); k /= Dn;
        const int ll = (int)(k % Lg); k /= Lg;
        const int uu = (int)k;
        const int ua = uu / u, ub = uu % u, la = ll / l, lb = ll % l;
        const int da = dd / dn, db = dd % dn, ra = rr / rt, rb = rr % rt;
        const long long ia = (((long long)ua * l + la) * dn + da) * rt + ra;
        const long long ib = (((long long)ub * l + lb) * dn + db) * rt + rb;
        const double a0 = A[ia], a1 = A[half + ia], b0 = A[ib], b1 = A[half + ib];
        Tout[idx] = (T)(a0 * (o00 * b0 + o01 * b1) + a1 * (o10 * b0 + o11 * b1));
    }
    __syncthreads();
}

}  // namespace

long long bmps_workspace(int W, int D, int chi) {
    const long long d = (long long)D * D, B = (long long)bmps_bond_max(D, chi);
    const long long slot = B * d * B;
    return (2LL * W + 2) * slot + B * B + d * d * d * d;
}

template <typename T>
__global__ void __launch_bounds__(kBmpsThreads, 2) k_bmps(const BmpsTask* __restrict__ tasks, int smem_elems) {
    extern __shared__ __align__(16) unsigned char dyn[];
    T* const sm = reinterpret_cast<T*>(dyn);
    const BmpsTask& t = tasks[blockIdx.x];
    __shared__ int a[17];                     // a[c] = bond left of tensor c; a[0] = a[W] = 1
    __shared__ int ph[16];                    // physical (down-leg) dimension of tensor c
    __shared__ int d5[5];
    __shared__ long long soff[257];
    __shared__ T red[kBmpsThreads / 32];
    __shared__ T sig[kBmpsMaxBond];
    __shared__ int sel[kBmpsMaxBond];
    __shared__ int flag;
    const int L = t.L, W = t.W, D = t.D, chi = t.chi;
    const int d = D * D;
    const long long B = bmps_bond_max(D, chi);
    const long long slot = B * d * B;
    T* bufA = reinterpret_cast<T*>(t.ws);
    T* bufB = bufA + (long long)W * slot;
    T* S = bufB + (long long)W * slot;
    T* Tm = S + slot;
    T* V = Tm + slot;
    T* Ts = V + B * B;
    long long ex = 0;                         // power-of-two exponent of the value
    if (threadIdx.x == 0) {
        soff[0] = 0;
        for (int r = 0; r < L; ++r)
            for (int c = 0; c < W; ++c) {
                const int s = r * W + c;
                const long long n = 2LL * (r == 0 ? 1 : D) * (c == 0 ? 1 : D) * (r == L - 1 ? 1 : D) *
                                    (c == W - 1 ? 1 : D);
                soff[s + 1] = soff[s] + n;
            }
    }
    __syncthreads();
    auto site = [&](int r, int c) {
        if (threadIdx.x == 0) {
            d5[0] = 2;
            d5[1] = r == 0 ? 1 : D;
            d5[2] = c == 0 ? 1 : D;
            d5[3] = r == L - 1 ? 1 : D;
            d5[4] = c == W - 1 ? 1 : D;
        }
        __syncthreads();
        const int s = r * W + c;
        int op = 0;
        if (t.op_site[0] == s) op = t.op_code[0];
        if (t.op_site[1] == s) op = t.op_code[1];
        bmps_site(t.A + soff[s], d5, op, Ts);
    };

    // ---- row 0: M_c[a = l][p = dn][b = rt]
    for (int c = 0; c < W; ++c) {
        site(0, c);
        const long long n = (long long)d5[2] * d5[2] * d5[3] * d5[3] * d5[4] * d5[4];
        for (long long k = threadIdx.x; k < n; k += blockDim.x) bufA[c * slot + k] = Ts[k];
        if (threadIdx.x == 0) {
            a[c] = d5[2] * d5[2];
            ph[c] = d5[3] * d5[3];
            if (c == W - 1) a[W] = d5[4] * d5[4];
        }
        __syncthreads();
    }
    for (int c = 0; c < W; ++c) ex += bmps_rescale(bufA + c * slot, (long long)a[c] * ph[c] * a[c + 1], red);

    for (int r = 1; r < L; ++r) {
        // ---- apply row r: N[(a, l)][dn][(b, rt)] = sum_u M[a][u][b] T[u][l][dn][rt]
        for (int c = 0; c < W; ++c) {
            site(r, c);
            const int lu = d5[1] * d5[1], ll = d5[2] * d5[2], ld = d5[3] * d5[3], lr = d5[4] * d5[4];
            const int ac = a[c], bc = a[c + 1];
            const T* M = bufA + c * slot;
            T* N = bufB + c * slot;
            const long long n = (long long)ac * ll * ld * bc * lr;
            for (long long idx = threadIdx.x; idx < n; idx += blockDim.x) {
                long long k = idx;
                const int x = (int)(k % lr); k /= lr;
                const int bb = (int)(k % bc); k /= bc;
                const int dn = (int)(k % ld); k /= ld;
                const int l = (int)(k % ll); k /= ll;
                const int aa = (int)k;
                T v = 0;
                for (int u = 0; u < lu; ++u)
                    v += M[((long long)aa * lu + u) * bc + bb] * Ts[(((long long)u * ll + l) * ld + dn) * lr + x];
                N[idx] = v;
            }
            __syncthreads();
            if (threadIdx.x == 0) ph[c] = ld;
        }
        __syncthreads();
        // new bonds: a[c] times the double-layer dimension of the row's horizontal
        // leg between columns c - 1 and c (d inside the row, 1 at its two ends)
        if (threadIdx.x == 0)
            for (int c = 1; c < W; ++c) a[c] *= d;
        __syncthreads();
        { T* tmp = bufA; bufA = bufB; bufB = tmp; }

        if (r < L - 1) {
            // Every SVD runs in shared memory when its matrix and V fit
            // (columns at odd strides: one thread per column reads them without
            // bank conflicts): the Jacobi rounds are chains of short dependent
            // reads, 20 times shorter there than through L2.
            // ---- right to left: right-orthonormalise
            for (int c = W - 1; c >= 1; --c) {
                const int ac = a[c], p = ph[c], bc = a[c + 1];
                T* M = bufA + c * slot;
                const int m = p * bc;
                const bool in_sm = (long long)ac * ((m | 1) + (ac | 1)) <= smem_elems;
                const int lm = in_sm ? m | 1 : m, lv = in_sm ? ac | 1 : ac;
                // M row-major [a][p b] is its transpose column-major: columns = the a rows
                T* Ms = in_sm ? sm : M;
                T* Vs = in_sm ? sm + (long long)ac * lm : V;
                if (in_sm) {
                    for (int idx = threadIdx.x; idx < ac * m; idx += blockDim.x) {
                        const int j = idx / m;
                        Ms[j * lm + idx - j * m] = M[idx];
                    }
                    __syncthreads();
                }
                block_jacobi(Ms, m, ac, lm, Vs, lv, &flag);
                const int k = bmps_select(Ms, m, ac, lm, ac, sig, sel, red);
                // new tensor c: row j = column sel[j] / sigma
                T* Mo = in_sm ? M : Tm;
                for (long long idx = threadIdx.x; idx < (long long)k * m; idx += blockDim.x) {
                    const int j = (int)(idx / m), i = (int)(idx - (long long)j * m);
                    const T sg = sig[sel[j]];
                    Mo[idx] = sg > T(0) ? Ms[(long long)sel[j] * lm + i] / sg : T(0);
                }
                __syncthreads();
                // tensor c - 1 times V Sigma: [x][p'][a] -> [x][p'][j]
                const int ap = a[c - 1] * ph[c - 1];
                T* Mp = bufA + (c - 1) * slot;
                for (long long idx = threadIdx.x; idx < (long long)ap * k; idx += blockDim.x) {
                    const int xp = (int)(idx / k), j = (int)(idx - (long long)xp * k);
                    const int cj = sel[j];
                    T v = 0;
                    for (int aa = 0; aa < ac; ++aa) v += Mp[(long long)xp * ac + aa] * Vs[(long long)cj * lv + aa];
                    S[idx] = v * sig[cj];
                }
                __syncthreads();
                if (!in_sm)
                    for (long long idx = threadIdx.x; idx < (long long)k * m; idx += blockDim.x) M[idx] = Tm[idx];
                for (long long idx = threadIdx.x; idx < (long long)ap * k; idx += blockDim.x) Mp[idx] = S[idx];
                __syncthreads();
                if (threadIdx.x == 0) a[c] = k;
                __syncthreads();
            }
            // ---- left to right: truncate every bond to chi
            for (int c = 0; c < W - 1; ++c) {
                const int ac = a[c], p = ph[c], bc = a[c + 1];
                T* M = bufA + c * slot;
                const int m = ac * p;
                const bool in_sm = (long long)bc * ((m | 1) + (bc | 1)) <= smem_elems;
                const int lm = in_sm ? m | 1 : m, lv = in_sm ? bc | 1 : bc;
                T* Ms = in_sm ? sm : S;
                T* Vs = in_sm ? sm + (long long)bc * lm : V;
                for (long long idx = threadIdx.x; idx < (long long)m * bc; idx += blockDim.x) {
                    const int i = (int)(idx / bc), j = (int)(idx - (long long)i * bc);
                    Ms[(long long)j * lm + i] = M[idx];
                }
                __syncthreads();
                block_jacobi(Ms, m, bc, lm, Vs, lv, &flag);
                const int k = bmps_select(Ms, m, bc, lm, chi, sig, sel, red);
                for (long long idx = threadIdx.x; idx < (long long)m * k; idx += blockDim.x) {
                    const int i = (int)(idx / k), j = (int)(idx - (long long)i * k);
                    const T sg = sig[sel[j]];
                    M[idx] = sg > T(0) ? Ms[(long long)sel[j] * lm + i] / sg : T(0);
                }
                // tensor c + 1 := Sigma V^T (k x b) times [b][q]
                const int q = ph[c + 1] * a[c + 2];
                T* Mn = bufA + (c + 1) * slot;
                for (long long idx = threadIdx.x; idx < (long long)k * q; idx += blockDim.x) {
                    const int j = (int)(idx / q), qq = (int)(idx - (long long)j * q);
                    const int cj = sel[j];
                    T v = 0;
                    for (int bb = 0; bb < bc; ++bb) v += Vs[(long long)cj * lv + bb] * Mn[(long long)bb * q + qq];
                    Tm[idx] = sig[cj] * v;
                }
                __syncthreads();
                for (long long idx = threadIdx.x; idx < (long long)k * q; idx += blockDim.x) Mn[idx] = Tm[idx];
                __syncthreads();
                if (threadIdx.x == 0) a[c + 1] = k;
                __syncthreads();
            }
        }
        for (int c = 0; c < W; ++c) ex += bmps_rescale(bufA + c * slot, (long long)a[c] * ph[c] * a[c + 1], red);
    }

    // ---- close: every physical leg has dimension 1 now; v := v M_c
    T* v = S;
    T* w = Tm;
    if (threadIdx.x == 0) v[0] = T(1);
    __syncthreads();
    for (int c = 0; c < W; ++c) {
        const int ac = a[c], bc = a[c + 1];
        const T* M = bufA + c * slot;   // [a][1][b]
        for (int j = threadIdx.x; j < bc; j += blockDim.x) {
            T s = 0;
            for (int aa = 0; aa < ac; ++aa) s += v[aa] * M[(long long)aa * bc + j];
            w[j] = s;
        }
        __syncthreads();
        ex += bmps_rescale(w, bc, red);
        T* tmp = v; v = w; w = tmp;
    }
    if (threadIdx.x == 0) {
        int e = 0;
        const double m = frexp((double)v[0], &e);
        t.out[0] = m;
        t.out[1] = (double)(ex + e);
    }
}

// One kernel of this translation unit, for loading its module up front (preload.cpp).
const void* bmps_module_anchor() { return reinterpret_cast<const void*>(&k_bmps<double>); }

cudaError_t launch_bmps(int dt, const BmpsTask* tasks, int ntasks, int D, int chi, cudaStream_t st) {
    if (ntasks <= 0) return cudaSuccess;
    // shared memory for the largest SVD of this shape, B columns of d B rows and
    // V, when it fits (larger ones stay in the workspace, all of them: with room for only
    // the small ones a block displaces the L1 cache the others live on, 5x5 D=3 chi=9 in
    // FP32 147.6 ms against 86.7).  FP32 also at one block an SM (8x8 chi=24 172 against
    // 181 ms); FP64 gains nothing by that (chi=16 1363 against 1356).
    const long long B = bmps_bond_max(D, chi), d = (long long)D * D, es = dt == 0 ? 8 : 4;
    const long long need = B * ((d * B | 1) + (B | 1)) * es;
    const long long most = 104 * 1024, one = 200 * 1024;
    const int bytes = (int)(need <= (dt == 0 ? most : one) ? need : 0);
    const int elems = bytes / (int)es;
    // the limit belongs to the function, not to the call: always the largest, so that calls of
    // other threads cannot lower it between here and the launch
    const cudaError_t e = dt == 0 ? cudaFuncSetAttribute(k_bmps<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)one)
                                  : cudaFuncSetAttribute(k_bmps<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)one);
    if (e != cudaSuccess) return e;
    if (dt == 0) k_bmps<double><<<ntasks, kBmpsThreads, bytes, st>>>(tasks, elems);
    else k_bmps<float><<<ntasks, kBmpsThreads, bytes, st>>>(tasks, elems);
    return cudaGetLastError();
}

}  // namespace tn
