// Reverse mode: the sweep over the tapes (see grf_adjoint.cu), in a translation unit of its own.
#include "grf_adjoint.cuh"

namespace grf {

// Reverse sweep of this column's tape: node adjoints are consumed (reset to zero) as they are
// propagated, so the column is clean for its next point.
//
// What bounds it: each column is a chain of entries, 24 bytes and 2.5 operands each. A read-modify-write of an
// operand's adjoint in global memory is a link of that chain. Contributions to the last kWindow entries (36% at
// 16 entries, half at 100) go to a window in shared memory instead, and the others are added by the memory
// (atomicAdd without a result: a column is one thread's, so the order is the program's; the product is rounded
// before the sum, 6-8% more rounding in the sweep than with fma, where plain read-modify-writes take 16% more time).
// An entry's adjoint is its window slot plus what farther entries left in global memory, which is final kWindow
// entries ahead, so entries and those adjoints are loaded kAhead entries before they are used. Comparisons with
// zero are taken on the integer pipe: the FP64 pipe, 16 clocks an instruction, is the next bound.
constexpr int kWindow = 16, kAhead = 4;

__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }

__device__ __forceinline__ void rev_sweep(const grf_rev::Tape& tape, int entries, long long col, double (*win)[kSweepThreads]) {
    const long long S = tape.stride;
    double* __restrict__ adj = tape.adj + col;
    const double2* __restrict__ w = tape.w + col;
    const ushort4* __restrict__ ix = tape.ix + col;
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 0; k < kWindow; ++k) win[k][t] = 0.0;
    double2 pw[kAhead];
    ushort4 po[kAhead];
    double pg[kAhead];
    auto fetch = [&](int k, int n) {
        if (n < 0) return;
        pw[k] = __ldcs(&w[n * S]);
        po[k] = __ldcs(&ix[n * S]);
        pg[k] = __ldcg(&adj[(kNLeaf + n) * S]);
    };
#pragma unroll
    for (int k = 0; k < kAhead; ++k) fetch(k, entries - 1 - k);
#pragma unroll 1
    for (int n0 = entries - 1; n0 >= 0; n0 -= kAhead) {
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int n = n0 - k;
            if (n < 0) break;
            const double2 pc = pw[k];
            const ushort4 oc = po[k];
            const double far = pg[k];
            fetch(k, n - kAhead);
            double g = win[n % kWindow][t];
            win[n % kWindow][t] = 0.0;  // the slot's next node is kWindow entries back
            if (nonzero(far)) {
                g += far;
                adj[(kNLeaf + n) * S] = 0.0;
            }
            if (!nonzero(g)) continue;
            auto give = [&](unsigned short o, double p) {
                if (o == grf_rev::kNone) return;
                const int m = (int)o - kNLeaf;  // its entry, negative for a leaf
                if (m >= 0 && m > n - kWindow) {
                    win[m % kWindow][t] = fma(p, g, win[m % kWindow][t]);
                } else {
                    atomicAdd(&adj[o * S], p * g);
                }
            };
            give(oc.x, pc.x);
            give(oc.y, pc.y);
            give(oc.z, 1.0);
        }
    }
}

// Sweeps tape column col (point q0 + col) and hands the leaves' adjoints to the stage's outputs:
// the values' to vbar / unbar / abar, the derivative and KO sums' to G (with periodic images),
// lambda's and g2's to the column's sums.
__global__ void __launch_bounds__(kSweepThreads, 7) adj_sweep_kernel(Geom g, AdjArgs a, grf_rev::Tape tape, int STAGE, long long q0) {
    const long long col = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long q = q0 + col;
    if (col >= tape.stride || q >= a.npts) return;
    double* adj = tape.adj;
    auto take = [&](int leaf) {
        const long long o = leaf * tape.stride + col;
        const double x = __ldcg(&adj[o]);
        adj[o] = 0.0;
        return x;
    };
    __shared__ double win[kWindow][kSweepThreads];
    rev_sweep(tape, a.count[col], col, win);
    const long long nxy = (long long)g.nx * g.ny;
    const int k = (int)(q / nxy);
    const long long rem = q - (long long)k * nxy;
    const int j = (int)(rem / g.nx), i = (int)(rem - (long long)j * g.nx);
    const long long p = gidx(g, i + NG, j + NG, k + NG);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        const long long o = f * g.fstride + p;
        const double vb = take(kLV + f);
        if (STAGE == 0) {
            a.unbar[o] += vb;
        } else {
            a.vbar[o] = vb;
            const double ub = take(kLUN + f);
            if (STAGE == 3) a.unbar[o] = ub;
            else a.unbar[o] += ub;
        }
        if (STAGE == 3) a.abar[o] = take(kLACC + f);
        store_with_images(g, a.G, kGKO + f, i, j, k, take(kLKO + f));
    }
#pragma unroll 1
    for (int m = 0; m < 72; ++m) store_with_images(g, a.G, m, i, j, k, take(kLD1 + m));
#pragma unroll 1
    for (int m = 0; m < 72; ++m) store_with_images(g, a.G, kGD2 + m, i, j, k, take(kLD2 + m));
    a.pbar[2 * col] += take(kLLAM);
    a.pbar[2 * col + 1] += take(kLG2);
}

void launch_adj_sweep(const Geom& g, const AdjArgs& a, const grf_rev::Tape& tape, int stage, long long q0, cudaStream_t st) {
    const int blocks = (int)((tape.stride + kSweepThreads - 1) / kSweepThreads);
    adj_sweep_kernel<<<blocks, kSweepThreads, 0, st>>>(g, a, tape, stage, q0);
}

}  // namespace grf
