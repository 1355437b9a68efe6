// Internal declarations of libg1g2 (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/g1g2.h"

namespace g1g2 {

using cplx = double2;  // interleaved (re, im), the layout of the ABI

// ---------------------------------------------------------------------------
// Launch bookkeeping: every kernel launch goes through one of these so that a
// failed launch is turned into G1G2_ECUDA and counted.
// ---------------------------------------------------------------------------
// Optional per-kernel timing with CUDA events on the launch stream (g1g2_profile).
struct Profiler {
  bool on = false;
  std::vector<cudaEvent_t> pool;
  size_t used = 0;
  struct Rec { const char *tag; int start, stop; };
  std::vector<Rec> recs;
  int record(cudaStream_t s) {
    if (used == pool.size()) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return -1;
      pool.push_back(e);
    }
    cudaEventRecord(pool[used], s);
    return (int)used++;
  }
  void clear() { used = 0; recs.clear(); }
  ~Profiler() { for (cudaEvent_t e : pool) cudaEventDestroy(e); }
};

struct Fp64Tc;   // digit workspaces of the tensor-core FP64 products (fp64_tc.cu)

struct Launcher {
  Fp64Tc *ftc = nullptr;
  cudaStream_t stream = nullptr;
  long long *counter = nullptr;
  Profiler *prof = nullptr;
  cudaError_t err = cudaSuccess;
  const char *tag = nullptr;
  int ev_start = -1;
  void before(const char *t) {
    tag = t;
    ev_start = (prof && prof->on) ? prof->record(stream) : -1;
  }
  void after_launch() {
    if (counter) ++*counter;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess && err == cudaSuccess) err = e;
    if (prof && prof->on && ev_start >= 0) {
      const int stop = prof->record(stream);
      if (stop >= 0) prof->recs.push_back({tag ? tag : "kernel", ev_start, stop});
    }
    ev_start = -1;
  }
};

// Launch that may begin while the previous kernel of the stream still runs (programmatic dependent launch): the
// kernel calls dependent_begin() before it reads or writes global memory, which waits until the previous kernel has
// finished and then lets the next one start, so that at most two are on the chip.  At nb <= 32 the kernels of a right-hand
// side last 8 to 30 us each, of which the launch and the set-up hidden this way are about two.  (With the next one let in
// before the wait, three were in flight and took room from the first: gradients at nb = 24 1203 us instead of 1139, memory
// integral at nb = 8 8.70 ms instead of 8.35.)  The previous kernel may still write what this one reads when this one starts,
// so its inputs are not read-only for its lifetime: no __ldg and no const __restrict__ on them (the read-only path).
template <class... KArgs, class... Args>
inline void launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                             Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
__device__ __forceinline__ void dependent_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependent_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dependent_begin() {
  dependent_wait();
  dependent_launch();
}

// Generic strided complex FP64 GEMM, batched:
//   C_b[m][n] = alpha * sum_k opA(A_b[m][k]) * opB(B_b[k][n]) + beta * C_b[m][n]
// (reduce = false), or C[m][n] = alpha * sum_b sum_k ... + beta * C (reduce = true).
struct ZGemm {
  int M = 0, N = 0, K = 0, batch = 1;
  const cplx *A = nullptr; long long sa_b = 0, sa_m = 0, sa_k = 0;
  const cplx *B = nullptr; long long sb_b = 0, sb_k = 0, sb_n = 0;
  cplx *C = nullptr;       long long sc_b = 0, sc_m = 0, sc_n = 0;
  cplx alpha{1.0, 0.0};
  double beta = 0.0;
  bool conjA = false, conjB = false;
  // the operand with fewer rows (its matrix, strides and contents) is that of the previous product of this stream of
  // calls: the tensor-core form then keeps its digits
  bool same_small = false;
};
void zgemm(Launcher &L, const ZGemm &g);
void zgemm_reduce(Launcher &L, const ZGemm &g, cplx *partial, int splits);

// The same products on the tensor cores from digits of the FP64 operands (fp64_tc.cu), FP64-accurate.  Both
// return false, with nothing launched, for a product that the CUDA-core kernels take (no workspace
// in L, too small, a general alpha, both operands batched): zgemm and zgemm_reduce ask them first.
bool fp64_tc_zgemm(Launcher &L, const ZGemm &g);
bool fp64_tc_zgemm_reduce(Launcher &L, const ZGemm &g);
// Workspaces for one context of basis size nb (nullptr when they do not fit: the CUDA-core kernels then take
// every product); pair_products: nb^2 x nb^2 x nb^2 products are among them.
Fp64Tc *fp64_tc_create(int nb, bool pair_products);
// smallest basis size with a product that takes this path (factorised: products with nfac factors among them)
int fp64_tc_min_nb(bool pair_products, bool factorised);
void fp64_tc_destroy(Fp64Tc *f);
// G1G2_ETIMEOUT when one of the kernels gave up on a barrier (synchronises the stream).
int fp64_tc_error(Fp64Tc *f, cudaStream_t stream);
// Digits of at most bytes per operand at a time: larger products run in panels (one that does not hold a tile, on the CUDA cores).
void fp64_tc_set_panel(Fp64Tc *f, size_t bytes);
// Sets the error word as a kernel that gave up does.
void fp64_tc_inject_error(Fp64Tc *f, cudaStream_t stream);

// out(a0,a1,a2,a3) = beta*out + alpha*op(in(a_p0, a_p1, a_p2, a_p3)), op = conj if conj.
void permute4(Launcher &L, int nb, const cplx *in, cplx *out, const int p[4], cplx alpha, double beta,
              bool conj);

// hHF = h + f D + Wm * vec(n), Wm[(ij),(lk)] (real or complex), Eq. (h_HF).
void hf_build(Launcher &L, int nb, const void *Wm, bool wm_real, const cplx *h, const cplx *D, double f,
              const cplx *n, cplx *hhf);
// The same product in double-single arithmetic on the FP32 pipe (tensor-core forms, real w):
// Wds holds the real Wm as (hi, lo) FP32 pairs; nsplit is scratch of nb^2 float4.
void hf_build_ds(Launcher &L, int nb, const float2 *Wds, const cplx *h, const cplx *D, double f, const cplx *n,
                 float4 *nsplit, cplx *hhf);
// nbar = 1 + eta n: 1 - n for fermions (eta = -1), 1 + n for bosons (eta = +1)
void one_pm(Launcher &L, int nb, const cplx *n, double eta, cplx *nbar);
inline void one_minus(Launcher &L, int nb, const cplx *n, cplx *nbar) { one_pm(L, nb, n, -1.0, nbar); }

// RK4 stage bookkeeping shared by the G1 and G2 updates.
struct Rk4Stage {
  int stage = -1;      // -1: write k to kout; 0..3: classical RK4 stage
  double dt = 0.0;
};
// dn = -i[hHF, n] - (I + I^dag) (I may be null); then the RK4 update of (y, ys, acc)
// or a plain write of dn to kout.
void g1_update(Launcher &L, int nb, const cplx *hhf, const cplx *n, const cplx *I, Rk4Stage st,
               cplx *y, cplx *ys, cplx *acc, cplx *kout);
// dG = -i (Cb - Ab + conj(Ab^T)) with ^T the (ij)<->(kl) transpose (dG = -i Cb when Ab is
// null); RK4 update or write k.
void g2_assemble(Launcher &L, int nb, const cplx *Cb, const cplx *Ab, Rk4Stage st, cplx *y, cplx *ys,
                 cplx *acc, cplx *kout);

// One Runge-Kutta stage (or one right-hand side) in the spin-restricted Hubbard basis (on-site
// w_ijkl = U_i d(i=j=k=l)): dn and dG2 from the stage input (n, G), with the commutator over the CSR pattern
// (rp, ci) of h^HF, and their updates according to stage (see Rk4Stage).  GW: Go is the same-spin
// block, propagated in the same launch into (Sy, Sys, Sacc), each block with Pi - (Pi_lkji)^* of the reduced
// Hubbard polarisation of the other.  The outputs must not overlap the stage input.
struct HubStage {
  int nb;
  const int *rp, *ci;
  int nnz;                 // rp[nb]
  const cplx *h, *D;       // D null without a drive
  double f;
  const double *U;
  const cplx *n, *G, *Go;
  int stage;
  double dt;
  cplx *ny, *nys, *nacc, *nk, *Gy, *Gys, *Gacc, *Gk, *Sy, *Sys, *Sacc;
};
void hubbard_stage(Launcher &L, const HubStage &p);

// Observables.
// red[0..] = {Re Tr(h n), Re Tr((hHF-h(t)) n), Re Tr n, Re Tr(D n)} for state n;
void obs_one_body(Launcher &L, int nb, const cplx *h, const cplx *D, double f, const cplx *hhf,
                  const cplx *n, double *red);
// red[0] = Re sum W[(ij),(kl)] G[(kl),(ij)], red[1] = count of non-finite entries of G.
void obs_two_body(Launcher &L, int nb, const cplx *W, const cplx *G, double *partials, double *red);
// W_acc += coeff * Re Tr(D n)
void accumulate_work(Launcher &L, int nb, const cplx *D, const cplx *n, double coeff, double *W_acc);
// out[s] = double occupancy of site s (spin-orbital index 2 s + spin); eta the statistics sign.
void double_occ(Launcher &L, int nb, const cplx *n, const cplx *G, double eta, double *out);
// count non-finite entries of x (length len) into *cnt (double, accumulated)
void count_nonfinite(Launcher &L, const cplx *x, long long len, double *cnt);

// Adjoint helpers: out = alpha x + beta y (y may be null); out = c (Y + Y^dag);
// acc += coeff * Re sum conj(x) y; out (+)= Wm^T x (adjoint of the Hartree-Fock build).
void zaxpby(Launcher &L, long long n, cplx alpha, const cplx *x, cplx beta, const cplx *y, cplx *out);
void tconj_add(Launcher &L, int nb, cplx c, const cplx *Y, cplx *out);
void herm_sum(Launcher &L, int nb, cplx c, const cplx *a, cplx *out);
void real_dot_acc(Launcher &L, long long n, const cplx *x, const cplx *y, double coeff, double *partials, double *acc);
// out = i (A B - B A) for nb x nb matrices
void commutator_i(Launcher &L, int nb, const cplx *A, const cplx *B, cplx *out);
void hf_build_t(Launcher &L, int nb, const void *Wm, bool wm_real, const cplx *x, cplx *out, bool accumulate);
// Cotangent of w through the Hartree-Fock matrix Wm[(ij),(lk)] = w_ikjl + eta w_iklj given the
// cotangent x of h^HF at the state n: wbar_abcd += c (x_ac conj(n_db) + eta x_ad conj(n_cb)).
void hf_wbar(Launcher &L, int nb, const cplx *x, const cplx *n, double c, double eta, cplx *wbar);
// out = projection of X onto the symmetries of w: (X + X_jilk + conj(X_klij) + conj(X_lkji)) / 4.
void w_symmetrize(Launcher &L, int nb, const cplx *X, cplx *out);

// Memory-integral HF-GKBA (nb <= kPairMaxNb).  pair_rotate: out_ab = sum_pq M_ap M_bq X_pq on the first or second index
// pair of an nb^4 tensor, M from S by form, X the tensor in or (from_a, second pair) i (in - in^dag).
// trapezoid_sum: dt times the trapezoid sum of npoints >= 2 tensors of length len.  mean_collision: h^HF
// and I of Eqs. (h_HF), (eom_gone-I).  heun_update: (n_out, u_out) = (n0, u0) + c1 (dn_prev, du_prev) +
// c2 (dn, du), the derivatives evaluated at (n, u).  *cnt += number of nonzero entries of x.
constexpr int kPairMaxNb = 32;
enum PairForm : int { kPairPlain, kPairAdj, kPairOnePlus, kPairTrans, kPairConj };
void pair_rotate(Launcher &L, int nb, bool second, bool from_a, const cplx *in, const cplx *S, PairForm form, double eta,
                 cplx *out);
void trapezoid_sum(Launcher &L, long long len, int npoints, const cplx *x, double dt, cplx *out);
void mean_collision(Launcher &L, int nb, const void *Wm, bool wm_real, const cplx *h, const cplx *n, const cplx *wP,
                    const cplx *G, cplx *hhf, cplx *I);
void heun_update(Launcher &L, int nb, const cplx *hhf, const cplx *n, const cplx *u, const cplx *I, const cplx *n0,
                 const cplx *u0, const cplx *dn_prev, const cplx *du_prev, double c1, double c2, cplx *dn, cplx *du,
                 cplx *n_out, cplx *u_out);
void count_nonzero(Launcher &L, const cplx *x, long long len, double *cnt);

// Measured FP64 FMA rate of the current device in TFLOP/s (eight independent DFMA chains
// per thread, best of three timed launches after two untimed ones); *err != 0 on a CUDA failure.
double dfma_rate(cudaStream_t stream, int *err);

// Text returned by g1g2_last_error_detail on this thread.
void set_error_detail(const std::string &what);

}  // namespace g1g2
