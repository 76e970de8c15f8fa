// PM engine: memory plan and launch sequences of the forward model (Sec. 2) and of the
// discrete adjoint with reverse time integration (Sec. 3.5-3.6), templated on the real
// type.  Included once per precision.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "cosmo.h"
#include "pm_internal.h"
#include "pm_engine.h"
#include "pm_kernels.cuh"
#include "bin_kernels.cuh"
#include "deposit_r2c.cuh"

namespace pmgb {

#define PMGB_CK(call)                                   \
  do {                                                  \
    cudaError_t e_ = (call);                            \
    if (e_ != cudaSuccess) { set_cuda_error(e_); return PM_ERR_CUDA; } \
  } while (0)
#define PMGB_RET(call)                                  \
  do {                                                  \
    int r_ = (call);                                    \
    if (r_ != PM_OK) return r_;                         \
  } while (0)

static inline int ilog2(long long v) { int r = 0; while ((1LL << r) < v) ++r; return r; }

// Optional per-category CUDA-event timing of the engine's launches on its stream, and a
// count of the kernels it launched.
enum ProfCat { P_SCATTER = 0, P_X_R2C, P_COLS, P_Z_FORCE, P_Z_ADJ, P_X_C2R, P_GATHER_FWD, P_GATHER_ADJ, P_OTHER, P_NCAT };

struct Prof {
  bool on = false;
  struct Rec { int cat; cudaEvent_t a, b; };
  std::vector<cudaEvent_t> pool;
  size_t used = 0;
  std::vector<Rec> recs;
  double ms[P_NCAT] = {};
  long long launches[P_NCAT] = {};
  cudaEvent_t cur = nullptr;
  cudaEvent_t get() {
    if (used == pool.size()) {
      cudaEvent_t e;
      cudaEventCreate(&e);
      pool.push_back(e);
    }
    return pool[used++];
  }
  void begin(cudaStream_t st, int cat, int nk) {
    launches[cat] += nk;
    if (!on) return;
    cur = get();
    cudaEventRecord(cur, st);
  }
  void end(cudaStream_t st, int cat) {
    if (!on) return;
    cudaEvent_t b = get();
    cudaEventRecord(b, st);
    recs.push_back(Rec{cat, cur, b});
  }
  int read(cudaStream_t st, double* ms_out, long long* n_out) {
    cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return PM_ERR_CUDA;
    for (const Rec& r : recs) {
      float t = 0.f;
      cudaEventElapsedTime(&t, r.a, r.b);
      ms[r.cat] += t;
    }
    recs.clear();
    used = 0;
    for (int c = 0; c < P_NCAT; ++c) {
      if (ms_out) ms_out[c] = ms[c];
      if (n_out) n_out[c] = launches[c];
      ms[c] = 0.0;
      launches[c] = 0;
    }
    return PM_OK;
  }
  ~Prof() {
    for (cudaEvent_t e : pool) cudaEventDestroy(e);
  }
};

template <typename T>
class Engine : public EngineBase {
 public:
  using C = cx_t<T>;

  ~Engine() override {
    if (st_) cudaStreamSynchronize(st_);
    if (cp_st_) {
      cudaStreamSynchronize(cp_st_);
      cudaStreamDestroy(cp_st_);
    }
    if (cp_in_) cudaEventDestroy(cp_in_);
    if (cp_done_) cudaEventDestroy(cp_done_);
    if (graph_exec_) cudaGraphExecDestroy(graph_exec_);
    for (void* p : allocs_) cudaFree(p);
    if (err_host_) cudaFreeHost(err_host_);
    live_bytes_add(-bytes_);
  }

  int check() override { return device_error(); }
  void set_first_wait(int spins) override { first_wait_ = spins; }

  long long scratch_bytes() const override { return bytes_; }

  int profile(int enable) override {
    PMGB_RET(prof_.read(st_, nullptr, nullptr));
    prof_.on = enable != 0;
    return PM_OK;
  }
  int profile_read(double* ms, long long* launches) override {
    PMGB_RET(prof_.read(st_, ms, launches));
    return device_error();
  }
  // PM_ERR_TIMEOUT if a bounded device wait gave up since the last check (clears the flag)
  int device_error() {
    PMGB_CK(cudaStreamSynchronize(st_));
    volatile int* flag = err_host_;
    if (*flag) {
      *flag = 0;
      return PM_ERR_TIMEOUT;
    }
    return PM_OK;
  }

  int init(const pm_config* cfg, const double* theta, const void* omega, cudaStream_t st) {
    cfg_ = *cfg;
    st_ = st;
    B_ = cfg->batch;
    np_ = cfg->n_ptcl;
    nm_ = cfg->n_mesh;
    n_ = cfg->n_steps;
    N_ = (long long)np_ * np_ * np_;
    M_ = (long long)nm_ * nm_ * nm_;
    mass_ = (T)((double)M_ / (double)N_);
    geo_.lg_np = ilog2(np_);
    geo_.np = np_;
    geo_.nm = nm_;
    geo_.ratio = nm_ / np_;
    geo_.inv_l = (T)(nm_ / cfg->box);
    geo_.N = N_;
    geo_.M = M_;
    lgN_ = ilog2(N_);
    e_d_ = fixed_top<T>(lgN_);
    {
      int dev = 0;
      PMGB_CK(cudaGetDevice(&dev));
      PMGB_CK(cudaDeviceGetAttribute(&nsm_, cudaDevAttrMultiProcessorCount, dev));
    }
    // particle loops (grid-stride): wave_grid; G_ is also the number of per-block partial sums of
    // the adjoint gather, Go_ of the other reductions over particles, whose kernels need few
    // registers and take more blocks (k_adjoint_init at 128^3 particles: 304 blocks 52 us, 1024 36)
    hf_ = cfg->half_force != 0 && sizeof(T) == 4;
    G_ = wave_grid((const void*)gather_adj_fn(), N_, true);
    Go_ = (int)std::min<long long>((N_ + kPtclThreads - 1) / kPtclThreads, kMaxRedBlocks);
    Gf_ = wave_grid((const void*)gather_fwd_fn(), N_);
    // The operators' gathers need few registers.  At 1024^3 (a 17 GB force mesh) more than two
    // blocks per SM in flight span more pages than the address translation holds: force 28.9 ->
    // 24.4 ms, force VJP 53.2 -> 47.2 ms with two; at 512^3 two are 1% slower than all that fit.
    const int most = nm_ >= 1024 ? 2 * nsm_ : kMaxRedBlocks;
    Gof_ = std::min(most, wave_grid((const void*)gather_fwd_fn<true>(), N_));
    Goa_ = std::min(most, wave_grid((const void*)gather_adj_fn<true>(), N_));
    Gpm_ = wave_grid((const void*)k_pi_max<T>, N_);
    Gc_ = wave_grid((const void*)k_bin_count<T>, N_);
    Gb1_ = wave_grid((const void*)k_bin_fill<T, 1>, N_);
    Gb4_ = wave_grid((const void*)k_bin_fill<T, 4>, N_);
    Gi_ = (int)std::max<long long>(1, std::min<long long>((N_ + 255) / 256, 8LL * nsm_ / std::min(B_, 8)));   // lattice loops
    Gm_ = (int)std::min<long long>((M_ + kPtclThreads - 1) / kPtclThreads, kMaxRedBlocks);
    Gz_ = (int)std::min<long long>((spec_len_cx(np_) + kPtclThreads - 1) / kPtclThreads, kMaxRedBlocks);
    const long long pv = (long long)B_ * 3 * N_;
    const long long sl = (long long)B_ * spec_len_cx(nm_);
    PMGB_RET(alloc(&s_, pv));
    PMGB_RET(alloc(&p_, pv));
    PMGB_RET(alloc(&a_, pv));
    PMGB_RET(alloc(&xi_, pv));
    PMGB_RET(alloc(&pi_, pv));
    PMGB_RET(alloc(&s1_, pv));
    lpt2_ = cfg->lpt_order == 2;
    if (lpt2_) PMGB_RET(alloc(&s2_, pv));
    PMGB_RET(alloc(&omega_, (long long)B_ * N_));
    // particle bins of the mesh-tile assignment (bin_kernels.cuh)
    PMGB_RET(bin_setup());
    if (small_rule(1) || small_rule(4)) {
      // sums of the small deposits, kept zero between calls
      const long long n = (small_rule(4) ? 4 : 1) * (long long)B_ * M_;
      PMGB_RET(alloc(&sacc_, n));
      PMGB_CK(cudaMemsetAsync(sacc_, 0, sizeof(long long) * n, st_));
    }
    for (int q = 0; q < 7; ++q) PMGB_RET(alloc(&spec_[q], sl));
    PMGB_RET(alloc(&dens_, (long long)B_ * M_));
    PMGB_RET(alloc(&fvec_, (long long)B_ * M_));
    if (hf_) PMGB_RET(alloc(&fexp_, (long long)B_ * nm_ * nm_));   // int8 exponent quadruple per row
    if (cfg->fixed_state) {
      PMGB_RET(alloc(&fix_u_, pv));
      PMGB_RET(alloc(&fix_w_, pv));
      const double l = cfg->box / nm_;
      fx_.u = fix_u_;
      fx_.w = fix_w_;
      fx_.to_w = (T)(std::ldexp(1.0, kFixEP) / l);
      fx_.from_u = (T)(l * std::ldexp(1.0, -kFixES));
      fx_.from_w = (T)(l * std::ldexp(1.0, -kFixEP));
      fx_.w_cells = (T)std::ldexp(1.0, -kFixEP);
      fx_.du = (T)std::ldexp(1.0, kFixES);
      fix_to_u_ = (T)(std::ldexp(1.0, kFixES) / l);
    }
    if (cfg->ckpt_every > 0) {
      nck_ = (n_ + cfg->ckpt_every - 1) / cfg->ckpt_every;
      PMGB_RET(alloc(&ck_s_, pv * nck_));
      PMGB_RET(alloc(&ck_p_, pv * nck_));
    }
    // TMA-staged column passes for the mesh-size spectra (nsm_: set above)
    // TMA-staged column passes for the mesh sizes that have them (PMGB_TMA=0 starts with
    // the unstaged form; pm_set_tuning and pm_autotune switch between the two)
    const char* env = getenv("PMGB_TMA");
    tune_.tma_columns = (env && env[0] == '0' && spec_zb(nm_) <= 1) ? 0 : 1;
    apply_tuning();
    tune_.tma_columns = use_tma_ ? 1 : 0;
    // the error flag lies in host memory that the device writes (only when a wait gives up), so
    // that a check is the synchronisation alone, without a copy
    if (!alloc_gate()) return PM_ERR_OOM;
    if (cudaError_t e = cudaHostAlloc((void**)&err_host_, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable)) {
      set_cuda_error(e);
      cudaGetLastError();
      return PM_ERR_OOM;
    }
    *err_host_ = 0;
    PMGB_CK(cudaHostGetDevicePointer((void**)&dev_err_, err_host_, 0));
    if (tma_supported(nm_))
      for (int q = 0; q < 7; ++q) PMGB_RET(make_spec_tensor_maps<T>(nm_, B_, spec_[q], &tmy_[q], &tmz_[q], &tmf_[q]));
    PMGB_CK(cudaMemcpyAsync(omega_, omega, sizeof(T) * B_ * N_, cudaMemcpyDeviceToDevice, st_));
    PMGB_RET(tables(theta));
    return PM_OK;
  }

  // ------------------------------------------------------------------ forward
  int forward(void* disp, void* mom, void* dens) override {
    counted_ = false;
    prof_.begin(st_, P_OTHER, lpt2_ ? 8 + 18 : 8);
    PMGB_RET(initial_conditions());
    prof_.end(st_, P_OTHER);
    for (int j = 0; j <= n_; ++j) {
      const int q = snap_of(j);
      PMGB_RET(force_chain(s_, nullptr, j == n_ || (q >= 0 && snap_dens_)));
      if (q >= 0 && snap_disp_)
        PMGB_CK(cudaMemcpyAsync(snap_disp_ + (long long)q * B_ * 3 * N_, s_, sizeof(T) * B_ * 3 * N_,
                                cudaMemcpyDeviceToDevice, st_));
      if (q >= 0 && snap_dens_)
        PMGB_CK(cudaMemcpyAsync(snap_dens_ + (long long)q * B_ * M_, dens_, sizeof(T) * B_ * M_,
                                cudaMemcpyDeviceToDevice, st_));
      T* cks = nullptr;
      T* ckp = nullptr;
      if (nck_ && j < n_ && j % cfg_.ckpt_every == 0) {
        cks = ck_s_ + (long long)(j / cfg_.ckpt_every) * B_ * 3 * N_;
        ckp = ck_p_ + (long long)(j / cfg_.ckpt_every) * B_ * 3 * N_;
      }
      const long long fis = 2 * spec_len_cx(nm_);
      StepCoef<T> sc{fkA_, fkB_, fdr_};
      T* snap_p = (q >= 0 && snap_mom_) ? snap_mom_ + (long long)q * B_ * 3 * N_ : nullptr;
      prof_.begin(st_, P_GATHER_FWD, 1);
      // the bins of the next step's deposit are counted at the new positions
      const bool count = j < n_ && !small_deposit(false);
      gather_fwd_fn()<<<dim3(Gf_, B_), kPtclThreads, 0, st_>>>(geo_, s_, p_, j == n_ ? a_ : nullptr, fvec_, fexp_, sc,
                                                              j, n_ + 1, cks, ckp, fused1_ ? bgf1_ : bg1_,
                                                              count ? bcount_ : nullptr, bkeys_, snap_p, fx_);
      counted_ = count;
      prof_.end(st_, P_GATHER_FWD);
      PMGB_CK(cudaGetLastError());
      // states observed between steps j and j + 1, from (s_{j+1}, p_{j+1/2})
      for (size_t k = 0; k < interp_.size(); ++k)
        if (interp_[k].j == j) PMGB_RET(interp_forward((int)k));
    }
    if (disp) PMGB_CK(cudaMemcpyAsync(disp, s_, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    if (mom) PMGB_CK(cudaMemcpyAsync(mom, p_, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    if (dens) PMGB_CK(cudaMemcpyAsync(dens, dens_, sizeof(T) * B_ * M_, cudaMemcpyDeviceToDevice, st_));
    have_fwd_ = true;
    have_dens_ = true;
    return PM_OK;
  }

  int eval_device(const void* target, double* loss, void* gw, double* gt) {
    PMGB_RET(forward(nullptr, nullptr, nullptr));
    PMGB_RET(loss_mse_dev(target, djdd_));
    if (loss) PMGB_CK(cudaMemcpyAsync(loss, scal_, sizeof(double) * B_, cudaMemcpyDeviceToDevice, st_));
    PMGB_RET(adjoint(djdd_, nullptr, nullptr, gw, gt));
    return PM_OK;
  }

  int loss_mse_dev(const void* target, void* djdd) {
    if (!have_fwd_) return PM_ERR_STATE;
    prof_.begin(st_, P_OTHER, 2);
    k_mse<T><<<dim3(Gm_, B_), kPtclThreads, 0, st_>>>(dens_, (const T*)target, (T*)djdd, M_, part_);
    PMGB_CK(cudaGetLastError());
    k_sum_partials<<<B_, 256, 0, st_>>>(part_, Gm_, scal_, 1.0 / (double)M_);
    prof_.end(st_, P_OTHER);
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  int loss_mse(const void* target, double* loss, void* djdd) override {
    PMGB_RET(loss_mse_dev(target, djdd));
    if (loss) {
      PMGB_CK(cudaMemcpyAsync(loss, scal_, sizeof(double) * B_, cudaMemcpyDefault, st_));
      if (is_host(loss)) return device_error();
    }
    return PM_OK;
  }

  // ------------------------------------------------------------------ adjoint
  int adjoint(const void* djdd, const void* djdx, const void* djdp, void* djdw, double* djdth) override {
    counted_ = false;
    if (!have_fwd_) return PM_ERR_STATE;
    PMGB_CK(cudaMemsetAsync(pimax_, 0, sizeof(unsigned) * 3 * B_, st_));
    const int nobs = n_ + 1 + (int)interp_.size();   // theta-term slots of the observations
    const bool obs_theta = snap_gmom_ || (!interp_.empty() && (interp_gdisp_ || interp_gdens_));
    if (obs_theta) PMGB_CK(cudaMemsetAsync(obs_part_, 0, sizeof(double) * nobs * B_ * Go_, st_));
    prof_.begin(st_, P_OTHER, 1);
    k_adjoint_init<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(geo_, mass_, s_, (const T*)djdd, (const T*)djdx,
                                                              (const T*)djdp, xi_, pi_, pimax_);
    prof_.end(st_, P_OTHER);
    PMGB_CK(cudaGetLastError());
    const long long fis = 2 * spec_len_cx(nm_);
    for (int j = n_; j >= 0; --j) {
      // cotangents of an observed state j enter xi while the positions are x_j
      const int q = snap_of(j);
      if (q >= 0 && (snap_gdisp_ || snap_gdens_)) {
        prof_.begin(st_, P_OTHER, 1);
        k_obs_cotangent<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(
            geo_, mass_, s_, snap_gdens_ ? snap_gdens_ + (long long)q * B_ * M_ : nullptr,
            snap_gdisp_ ? snap_gdisp_ + (long long)q * B_ * 3 * N_ : nullptr, xi_);
        prof_.end(st_, P_OTHER);
        PMGB_CK(cudaGetLastError());
      }
      // positions observed between steps j and j + 1: (s_j, p_{j+1/2}) are held now
      for (size_t k = 0; k < interp_.size(); ++k)
        if (interp_[k].j == j && (interp_gdisp_ || interp_gdens_)) {
          prof_.begin(st_, P_OTHER, 1);
          k_obs_interp<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(
              geo_, mass_, s_, p_, obs_fac_ + (long long)k * B_,
              interp_gdens_ ? interp_gdens_ + (long long)k * B_ * M_ : nullptr,
              interp_gdisp_ ? interp_gdisp_ + (long long)k * B_ * 3 * N_ : nullptr, xi_, pi_,
              obs_part_ + (long long)(n_ + 1 + k) * B_ * Go_, pimax_);
          prof_.end(st_, P_OTHER);
          PMGB_CK(cudaGetLastError());
        }
      // a momentum observed at step j: its share c of the cotangent enters pi before the
      // force VJP, the rest after the reverse step
      const T* vmom = (q >= 0 && snap_gmom_) ? snap_gmom_ + (long long)q * B_ * 3 * N_ : nullptr;
      if (vmom) {
        prof_.begin(st_, P_OTHER, 1);
        k_obs_momentum<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(geo_, pi_, vmom, obs_c_, j, n_ + 1, 0, nullptr,
                                                                  nullptr, pimax_);
        prof_.end(st_, P_OTHER);
        PMGB_CK(cudaGetLastError());
      }
      PMGB_RET(force_chain(s_, pi_, false));
      const T* ckp = nullptr;
      const T* cks = nullptr;
      if (nck_) {
        if (j < n_ && j % cfg_.ckpt_every == 0) ckp = ck_p_ + (long long)(j / cfg_.ckpt_every) * B_ * 3 * N_;
        if (j >= 1 && (j - 1) % cfg_.ckpt_every == 0)
          cks = ck_s_ + (long long)((j - 1) / cfg_.ckpt_every) * B_ * 3 * N_;
      }
      StepCoef<T> sc{rkA_, rkB_, rdr_};
      double* ppa = part_ + (long long)(2 * j) * B_ * G_;
      double* pxp = part_ + (long long)(2 * j + 1) * B_ * G_;
      const bool count = j > 0 && !small_deposit(true);
      prof_.begin(st_, P_GATHER_ADJ, 1);
      gather_adj_fn()<<<dim3(G_, B_), kPtclThreads, 0, st_>>>(geo_, mass_, s_, p_, xi_, pi_, vmom ? a_ : nullptr,
                                                              nullptr, fvec_, fexp_, sc, j, n_ + 1, ckp, cks, ppa, pxp,
                                                              pimax_, fused4_ ? bgf4_ : bg4_,
                                                              count ? bcount_ : nullptr, bkeys_, fx_);
      counted_ = count;
      prof_.end(st_, P_GATHER_ADJ);
      PMGB_CK(cudaGetLastError());
      if (vmom) {
        prof_.begin(st_, P_OTHER, 1);
        k_obs_momentum<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(geo_, pi_, vmom, obs_c_, j, n_ + 1, 1, a_,
                                                                  obs_part_ + (long long)j * B_ * Go_, pimax_);
        prof_.end(st_, P_OTHER);
        PMGB_CK(cudaGetLastError());
      }
    }
    // per-step sums: part_[(2j+q)][b][G] -> steps_[(2j+q)][b]
    prof_.begin(st_, P_OTHER, lpt2_ ? 12 + 27 : 12);
    k_sum_partials<<<2 * (n_ + 1) * B_, 256, 0, st_>>>(part_, G_, steps_, 1.0);
    PMGB_CK(cudaGetLastError());
    PMGB_RET(ic_adjoint(djdw));
    // theta
    ThetaIn in;
    in.step_pa = steps_;  // layout [(2j+q)][b]: pa at q = 0, xp at q = 1
    in.step_xp = steps_ + B_;
    in.w_pa = wpa_;
    in.w_xp = wxp_;
    in.xs = scal_ + 2 * B_;
    in.ps = scal_ + 3 * B_;
    in.dlp = scal_ + 4 * B_;
    in.dd1 = dd1_;
    in.dgd = dgd_;
    in.xs2 = lpt2_ ? scal_ + 9 * B_ : nullptr;
    in.ps2 = lpt2_ ? scal_ + 10 * B_ : nullptr;
    in.dd2 = dd2_;
    in.dgd2 = dgd2_;
    in.nstep1 = n_ + 1;
    in.batch = B_;
    in.step_stride = 2 * B_;
    k_final_theta<<<(B_ + 31) / 32, 32, 0, st_>>>(in, theta_out_);
    if (obs_theta) {
      k_sum_partials<<<nobs * B_, 256, 0, st_>>>(obs_part_, Go_, obs_sums_, 1.0);
      k_obs_theta<<<(B_ + 31) / 32, 32, 0, st_>>>(obs_sums_, obs_w_, nobs, B_, theta_out_);
    }
    prof_.end(st_, P_OTHER);
    PMGB_CK(cudaGetLastError());
    have_fwd_ = false;
    if (djdth) {
      PMGB_CK(cudaMemcpyAsync(djdth, theta_out_, sizeof(double) * 5 * B_, cudaMemcpyDefault, st_));
      if (is_host(djdth)) return device_error();
    }
    return PM_OK;
  }

  // ------------------------------------------------------------------ operators
  int op_density(const void* disp, void* dens) override {
    counted_ = false;
    if (reinterpret_cast<uintptr_t>(dens) % (4 * sizeof(T))) return PM_ERR_ARG;   // vector stores
    have_fwd_ = false;
    const T* s = nullptr;
    PMGB_RET(op_input(disp, dens, (long long)B_ * M_, nullptr, 0, s_, &s));
    PMGB_RET(scatter(s, nullptr, (T*)dens, M_));
    return PM_OK;
  }

  // The operators read the caller's particles where they lie: the deposit reads all of them
  // before the gather writes a result.  Only inputs that overlap an output, or that lie off
  // their elements' alignment, which kernels cannot read, are copied first (into buf).
  int op_input(const void* in, const void* out0, long long n0, const void* out1, long long n1, T* buf, const T** use) {
    auto meets = [&](const void* out, long long n) {
      const uintptr_t a = (uintptr_t)in, b = (uintptr_t)out;
      return out && a < b + sizeof(T) * n && b < a + sizeof(T) * B_ * 3 * N_;
    };
    *use = (const T*)in;
    if (meets(out0, n0) || meets(out1, n1) || (uintptr_t)in % sizeof(T)) {
      PMGB_CK(cudaMemcpyAsync(buf, in, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
      *use = buf;
    }
    return PM_OK;
  }

  int op_force(const void* disp, const void* pi, void* acc, void* alpha) override {
    counted_ = false;
    have_fwd_ = false;
    const long long pv = (long long)B_ * 3 * N_;
    const T* s = nullptr;
    PMGB_RET(op_input(disp, acc, pv, pi ? alpha : nullptr, pv, s_, &s));
    if (!pi) {
      PMGB_RET(force_chain(s, nullptr, false));
      const auto fn = gather_fwd_fn<true>();
      fn<<<dim3(Gof_, B_), kPtclThreads, 0, st_>>>(
          geo_, const_cast<T*>(s), nullptr, (T*)acc, fvec_, fexp_, StepCoef<T>{}, 0, 1, nullptr, nullptr, bg1_, nullptr,
          nullptr, nullptr, FixState<T>{});
    } else {
      const T* q = nullptr;
      PMGB_RET(op_input(pi, acc, pv, alpha, pv, pi_, &q));
      PMGB_CK(cudaMemsetAsync(pimax_, 0, sizeof(unsigned) * 3 * B_, st_));
      k_pi_max<T><<<dim3(Gpm_, B_), kPtclThreads, 0, st_>>>(q, N_, pimax_);
      PMGB_RET(force_chain(s, q, false));
      const auto fn = gather_adj_fn<true>();
      fn<<<dim3(Goa_, B_), kPtclThreads, 0, st_>>>(
          geo_, mass_, const_cast<T*>(s), nullptr, nullptr, const_cast<T*>(q), (T*)acc, (T*)alpha, fvec_, fexp_,
          StepCoef<T>{}, 0, 1, nullptr, nullptr, nullptr, nullptr, nullptr, bg4_, nullptr, nullptr, FixState<T>{});
    }
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  int op_fft(int dir, const void* in, void* out) override {
    have_fwd_ = false;
    const long long rows = (long long)B_ * nm_ * nm_;
    const int grid = (int)std::min<long long>((rows + 7) / 8, 8LL * nsm_);
    if (dir < 0) {
      PMGB_RET(r2c_real(nm_, (const T*)in, (long long)M_, spec_[0]));
      k_spec_std<T, true><<<grid, 256, 0, st_>>>(spec_[0], (C*)out, nm_, rows);
    } else {
      k_spec_std<T, false><<<grid, 256, 0, st_>>>((const C*)in, spec_[0], nm_, rows);
      PMGB_CK(cudaGetLastError());
      PMGB_RET(c2r_real(nm_, spec_[0], (T*)out, (long long)M_));
    }
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // New theta (host, [batch][5]) and/or omega (host or device): tables are recomputed on
  // the host and copied into the existing device buffers.
  int set_inputs(const double* theta, const void* omega) override {
    if (theta) PMGB_RET(tables(theta));
    if (omega) PMGB_CK(cudaMemcpyAsync(omega_, omega, sizeof(T) * B_ * N_, cudaMemcpyDefault, st_));
    have_fwd_ = false;
    return PM_OK;
  }

  // One gradient evaluation with host or device buffers: omega in, target in, forward,
  // MSE loss, adjoint, loss / grad_omega / grad_theta out.  Host outputs synchronise.
  int gradient(const void* omega, const void* target, double* loss, void* grad_omega, double* grad_theta) override {
    // allocated on first use, each on its own (a failed allocation is retried next call)
    if (!tgt_) PMGB_RET(alloc(&tgt_, (long long)B_ * M_));
    if (!djdd_) PMGB_RET(alloc(&djdd_, (long long)B_ * M_));
    if (!gw_) PMGB_RET(alloc(&gw_, (long long)B_ * N_));
    // The target is first read by the loss, after the whole forward run: its upload goes
    // on a copy stream of its own, ordered after the work already queued (the previous
    // call's loss reads tgt_) and waited for before the loss, so that it overlaps the
    // forward run.
    if (!cp_st_) {
      PMGB_CK(cudaStreamCreateWithFlags(&cp_st_, cudaStreamNonBlocking));
      PMGB_CK(cudaEventCreateWithFlags(&cp_in_, cudaEventDisableTiming));
      PMGB_CK(cudaEventCreateWithFlags(&cp_done_, cudaEventDisableTiming));
    }
    PMGB_CK(cudaEventRecord(cp_in_, st_));
    PMGB_CK(cudaStreamWaitEvent(cp_st_, cp_in_, 0));
    PMGB_CK(cudaMemcpyAsync(tgt_, target, sizeof(T) * B_ * M_, cudaMemcpyDefault, cp_st_));
    PMGB_CK(cudaEventRecord(cp_done_, cp_st_));
    if (omega) PMGB_CK(cudaMemcpyAsync(omega_, omega, sizeof(T) * B_ * N_, cudaMemcpyDefault, st_));
    PMGB_RET(forward(nullptr, nullptr, nullptr));
    PMGB_CK(cudaStreamWaitEvent(st_, cp_done_, 0));
    PMGB_RET(loss_mse_dev(tgt_, djdd_));
    PMGB_RET(adjoint(djdd_, nullptr, nullptr, gw_, nullptr));
    if (loss) {
      PMGB_CK(cudaMemcpyAsync(loss, scal_, sizeof(double) * B_, cudaMemcpyDefault, st_));
    }
    if (grad_omega) PMGB_CK(cudaMemcpyAsync(grad_omega, gw_, sizeof(T) * B_ * N_, cudaMemcpyDefault, st_));
    if (grad_theta) PMGB_CK(cudaMemcpyAsync(grad_theta, theta_out_, sizeof(double) * 5 * B_, cudaMemcpyDefault, st_));
    if ((loss && is_host(loss)) || (grad_omega && is_host(grad_omega)) || (grad_theta && is_host(grad_theta)))
      return device_error();
    return PM_OK;
  }

  // Shell-averaged P(k) of dens ([B][M]; null: the last forward density), n_mesh/2 bins
  int power_spectrum(const void* dens, double* pk, double* kmean, double* nmodes) override {
    const int nb = nm_ / 2;
    if (!dens && !have_dens_) return PM_ERR_STATE;
    PMGB_RET(power_dev(dens ? (const T*)dens : dens_));
    if (pk) PMGB_CK(cudaMemcpyAsync(pk, pw_out_, sizeof(double) * B_ * nb, cudaMemcpyDefault, st_));
    if (kmean) PMGB_CK(cudaMemcpyAsync(kmean, pw_out_ + B_ * nb, sizeof(double) * nb, cudaMemcpyDefault, st_));
    if (nmodes) PMGB_CK(cudaMemcpyAsync(nmodes, pw_out_ + (B_ + 1) * nb, sizeof(double) * nb, cudaMemcpyDefault, st_));
    return device_error();
  }

  // Objective on the shell power of delta (the last forward density when dens is null):
  // J_b = sum w (P - T)^2 and dJ/d delta = IDFT_unnorm[g(|n|) delta^] (k_power_loss,
  // k_power_grad, one inverse transform).
  int loss_power(const void* dens, const double* tgt, const double* w, double* loss, void* djdd) override {
    if (!dens && !have_dens_) return PM_ERR_STATE;
    const int nb = nm_ / 2;
    PMGB_RET(power_dev(dens ? (const T*)dens : dens_));
    if (!pl_buf_) PMGB_RET(alloc(&pl_buf_, (long long)B_ * (3 * nb + 1)));
    double* dt = pl_buf_;
    double* dw = pl_buf_ + (long long)B_ * nb;
    double* dg = pl_buf_ + 2LL * B_ * nb;
    double* dl = pl_buf_ + 3LL * B_ * nb;
    PMGB_CK(cudaMemcpyAsync(dt, tgt, sizeof(double) * B_ * nb, cudaMemcpyDefault, st_));
    PMGB_CK(cudaMemcpyAsync(dw, w, sizeof(double) * B_ * nb, cudaMemcpyDefault, st_));
    const double vol = cfg_.box * cfg_.box * cfg_.box;
    k_power_loss<<<B_, kPowerThreads, 0, st_>>>(pw_out_, pw_out_ + (B_ + 1) * nb, dt, dw, nb,
                                                2.0 * vol / ((double)M_ * (double)M_), dl, dg);
    const PowerRuns pr = power_runs(nm_, spec_lzb(nm_));
    k_power_grad<T><<<dim3(power_grid(pr), B_), kPowerThreads, 0, st_>>>(spec_[6], pr, spec_len_cx(nm_), nb, dg);
    PMGB_CK(cudaGetLastError());
    PMGB_RET(c2r_real(nm_, spec_[6], (T*)djdd, M_));
    if (loss) {
      PMGB_CK(cudaMemcpyAsync(loss, dl, sizeof(double) * B_, cudaMemcpyDefault, st_));
      if (is_host(loss)) return device_error();
    }
    return PM_OK;
  }

  // Shell power of d into pw_out_ (pk [B][nb], kmean [nb], nmodes [nb]); leaves delta^ in
  // spec_[6].  Deterministic: per-bin int64 fixed point scaled from a first max pass.
  int power_dev(const T* d) {
    const int nb = nm_ / 2;
    if (!pw_acc_) PMGB_RET(alloc(&pw_acc_, (long long)B_ * nb));
    if (!pw_max_) PMGB_RET(alloc(&pw_max_, (long long)B_ * nb));
    if (!pw_out_) PMGB_RET(alloc(&pw_out_, (long long)(B_ + 2) * nb));
    if (!pw_modes_) {
      // the modes of each bin: constants of the mesh side, counted once per context
      unsigned long long* m = nullptr;
      PMGB_RET(alloc(&m, 2LL * nb));
      PMGB_CK(cudaMemsetAsync(m, 0, sizeof(unsigned long long) * 2 * nb, st_));
      k_power_modes<<<std::min(4 * nsm_, (nb * nb + kPowerThreads - 1) / kPowerThreads), kPowerThreads, 0, st_>>>(
          nb, m, m + nb);
      PMGB_CK(cudaGetLastError());
      pw_modes_ = m;
    }
    PMGB_RET(r2c_real(nm_, d, M_, spec_[6]));
    PMGB_CK(cudaMemsetAsync(pw_acc_, 0, sizeof(unsigned long long) * B_ * nb, st_));
    PMGB_CK(cudaMemsetAsync(pw_max_, 0, sizeof(unsigned) * B_ * nb, st_));
    const long long is = spec_len_cx(nm_);
    const PowerRuns pr = power_runs(nm_, spec_lzb(nm_));
    const dim3 grid(power_grid(pr), B_);
    k_power_max<T><<<grid, kPowerThreads, 0, st_>>>(spec_[6], pr, is, nb, pw_max_);
    k_power_acc<T><<<grid, kPowerThreads, 0, st_>>>(spec_[6], pr, is, nb, ilog2(M_), pw_max_, pw_acc_);
    const double vol = cfg_.box * cfg_.box * cfg_.box;
    k_power_final<T><<<(B_ * nb + 255) / 256, 256, 0, st_>>>(pw_acc_, pw_modes_, pw_modes_ + nb, pw_max_, ilog2(M_),
                                                           nb, B_, vol / ((double)M_ * (double)M_),
                                                           2.0 * M_PI / cfg_.box, pw_out_, pw_out_ + B_ * nb,
                                                           pw_out_ + (B_ + 1) * nb);
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }
  // four resident blocks per SM: each block adds its bins to the global ones once
  int power_grid(const PowerRuns& pr) const {
    return (int)std::min<long long>(4LL * nsm_, (pr.count + kPowerThreads - 1) / kPowerThreads);
  }

  // One gradient evaluation on device buffers, captured once into a CUDA graph on the
  // context stream and replayed afterwards (re-captured when the pointers change).
  int gradient_graph(const void* target, double* loss, void* gw, double* gt) override {
    if (st_ == 0) return PM_ERR_ARG;  // the legacy default stream cannot be captured
    if ((loss && is_host(loss)) || (gw && is_host(gw)) || (gt && is_host(gt)) || is_host(target)) return PM_ERR_ARG;
    if (!djdd_) PMGB_RET(alloc(&djdd_, (long long)B_ * M_));
    const void* args[4] = {target, loss, gw, gt};
    bool same = graph_exec_ != nullptr;
    for (int i = 0; i < 4 && same; ++i) same = args[i] == graph_args_[i];
    if (!same) {
      if (graph_exec_) {
        cudaGraphExecDestroy(graph_exec_);
        graph_exec_ = nullptr;
      }
      PMGB_RET(eval_device(target, loss, gw, gt));  // warm-up outside the capture
      PMGB_CK(cudaStreamSynchronize(st_));
      cudaGraph_t g = nullptr;
      PMGB_CK(cudaStreamBeginCapture(st_, cudaStreamCaptureModeThreadLocal));
      const int r = eval_device(target, loss, gw, gt);
      const cudaError_t e = cudaStreamEndCapture(st_, &g);
      if (r != PM_OK) {
        if (g) cudaGraphDestroy(g);
        return r;
      }
      PMGB_CK(e);
      const cudaError_t ei = cudaGraphInstantiate(&graph_exec_, g, 0);
      cudaGraphDestroy(g);
      PMGB_CK(ei);
      for (int i = 0; i < 4; ++i) graph_args_[i] = args[i];
    }
    PMGB_CK(cudaGraphLaunch(graph_exec_, st_));
    return PM_OK;
  }

  int op_za(void* s1) override {
    have_fwd_ = false;
    PMGB_RET(initial_conditions());
    PMGB_CK(cudaMemcpyAsync(s1, s1_, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    return PM_OK;
  }

  // Observed intermediate states: step -> snapshot index; the forward copies s_j and
  // delta_j out, the adjoint adds their cotangents at step j.  A captured gradient graph
  // is dropped (it holds the old settings).
  int set_snapshots(int ns, const int* steps, void* disp, void* dens, const void* gdisp, const void* gdens) override {
    if (ns < 0 || ns > PM_MAX_SNAPSHOTS || (ns > 0 && !steps)) return PM_ERR_ARG;
    std::vector<int> map(n_ + 1, -1);
    for (int q = 0; q < ns; ++q) {
      if (steps[q] < 0 || steps[q] > n_ || (q > 0 && steps[q] <= steps[q - 1])) return PM_ERR_ARG;
      map[steps[q]] = q;
    }
    if (ns == 0) map.clear();
    snap_of_ = map;
    snap_mom_ = nullptr;
    snap_gmom_ = nullptr;
    snap_disp_ = ns ? (T*)disp : nullptr;
    snap_dens_ = ns ? (T*)dens : nullptr;
    snap_gdisp_ = ns ? (const T*)gdisp : nullptr;
    snap_gdens_ = ns ? (const T*)gdens : nullptr;
    if (graph_exec_) {
      cudaGraphExecDestroy(graph_exec_);
      graph_exec_ = nullptr;
    }
    return PM_OK;
  }
  int snap_of(int j) const { return snap_of_.empty() ? -1 : snap_of_[j]; }

  int set_snapshot_momenta(void* mom, const void* gmom) override {
    if (snap_of_.empty()) return PM_ERR_STATE;
    snap_mom_ = (T*)mom;
    snap_gmom_ = (const T*)gmom;
    if (graph_exec_) {
      cudaGraphExecDestroy(graph_exec_);
      graph_exec_ = nullptr;
    }
    return PM_OK;
  }

  // Observed positions at scale factors between steps: each a_q in (a0, a1] (ascending)
  // lies in step j + 1 = (a_j, a_{j+1}]; the partial drift factor and its d/dOmega_m per
  // instance come from the host tables.
  int set_interp_snapshots(int na, const double* a, void* disp, void* dens, const void* gdisp,
                           const void* gdens) override {
    if (na < 0 || na > PM_MAX_SNAPSHOTS || (na > 0 && !a)) return PM_ERR_ARG;
    for (int k = 0; k < na; ++k)
      if (!(a[k] > cfg_.a0) || !(a[k] <= cfg_.a1) || (k > 0 && !(a[k] > a[k - 1]))) return PM_ERR_ARG;
    interp_a_.assign(a, a + na);
    interp_disp_ = na ? (T*)disp : nullptr;
    interp_dens_ = na ? (T*)dens : nullptr;
    interp_gdisp_ = na ? (const T*)gdisp : nullptr;
    interp_gdens_ = na ? (const T*)gdens : nullptr;
    PMGB_RET(tables(theta_host_.data()));
    if (graph_exec_) {
      cudaGraphExecDestroy(graph_exec_);
      graph_exec_ = nullptr;
    }
    return PM_OK;
  }

  // s(a_k) = s_{j+1} + (Dp_j(a_k) - D_{j+1}) p_{j+1/2} and, if asked, delta(a_k) by the
  // global-atomic fixed-point deposit into the force mesh, free until the next force chain
  // (the bins of the tile deposit are counted for the next step already).
  int interp_forward(int k) {
    T* out = interp_disp_ ? interp_disp_ + (long long)k * B_ * 3 * N_ : xi_;
    prof_.begin(st_, P_OTHER, interp_dens_ ? 3 : 1);
    k_interp_state<T><<<dim3(256, B_), 256, 0, st_>>>(s_, p_, obs_cf_ + (long long)k * B_, out, 3 * N_);
    PMGB_CK(cudaGetLastError());
    if (interp_dens_) {
      unsigned long long* acc = reinterpret_cast<unsigned long long*>(fvec_);
      PMGB_CK(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * B_ * M_, st_));
      k_scatter<T, 1><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(geo_, out, nullptr, acc, e_d_, nullptr);
      k_density_out<T><<<1024, 256, 0, st_>>>((const long long*)acc, interp_dens_ + (long long)k * B_ * M_,
                                              (long long)B_ * M_, (T)(mass_ * std::ldexp(1.0, -e_d_)));
      PMGB_CK(cudaGetLastError());
    }
    prof_.end(st_, P_OTHER);
    return PM_OK;
  }

  int get_fixed_state(long long* u, long long* w) override {
    if (!fx_.u) return PM_ERR_STATE;
    if (u) PMGB_CK(cudaMemcpyAsync(u, fix_u_, sizeof(long long) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    if (w) PMGB_CK(cudaMemcpyAsync(w, fix_w_, sizeof(long long) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    return PM_OK;
  }

  int op_ic(void* s0, void* p0) override {
    have_fwd_ = false;
    PMGB_RET(initial_conditions());
    if (s0) PMGB_CK(cudaMemcpyAsync(s0, s_, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    if (p0) PMGB_CK(cudaMemcpyAsync(p0, p_, sizeof(T) * B_ * 3 * N_, cudaMemcpyDeviceToDevice, st_));
    return PM_OK;
  }

 private:
  template <typename U> int alloc(U** p, long long count) {
    void* q = nullptr;
    const size_t bytes = sizeof(U) * (size_t)(count > 0 ? count : 1);
    if (!alloc_gate()) return PM_ERR_OOM;   // injected failure (test hook)
    cudaError_t e = cudaMalloc(&q, bytes);
    if (e != cudaSuccess) { set_cuda_error(e); cudaGetLastError(); return PM_ERR_OOM; }
    allocs_.push_back(q);
    bytes_ += (long long)bytes;
    live_bytes_add((long long)bytes);
    *p = (U*)q;
    return PM_OK;
  }
  static bool is_host(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) { cudaGetLastError(); return true; }
    return at.type == cudaMemoryTypeHost || at.type == cudaMemoryTypeUnregistered;
  }
  // real view of spectrum buffer q (after C2R)
  T* rmesh(int q) { return reinterpret_cast<T*>(spec_[q]); }

  // ---------------------------------------------------------------- host tables
  int tables(const double* theta) {
    const int n1 = n_ + 1;
    if (theta != theta_host_.data()) theta_host_.assign(theta, theta + 5 * B_);
    const int nq = (int)interp_a_.size();
    // observations: share c_j of a momentum cotangent at step j that enters pi before the
    // force VJP, the theta weights of the momentum (slot j) and interpolated-position
    // (slot n + 1 + q) terms, and per interpolated position its step, drift factor and the
    // forward coefficient Dp_j(a) - D_{j+1}
    std::vector<T> oc((size_t)B_ * n1), ofac((size_t)std::max(1, nq) * B_), ocf((size_t)std::max(1, nq) * B_);
    std::vector<double> ow((size_t)(n1 + nq) * B_, 0.0);
    interp_.assign(nq, InterpObs{});
    std::vector<T> fkA(B_ * n1), fkB(B_ * n1), fdr(B_ * n1), rkA(B_ * n1), rkB(B_ * n1), rdr(B_ * n1);
    std::vector<double> wpa(n1 * B_), wxp(n1 * B_), dd1(B_), dgd(B_), dd2(B_), dgd2(B_);
    std::vector<T> d1(B_), gd(B_), d2(B_), gd2(B_), gcoef(B_);
    const int maxn2 = 3 * (np_ / 2) * (np_ / 2);
    const double kfp = 2.0 * M_PI / cfg_.box;
    const double lp = cfg_.box / np_;
    std::vector<T> amp((size_t)B_ * (maxn2 + 1));
    std::vector<double> hdl((size_t)B_ * 5 * (maxn2 + 1));
    for (int b = 0; b < B_; ++b) {
      const double* th = theta + 5 * b;
      const double om = th[2];
      cosmo::TimeCoef tc;
      cosmo::time_coefficients(cfg_.a0, cfg_.a1, n_, om, tc);
      for (int j = 0; j <= n_; ++j) {
        const int o = b * n1 + j;
        fkA[o] = (T)(j >= 1 ? tc.k2[j - 1] : 0.0);
        fkB[o] = (T)(j < n_ ? tc.k1[j] : 0.0);
        fdr[o] = (T)(j < n_ ? tc.dd[j] : 0.0);
        rkA[o] = (T)(j < n_ ? tc.k1[j] : 0.0);
        rkB[o] = (T)(j >= 1 ? tc.k2[j - 1] : 0.0);
        rdr[o] = (T)(j >= 1 ? tc.dd[j - 1] : 0.0);
        double w = 0.0;
        if (j < n_) w += tc.dk1[j] + tc.k1[j] / om;
        if (j >= 1) w += tc.dk2[j - 1] + tc.k2[j - 1] / om;
        wpa[j * B_ + b] = w;
        wxp[j * B_ + b] = j >= 1 ? tc.ddd[j - 1] : 0.0;
        const double k1n = j < n_ ? tc.k1[j] : 0.0, k2j = j >= 1 ? tc.k2[j - 1] : 0.0;
        const double c = (k1n + k2j) != 0.0 ? k2j / (k1n + k2j) : 0.0;
        oc[(size_t)b * n1 + j] = (T)c;
        ow[(size_t)j * B_ + b] = (j >= 1 ? tc.dk2[j - 1] + k2j / om : 0.0) - c * w;
      }
      for (int k = 0; k < nq; ++k) {
        cosmo::PartialDrift pd;
        cosmo::partial_drift(cfg_.a0, cfg_.a1, n_, om, interp_a_[k], pd);
        interp_[k].j = pd.j;
        ofac[(size_t)k * B_ + b] = (T)pd.fac;
        ocf[(size_t)k * B_ + b] = (T)(pd.fac - tc.dd[pd.j]);
        ow[(size_t)(n1 + k) * B_ + b] = pd.dfac;
      }
      d1[b] = (T)tc.d1_a0;
      gd[b] = (T)tc.gd_a0;
      d2[b] = (T)tc.d2_a0;
      gd2[b] = (T)tc.gd2_a0;
      dd2[b] = tc.dd2_a0;
      dgd2[b] = tc.dgd2_a0;
      dd1[b] = tc.dd1_a0;
      dgd[b] = tc.dgd_a0;
      // H_c = -i k_c G / M with G = -3/2 Om / k^2: per mode f_c * coef / n^2 * (-i)
      const double kfm = 2.0 * M_PI / cfg_.box;
      gcoef[b] = (T)(-1.5 * om / (kfm * (double)M_));
      // ZA amplitude sqrt(P / l_p^3) / n_p^3 and 1/2 dlnP/dtheta per integer |n|^2
      std::vector<double> p, dl;
      cosmo::plin_tables(th, kfp, maxn2, p, dl);
      for (int n2 = 0; n2 <= maxn2; ++n2) {
        amp[(size_t)b * (maxn2 + 1) + n2] = (T)(n2 ? std::sqrt(p[n2] / (lp * lp * lp)) / (double)N_ : 0.0);
        for (int j = 0; j < 5; ++j)
          hdl[((size_t)b * 5 + j) * (maxn2 + 1) + n2] = n2 ? 0.5 * dl[(size_t)j * (maxn2 + 1) + n2] : 0.0;
      }
    }
    maxn2_ = maxn2;
    inv_kfp_ = (T)(1.0 / kfp);
    PMGB_RET(upload(&fkA_, fkA));
    PMGB_RET(upload(&fkB_, fkB));
    PMGB_RET(upload(&fdr_, fdr));
    PMGB_RET(upload(&rkA_, rkA));
    PMGB_RET(upload(&rkB_, rkB));
    PMGB_RET(upload(&rdr_, rdr));
    PMGB_RET(upload(&obs_c_, oc));
    PMGB_RET(upload_grow(&obs_fac_, ofac, obs_fac_n_));
    PMGB_RET(upload_grow(&obs_cf_, ocf, obs_cf_n_));
    PMGB_RET(upload_grow(&obs_w_, ow, obs_w_n_));
    if (obs_sums_n_ < (long long)(n1 + nq) * B_) {
      PMGB_RET(alloc(&obs_sums_, (long long)(n1 + nq) * B_));
      PMGB_RET(alloc(&obs_part_, (long long)(n1 + nq) * B_ * Go_));
      obs_sums_n_ = (long long)(n1 + nq) * B_;
    }
    PMGB_RET(upload(&wpa_, wpa));
    PMGB_RET(upload(&wxp_, wxp));
    PMGB_RET(upload(&dd1_, dd1));
    PMGB_RET(upload(&dgd_, dgd));
    PMGB_RET(upload(&d1_, d1));
    PMGB_RET(upload(&gd_, gd));
    PMGB_RET(upload(&d2_, d2));
    PMGB_RET(upload(&gd2_, gd2));
    PMGB_RET(upload(&dd2_, dd2));
    PMGB_RET(upload(&dgd2_, dgd2));
    unit_ = (T)(1.0 / (double)N_);
    PMGB_RET(upload(&gcoef_, gcoef));
    PMGB_RET(upload(&amp_, amp));
    PMGB_RET(upload(&hdl_, hdl));
    if (cfg_.deconv) {
      std::vector<T> dt(nm_);
      for (int i = 0; i < nm_; ++i) {
        const int f = i < nm_ / 2 ? i : i - nm_;
        const double x = M_PI * f / nm_;
        const double sc = f == 0 ? 1.0 : std::sin(x) / x;
        dt[i] = (T)(1.0 / (sc * sc * sc * sc));
      }
      PMGB_RET(upload(&dtab_, dt));
    }
    // twiddles: table of size L at [L, 2L): exp(-2 pi i m / L)
    std::vector<C> tw(4096);
    for (int L = 1; L <= 2048; L *= 2)
      for (int m = 0; m < L; ++m) {
        const double ang = -2.0 * M_PI * (double)m / (double)L;
        tw[L + m].x = (T)std::cos(ang);
        tw[L + m].y = (T)std::sin(ang);
      }
    PMGB_RET(upload(&tw_, tw));
    if (pimax_) return PM_OK;
    PMGB_RET(alloc(&pimax_, 3 * B_));
    PMGB_RET(alloc(&e_pi_, 3 * B_));
    PMGB_RET(alloc(&part_, (long long)(2 * (n_ + 1) + 16) * B_ * kMaxRedBlocks));
    PMGB_RET(alloc(&steps_, (long long)2 * (n_ + 1) * B_));
    PMGB_RET(alloc(&scal_, (long long)16 * B_));
    PMGB_RET(alloc(&theta_out_, (long long)5 * B_));
    return PM_OK;
  }
  // upload into a buffer that is reallocated when the table outgrows it (cap: elements held)
  template <typename U> int upload_grow(U** d, const std::vector<U>& h, long long& cap) {
    if ((long long)h.size() > cap) {
      PMGB_RET(alloc(d, (long long)h.size()));   // the old buffer stays owned until pm_destroy
      cap = (long long)h.size();
    }
    PMGB_CK(cudaMemcpyAsync(*d, h.data(), sizeof(U) * h.size(), cudaMemcpyHostToDevice, st_));
    PMGB_CK(cudaStreamSynchronize(st_));
    return PM_OK;
  }
  template <typename U> int upload(U** d, const std::vector<U>& h) {
    if (!*d) PMGB_RET(alloc(d, (long long)h.size()));
    PMGB_CK(cudaMemcpyAsync(*d, h.data(), sizeof(U) * h.size(), cudaMemcpyHostToDevice, st_));
    PMGB_CK(cudaStreamSynchronize(st_));
    return PM_OK;
  }

  // ---------------------------------------------------------------- FFT helpers
  SeqMap ymap(int n) const {
    return SeqMap{n / 2, 1, n / 2, (long long)n * (n / 2), n, spec_len_cx(n), B_ * n * (n / 2), 0};
  }
  SeqMap yside(int n) const {
    return SeqMap{1, n, n, spec_len_cx(n), B_, 0, B_ * n, spec_main_len(n)};
  }
  SeqMap zmap(int n) const {
    return SeqMap{(long long)n * (n / 2), 1, n / 2, n / 2, n, spec_len_cx(n), B_ * n * (n / 2), 0};
  }
  SeqMap zside(int n) const {
    return SeqMap{n, 1, n, spec_len_cx(n), B_, 0, B_ * n, spec_main_len(n)};
  }
  int spec_index(const C* p) const {
    for (int q = 0; q < 7; ++q)
      if (spec_[q] == p) return q;
    return -1;
  }
  // column pass over up to 4 spectra: mesh spectra (z-blocked main rows at 1024^3, see
  // spec_row) take the TMA-staged passes, lattice spectra (plain order) the unstaged ones
  int cols(int n, int dir, bool zaxis, C* const* bufs, int nb, bool mesh = true) {
    SeqMap mm = zaxis ? zmap(n) : ymap(n);
    const SeqMap ms = zaxis ? zside(n) : yside(n);
    if (use_tma_ && mesh && n == nm_) {
      CUtensorMap maps[4];
      for (int q = 0; q < nb; ++q) {
        const int i = spec_index(bufs[q]);
        if (i < 0) return PM_ERR_STATE;
        maps[q] = zaxis ? tmz_[i] : tmy_[i];
      }
      PMGB_RET(fft_cols_tma<T>(n, B_, dir, zaxis ? 1 : 0, maps, bufs, nb, tw_, WaitCtl{dev_err_, first_wait_}, nsm_, st_));
      PMGB_CK(cudaGetLastError());
      mm.nseq = 0;   // the side planes are left
    }
    // one launch over the main columns (unless staged above) and the side planes
    ColBufs<T> b{};
    for (int q = 0; q < nb; ++q) b.p[q] = bufs[q];
    PMGB_RET(fft_cols<T>(n, dir, mm, ms, b, nb, tw_, st_));
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }
  int r2c_real(int n, const T* in, long long in_is, C* out) {
    RowJob<T> job{};
    job.b[0] = RowBuf<T>{(void*)in, in_is, out};
    job.lzb = spec_lzb(n);
    PMGB_RET(fft_x_r2c<T>(n, job, 1, B_ * n * n, tw_, st_));
    C* bufs[1] = {out};
    PMGB_RET(cols(n, -1, false, bufs, 1));
    PMGB_RET(cols(n, -1, true, bufs, 1));
    return PM_OK;
  }
  int c2r_real(int n, C* in, T* out, long long out_is) {
    C* bufs[1] = {in};
    PMGB_RET(cols(n, +1, true, bufs, 1));
    PMGB_RET(cols(n, +1, false, bufs, 1));
    RowJob<T> job{};
    job.b[0] = RowBuf<T>{(void*)out, out_is, in};
    job.lzb = spec_lzb(n);
    PMGB_RET(fft_x_c2r<T>(n, job, 1, B_ * n * n, tw_, st_));
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // Bins of the tile-owner deposit, sized for every tile shape that may run (max_bin_keys);
  // the tile shape and threads per tile of the density-only deposit (forward) and of the
  // density + pi deposit (adjoint) are set separately (pm_tuning).
  int bin_setup() {
    // Deposit shapes.  Tiles long in x: the lattice neighbours of a warp spread over more rows'
    // lines, and the write-out stores whole ones.  2^12 cells for the density, 2^11 with the pi sums
    // (three blocks of 512 threads per SM); 2^10 where a mesh makes fewer than two such tiles per
    // SM.  Deposit and x pass separately: fused, the four-quantity tile is one 128 KB block per SM
    // whose phases cannot overlap (force VJP at 512^3 7.06 ms fused, 6.37 ms so; with the former
    // tiles of 8 x 16 x 16 6.43 ms; at 1024^3 59.9, 51.3 and 51.9 ms).
    const bool few = (long long)B_ * M_ < (2LL * nsm_ << 12);
    const int td[3] = {few ? 2 : 3, few ? 2 : 4, few ? 6 : 5}, ta[3] = {2, few ? 2 : 3, 6};
    for (int c = 0; c < 3; ++c) tune_.tile_log2_density[c] = td[c], tune_.tile_log2_adjoint[c] = ta[c];
    tune_.threads_density = 256;
    tune_.threads_adjoint = 512;
    tune_.tma_columns = 1;
    // The density deposit of 128^3 meshes is faster fused: force, separate / fused, with 64^3
    // particles x 2, 4, 8 and 16 instances 162 / 158, 246 / 242, 412 / 405 and 755 / 741 us, 32^3 x 16
    // 591 / 577, 128^3 x 1 and 4 221 / 205 and 553 / 543 (the VJP's is not: 64^3 x 8 774 / 807; nor are
    // larger meshes: 128^3 on 256^3 412 / 418, 256^3 on 512^3 2771 / 2861).  In FP64 the two forms are
    // within 1% of each other at 128^3 to 512^3.  (Few particles: the atomics, see small_deposit.)
    tune_.fused_x = nm_ == 128 && !cfg_.fixed_state && !small_rule(1) ? 1 : 0;
    tune0_ = tune_;
    max_bins_ = (long long)B_ * max_bin_keys(ilog2(nm_)) + 1;
    PMGB_RET(alloc(&bkeys_, (long long)B_ * N_));
    PMGB_RET(alloc(&brec0_, (long long)B_ * N_));
    PMGB_RET(alloc(&brec1_, (long long)B_ * N_));
    PMGB_RET(alloc(&bcount_, max_bins_));
    PMGB_RET(alloc(&bstart_, max_bins_));
    PMGB_RET(alloc(&bcursor_, max_bins_));
    PMGB_RET(alloc(&bsums_, (max_bins_ + kScanBlock - 1) / kScanBlock));
    PMGB_CK(cudaMemsetAsync(bcount_, 0, sizeof(unsigned) * max_bins_, st_));
    ensure_smem_attr((const void*)k_pull_scatter<T, 4, 256>, 4 * 8 * 2048);
    ensure_smem_attr((const void*)k_pull_scatter<T, 4, 512>, 4 * 8 * 2048);
    apply_tuning();
    return PM_OK;
  }
  void apply_tuning() {
    const int lg = ilog2(nm_);
    bg1_ = make_bin_geo(lg, tune_.tile_log2_density[2], tune_.tile_log2_density[1], tune_.tile_log2_density[0]);
    bg4_ = make_bin_geo(lg, tune_.tile_log2_adjoint[2], tune_.tile_log2_adjoint[1], tune_.tile_log2_adjoint[0]);
    use_tma_ = tune_.tma_columns != 0 && tma_supported(nm_);
    // deposit fused with the R2C x pass: tiles of whole x rows, R rows split over (y, z)
    // (with the fixed-point state the forward and the reverse deposit take the same x pass,
    // so that both see bitwise the same forces)
    fused1_ = (tune_.fused_x & 1) != 0 && fused_rows<T>(nm_, 1) > 0 && !cfg_.fixed_state;
    fused4_ = (tune_.fused_x & 2) != 0 && fused_rows<T>(nm_, 1) > 0 && !cfg_.fixed_state;
    if (fused_rows<T>(nm_, 1) > 0) {
      auto geo = [&](int rows) {
        const int lr = ilog2(rows);
        return make_bin_geo(lg, lg, (lr + 1) / 2, lr / 2);
      };
      bgf1_ = geo(fused_rows<T>(nm_, 1));
      bgf4_ = geo(fused_rows<T>(nm_, 4));
    }
  }
  int get_tuning(pm_tuning* t) override {
    *t = tune_;
    return PM_OK;
  }
  int set_tuning(const pm_tuning* t) override {
    if (!tile_ok(t->tile_log2_density, 12) || !tile_ok(t->tile_log2_adjoint, 11)) return PM_ERR_ARG;
    if ((t->threads_density != 256 && t->threads_density != 512) ||
        (t->threads_adjoint != 256 && t->threads_adjoint != 512))
      return PM_ERR_ARG;
    if (t->tma_columns != 0 && t->tma_columns != 1) return PM_ERR_ARG;
    if (t->tma_columns && !tma_supported(nm_)) return PM_ERR_ARG;
    if (!t->tma_columns && spec_zb(nm_) > 1) return PM_ERR_ARG;   // z-blocked rows: staged passes only
    if (t->fused_x < 0 || t->fused_x > 3 || (t->fused_x && (fused_rows<T>(nm_, 1) == 0 || cfg_.fixed_state)))
      return PM_ERR_ARG;
    tune_ = *t;
    apply_tuning();
    return PM_OK;
  }

  // Autotuner: times every candidate of the tunable launches on this context's current
  // particle state (the final state of the last forward run, or the Zel'dovich state if
  // none) and keeps the fastest.  Candidates: deposit tile shapes (2^9..2^11 cells) x 256
  // or 512 threads, separately for the density-only and the density + pi deposit; the
  // y column pass with or without TMA staging.  Each candidate is timed `reps` times with
  // CUDA events on the context's stream (median).  The deposit sums are exact integers, the
  // same for every shape.  Fused and separate x passes, and the two column-pass forms, run the
  // same radix stages but may round differently in the last bit (from 512^3 on the staged
  // adjoint z pass applies Green's function once, after its sum).
  int autotune(int reps, pm_tuning* chosen, double* ms_best) override {
    counted_ = false;
    if (reps < 1) reps = 3;
    const bool prof_on = prof_.on;
    prof_.on = false;
    if (!have_fwd_) {
      PMGB_RET(initial_conditions());
    }
    // synthetic adjoint state for the pi deposit: every pi_c = 7.1e-4 (bit pattern
    // 0x3A3A3A3A), fixed-point exponents set from that maximum on the host
    PMGB_CK(cudaMemsetAsync(xi_, 0x3A, sizeof(T) * B_ * 3 * N_, st_));
    {
      float v;
      const unsigned bits = 0x3A3A3A3Au;
      std::memcpy(&v, &bits, 4);
      const int E = std::ilogb(v) + 1;
      std::vector<int> e(3 * B_, fixed_top<T>(lgN_) - E);
      PMGB_CK(cudaMemcpyAsync(e_pi_, e.data(), sizeof(int) * e.size(), cudaMemcpyHostToDevice, st_));
      PMGB_CK(cudaStreamSynchronize(st_));
    }
    cudaEvent_t e0, e1;
    PMGB_CK(cudaEventCreate(&e0));
    PMGB_CK(cudaEventCreate(&e1));
    auto time_it = [&](auto&& fn, double* ms) -> int {
      std::vector<float> t;
      PMGB_RET(fn());   // warm-up
      for (int r = 0; r < reps; ++r) {
        PMGB_CK(cudaEventRecord(e0, st_));
        PMGB_RET(fn());
        PMGB_CK(cudaEventRecord(e1, st_));
        PMGB_CK(cudaEventSynchronize(e1));
        float x = 0.f;
        PMGB_CK(cudaEventElapsedTime(&x, e0, e1));
        t.push_back(x);
      }
      std::sort(t.begin(), t.end());
      *ms = t[t.size() / 2];
      return PM_OK;
    };
    static const int kTiles[][3] = {{3, 4, 4}, {3, 3, 5}, {3, 3, 4}, {2, 4, 5}, {2, 4, 4}, {3, 3, 3},
                                    {2, 3, 5}, {4, 4, 4}, {3, 4, 5}, {3, 5, 4}, {2, 3, 6}, {2, 2, 6}, {2, 2, 7}};
    const int lg = ilog2(nm_);
    // the separate deposit that runs with shapes t
    auto separate = [&](const pm_tuning& t, int nq, const SepTargets& tg) {
      const T* pi = nq ? xi_ : nullptr;
      if (small_deposit(nq != 0, t)) return scatter_small(s_, pi, tg.d, tg.dis, tg);
      const int* l = nq ? t.tile_log2_adjoint : t.tile_log2_density;
      return deposit(s_, pi, tg.d, tg.dis, make_bin_geo(lg, l[2], l[1], l[0]),
                     nq ? t.threads_adjoint : t.threads_density, false, nullptr, &tg);
    };
    pm_tuning best = tune_;
    double best_ms[3] = {1e30, 1e30, 1e30};
    for (int nq = 0; nq < 2; ++nq) {
      for (const auto& tl : kTiles) {
        const int l[3] = {tl[0], tl[1], tl[2]};
        if (!tile_ok(l, nq ? 11 : 12)) continue;
        for (int nt : {256, 512}) {
          pm_tuning cand = best;
          std::copy(l, l + 3, nq ? cand.tile_log2_adjoint : cand.tile_log2_density);
          (nq ? cand.threads_adjoint : cand.threads_density) = nt;
          cand.fused_x &= nq ? 1 : 2;
          double ms = 0;
          PMGB_RET(time_it([&]() { return separate(cand, nq, sep_targets(false)); }, &ms));
          if (ms < best_ms[nq]) {
            best_ms[nq] = ms;
            best = cand;
          }
        }
      }
    }
    // deposit fused with the R2C x pass against the chosen separate deposit + x pass, for
    // the density deposit (bit 0) and the density + pi deposit (bit 1) separately
    if (fused_rows<T>(nm_, 1) > 0 && !cfg_.fixed_state) {
      best.fused_x = 0;
      for (int nq = 0; nq < 2; ++nq) {
        double ms_sep = 0, ms_fused = 0;
        const SepTargets tg = sep_targets(false);
        PMGB_RET(time_it([&]() {
          PMGB_RET(separate(best, nq, tg));
          RowJob<T> job{};
          job.b[0] = RowBuf<T>{tg.d, tg.dis, spec_[0]};
          if (nq)
            for (int c = 0; c < 3; ++c) job.b[1 + c] = RowBuf<T>{tg.p[c], tg.pis, spec_[4 + c]};
          job.lzb = spec_lzb(nm_);
          return fft_x_r2c<T>(nm_, job, nq ? 4 : 1, B_ * nm_ * nm_, tw_, st_);
        }, &ms_sep));
        FusedOut<T> fo{};
        fo.spec[0] = spec_[0];
        for (int c = 0; c < 3; ++c) fo.spec[1 + c] = nq ? spec_[4 + c] : nullptr;
        PMGB_RET(time_it([&]() { return deposit(s_, nq ? xi_ : nullptr, nullptr, 0, nq ? bgf4_ : bgf1_, 0, false, &fo); },
                         &ms_fused));
        if (ms_fused < ms_sep) best.fused_x |= 1 << nq;
        fused_ms_[2 * nq] = ms_sep;
        fused_ms_[2 * nq + 1] = ms_fused;
      }
    }
    if (tma_supported(nm_)) {
      C* b1[1] = {spec_[6]};
      for (int tma = 1; tma >= (spec_zb(nm_) > 1 ? 1 : 0); --tma) {   // blocked rows: staged passes only
        use_tma_ = tma != 0;
        double ms = 0;
        PMGB_RET(time_it([&]() { return cols(nm_, -1, false, b1, 1); }, &ms));
        if (ms < best_ms[2]) {
          best_ms[2] = ms;
          best.tma_columns = tma;
        }
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    tune_ = best;
    apply_tuning();
    prof_.on = prof_on;
    if (chosen) *chosen = best;
    if (ms_best)
      for (int k = 0; k < 3; ++k) ms_best[k] = best_ms[k] < 1e29 ? best_ms[k] : 0.0;
    return PM_OK;
  }

  // CIC assignment (Sec. 2.2, Eq. 10) of the density contrast -- and with pi of the three
  // adjoint sums pi_c W -- by binning the particles over mesh tiles and one CTA per tile
  // (bin_kernels.cuh).  delta goes to dout (instance stride dis); the pi sums go to the real
  // views of spec_[4..6].
  // Real meshes of the separate deposit, transformed by the x pass of the R2C next: in place
  // in the spectrum buffers (delta in spec_[0] or dens_, pi_c in spec_[4 + c]) when the
  // main rows are in plain order; with z-blocked rows the x pass cannot run in place, and
  // the meshes go to the force mesh buffer (free until the chain's last pass) instead.
  struct SepTargets {
    T* d;
    long long dis;
    T* p[3];
    long long pis;
  };
  SepTargets sep_targets(bool keep_density) {
    SepTargets tg;
    const long long sis = 2 * spec_len_cx(nm_);
    if (spec_zb(nm_) <= 1) {
      tg.d = keep_density ? dens_ : rmesh(0);
      tg.dis = keep_density ? M_ : sis;
      for (int c = 0; c < 3; ++c) tg.p[c] = rmesh(4 + c);
      tg.pis = sis;
    } else {
      T* f = reinterpret_cast<T*>(fvec_);
      tg.d = keep_density ? dens_ : f;
      tg.dis = M_;
      for (int c = 0; c < 3; ++c) tg.p[c] = f + (long long)(1 + c) * B_ * M_;
      tg.pis = M_;
    }
    return tg;
  }
  // Deposits of few particles (nq sums per cell) skip the bins: 64-bit global atomics into an
  // integer mesh and one conversion, two launches instead of five.  The terms are rounded as
  // in the tile deposit and the sums are exact, so the meshes are the same bit for bit.  The
  // line: the atomics run at about 1e11 per second, 8 nq per particle, against some 20 us that
  // the bins take at least; and the integer mesh is 8 nq bytes per cell, read and cleared.
  bool small_rule(int nq) const {
    return nq * (long long)B_ * N_ <= (1LL << 18) && nq * (long long)B_ * M_ <= (1LL << 21);
  }
  // Within the rule the default shape stands for this deposit (the tuner's candidate of that
  // shape times it); any other shape, and the fused form, run as asked.
  bool small_deposit(bool pi) const { return small_deposit(pi, tune_); }
  bool small_deposit(bool pi, const pm_tuning& t) const {
    const int* l = pi ? t.tile_log2_adjoint : t.tile_log2_density;
    const int* l0 = pi ? tune0_.tile_log2_adjoint : tune0_.tile_log2_density;
    return small_rule(pi ? 4 : 1) && std::equal(l, l + 3, l0) && !(t.fused_x & (pi ? 2 : 1)) &&
           (pi ? t.threads_adjoint == tune0_.threads_adjoint : t.threads_density == tune0_.threads_density);
  }
  int scatter_small(const T* s, const T* pi, T* dout, long long dis, const SepTargets& tg) {
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(sacc_);
    const dim3 gp((unsigned)std::min<long long>((N_ + kPtclThreads - 1) / kPtclThreads, kMaxRedBlocks), B_);
    const dim3 gm((unsigned)std::min<long long>((M_ + kPtclThreads - 1) / kPtclThreads, kMaxRedBlocks), B_);
    if (pi) {
      k_scatter<T, 4><<<gp, kPtclThreads, 0, st_>>>(geo_, s, pi, acc, e_d_, e_pi_);
      k_mesh_out<T, 4><<<gm, kPtclThreads, 0, st_>>>(sacc_, M_, e_d_, e_pi_, mass_, dout, dis, tg.p[0], tg.p[1], tg.p[2],
                                                     tg.pis);
    } else {
      k_scatter<T, 1><<<gp, kPtclThreads, 0, st_>>>(geo_, s, nullptr, acc, e_d_, nullptr);
      k_mesh_out<T, 1><<<gm, kPtclThreads, 0, st_>>>(sacc_, M_, e_d_, nullptr, mass_, dout, dis, nullptr, nullptr, nullptr,
                                                     0);
    }
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }
  int scatter(const T* s, const T* pi, T* dout, long long dis, const FusedOut<T>* fo = nullptr,
              const SepTargets* tg = nullptr) {
    if (pi) {
      prof_.begin(st_, P_OTHER, 1);
      k_pi_exponents<<<(3 * B_ + 63) / 64, 64, 0, st_>>>(pimax_, e_pi_, 3 * B_, fixed_top<T>(lgN_));
      prof_.end(st_, P_OTHER);
      PMGB_CK(cudaGetLastError());
      PMGB_CK(cudaMemsetAsync(pimax_, 0, sizeof(unsigned) * 3 * B_, st_));
    }
    const bool pre = counted_;
    counted_ = false;
    if (!fo && small_deposit(pi != nullptr)) {
      prof_.begin(st_, P_SCATTER, 2);
      PMGB_RET(scatter_small(s, pi, dout, dis, tg ? *tg : sep_targets(false)));
      prof_.end(st_, P_SCATTER);
      return PM_OK;
    }
    prof_.begin(st_, P_SCATTER, pre ? 4 : 5);
    if (fo)
      PMGB_RET(deposit(s, pi, nullptr, 0, pi ? bgf4_ : bgf1_, 0, pre, fo));
    else
      PMGB_RET(pi ? deposit(s, pi, dout, dis, bg4_, tune_.threads_adjoint, pre, nullptr, tg)
                  : deposit(s, nullptr, dout, dis, bg1_, tune_.threads_density, pre));
    prof_.end(st_, P_SCATTER);
    return PM_OK;
  }
  // binning + tile-owner deposit with tile geometry bg and nt threads per tile (e_pi_
  // must hold the pi exponents when pi is given)
  // (precounted: the previous gather already counted the bins of s with geometry bg)
  // (fo: the deposit fused with the R2C x pass, into the half spectra of fo; bg is then
  // the whole-row geometry of fused_rows)
  int deposit(const T* s, const T* pi, T* dout, long long dis, const BinGeo& bg, int nt, bool precounted = false,
              const FusedOut<T>* fo = nullptr, const SepTargets* tg = nullptr) {
    const long long nbin = (long long)B_ * bg.nkeys + 1;
    if (nbin > max_bins_) return PM_ERR_STATE;
    const int nscan = (int)((nbin + kScanBlock - 1) / kScanBlock);
    if (!precounted) k_bin_count<T><<<dim3(Gc_, B_), kPtclThreads, 0, st_>>>(geo_, bg, s, bcount_, bkeys_);
    k_scan_blocks<<<nscan, 256, 0, st_>>>(bcount_, bstart_, bsums_, nbin);
    k_scan_add<<<nscan, 256, 0, st_>>>(bstart_, bcursor_, bsums_, nbin);
    if (pi)
      k_bin_fill<T, 4><<<dim3(Gb4_, B_), kPtclThreads, 0, st_>>>(geo_, bg, s, pi, e_pi_, bkeys_, bcursor_, brec0_,
                                                               brec1_);
    else
      k_bin_fill<T, 1><<<dim3(Gb1_, B_), kPtclThreads, 0, st_>>>(geo_, bg, s, nullptr, nullptr, bkeys_, bcursor_,
                                                               brec0_, nullptr);
    if (fo) {
      if (pi)
        PMGB_RET((launch_pull_r2c<T, 4>(nm_, bg, B_, brec0_, brec1_, bstart_, e_d_, e_pi_, mass_, *fo, tw_, st_)));
      else
        PMGB_RET((launch_pull_r2c<T, 1>(nm_, bg, B_, brec0_, nullptr, bstart_, e_d_, nullptr, mass_, *fo, tw_, st_)));
      PMGB_CK(cudaGetLastError());
      return PM_OK;
    }
    const int cells = 1 << (bg.lx + bg.ly + bg.lz);
    const SepTargets dt = tg ? *tg : sep_targets(false);
    const long long pis = dt.pis;
    const dim3 grid(bg.ntiles, B_);
    if (pi) {
      if (nt == 512)
        k_pull_scatter<T, 4, 512><<<grid, 512, 4 * 8 * cells, st_>>>(
            geo_, bg, brec0_, brec1_, bstart_, e_d_, e_pi_, mass_, dout, dis, dt.p[0], dt.p[1], dt.p[2], pis);
      else
        k_pull_scatter<T, 4, 256><<<grid, 256, 4 * 8 * cells, st_>>>(
            geo_, bg, brec0_, brec1_, bstart_, e_d_, e_pi_, mass_, dout, dis, dt.p[0], dt.p[1], dt.p[2], pis);
    } else {
      if (nt == 512)
        k_pull_scatter<T, 1, 512><<<grid, 512, 8 * cells, st_>>>(geo_, bg, brec0_, nullptr, bstart_, e_d_,
                                                                  nullptr, mass_, dout, dis, nullptr, nullptr,
                                                                  nullptr, 0);
      else
        k_pull_scatter<T, 1, 256><<<grid, 256, 8 * cells, st_>>>(geo_, bg, brec0_, nullptr, bstart_, e_d_,
                                                                  nullptr, mass_, dout, dis, nullptr, nullptr,
                                                                  nullptr, 0);
    }
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // Force on the mesh (Sec. 2.2): scatter -> R2C -> Green's function and -ik -> 3 C2R into
  // the [cell][4] mesh fvec_.  With pi also the adjoint chain: pi scatter -> 3 R2C ->
  // sum_c conj(H_c) -> C2R (psi, the fourth component).  The x and y components share
  // the inverse z transform of G delta^ (-i k_1, -i k_2 are constant along a z column and
  // are applied in the y and x passes); the adjoint's x and y terms are combined in the
  // forward y pass, so the z passes transform 3 columns each instead of 4.
  int force_chain(const T* s, const T* pi, bool keep_density) {
    // delta goes to the real view of spec_[0] (transformed in place) or, when the final
    // density is kept for the objective, to dens_
    if (pi ? fused4_ : fused1_) {
      // deposit and x pass in one kernel: delta (and pi_c) straight into the half spectra
      FusedOut<T> fo{};
      fo.spec[0] = spec_[0];
      for (int c = 0; c < 3; ++c) fo.spec[1 + c] = pi ? spec_[4 + c] : nullptr;
      fo.dens = keep_density ? dens_ : nullptr;
      PMGB_RET(scatter(s, pi, nullptr, 0, &fo));
    } else {
      SepTargets tg = sep_targets(keep_density);
      PMGB_RET(scatter(s, pi, tg.d, tg.dis, nullptr, &tg));
      const int nb = pi ? 4 : 1;
      RowJob<T> job{};
      job.b[0] = RowBuf<T>{tg.d, tg.dis, spec_[0]};
      if (pi)
        for (int c = 0; c < 3; ++c) job.b[1 + c] = RowBuf<T>{tg.p[c], tg.pis, spec_[4 + c]};
      job.lzb = spec_lzb(nm_);
      prof_.begin(st_, P_X_R2C, 1);
      PMGB_RET(fft_x_r2c<T>(nm_, job, nb, B_ * nm_ * nm_, tw_, st_));
      prof_.end(st_, P_X_R2C);
      PMGB_CK(cudaGetLastError());
    }
    // y forward: delta (and P_0) in place; the adjoint's P_1 and P_2 merge into
    // V = i (k_1 P_1 + k_2 P_2) in spec_[5]
    C* fwdb[2] = {spec_[0], spec_[4]};
    prof_.begin(st_, P_COLS, (use_tma_ ? 2 : 1) * (pi ? 2 : 1));
    PMGB_RET(cols(nm_, -1, false, fwdb, pi ? 2 : 1));
    if (pi) PMGB_RET(cols_yx(false, spec_[5], spec_[6]));
    prof_.end(st_, P_COLS);
    // z: delta^ -> z force (spec_[1]) and U = IFFT_z(G delta^) (spec_[2])
    ZJob<T> zf{};
    zf.in[0] = spec_[0];
    zf.out[0] = spec_[1];
    zf.out[1] = spec_[2];
    zf.coef = gcoef_;
    zf.dtab = dtab_;
    zf.batch = B_;
    prof_.begin(st_, P_Z_FORCE, use_tma_ ? 2 : 1);
    if (use_tma_) {
      const CUtensorMap fo[2] = {tmf_[1], tmf_[2]};   // z force, U
      PMGB_RET(fft_fused_tma<T>(nm_, false, &tmf_[0], fo, zf, tw_, WaitCtl{dev_err_, first_wait_}, nsm_, st_));
      PMGB_RET(fft_fused_z<T>(nm_, zf, false, false, tw_, st_));
    } else {
      PMGB_RET(fft_fused_z<T>(nm_, zf, false, true, tw_, st_));
    }
    prof_.end(st_, P_Z_FORCE);
    PMGB_CK(cudaGetLastError());
    if (pi) {
      // z: G (i k_0 P_0 + V) -> psi (spec_[0])
      ZJob<T> za = zf;
      za.in[0] = spec_[4];
      za.in[1] = spec_[5];
      za.out[0] = spec_[0];
      za.out[1] = nullptr;
      prof_.begin(st_, P_Z_ADJ, use_tma_ ? 2 : 1);
      if (use_tma_) {
        const CUtensorMap pm2[2] = {tmf_[4], tmf_[5]};
        PMGB_RET(fft_fused_tma<T>(nm_, true, pm2, &tmf_[0], za, tw_, WaitCtl{dev_err_, first_wait_}, nsm_, st_));   // psi -> spec_[0]
        PMGB_RET(fft_fused_z<T>(nm_, za, true, false, tw_, st_));
      } else {
        PMGB_RET(fft_fused_z<T>(nm_, za, true, true, tw_, st_));
      }
      prof_.end(st_, P_Z_ADJ);
      PMGB_CK(cudaGetLastError());
    }
    // y inverse: z force (and psi) in place; U splits into the y force (spec_[2]) and the
    // x force before its -i k_x (spec_[3])
    C* invb[2] = {spec_[1], spec_[0]};
    prof_.begin(st_, P_COLS, use_tma_ ? 4 : 2);
    PMGB_RET(cols(nm_, +1, false, invb, pi ? 2 : 1));
    PMGB_RET(cols_yx(true, spec_[2], spec_[3]));
    prof_.end(st_, P_COLS);
    // C2R of f_0..2 (and psi) into one interleaved [cell][4] mesh for the gathers; the x
    // force takes its -i k_x here
    C* c2rb[4] = {spec_[1], spec_[2], spec_[3], spec_[0]};
    RowJob<T> jc{};
    for (int q = 0; q < 4; ++q) jc.b[q] = RowBuf<T>{nullptr, 0, (q < 3 || pi) ? c2rb[q] : nullptr};
    jc.lzb = spec_lzb(nm_);
    prof_.begin(st_, P_X_C2R, 1);
    PMGB_RET(fft_x_c2r4<T>(nm_, jc, B_ * nm_ * nm_, 2, fvec_, reinterpret_cast<signed char*>(fexp_), tw_, st_));
    prof_.end(st_, P_X_C2R);
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // y pass of the separable force components on the mesh spectra: split (inverse) u ->
  // u = IFFT(-i k_1 u), b = IFFT(u); merge (forward) u = i (k_1 FFT(u) + k_2 FFT(b))
  int cols_yx(bool split, C* u, C* b) {
    const int n = nm_;
    SeqMap mm = ymap(n);
    if (use_tma_) {
      const int iu = spec_index(u), ib = spec_index(b);
      if (iu < 0 || ib < 0) return PM_ERR_STATE;
      const CUtensorMap um[2] = {tmy_[iu], tmy_[ib]};
      if (split)
        PMGB_RET(fft_ysplit_tma<T>(n, B_, um, u, b, tw_, WaitCtl{dev_err_, first_wait_}, nsm_, st_));
      else
        PMGB_RET(fft_ymerge_tma<T>(n, B_, um, u, tw_, WaitCtl{dev_err_, first_wait_}, nsm_, st_));
      PMGB_CK(cudaGetLastError());
      mm.nseq = 0;
    }
    // the main columns (unless staged above) and the side planes (kx = n/2: side
    // sequences, so that k_2 = 0 there) in one launch
    PMGB_RET(split ? fft_cols_split<T>(n, mm, yside(n), u, b, tw_, st_)
                   : fft_cols_merge<T>(n, mm, yside(n), u, b, tw_, st_));
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // Zel'dovich ICs (Sec. 2.1): omega -> R2C -> B_c = i k_c sqrt(P/l_p^3)/k^2 -> 3 C2R -> s1
  int initial_conditions() {
    const long long lis = spec_len_cx(np_);
    // the lattice transforms use spec_[0..3] with the lattice instance stride
    PMGB_RET(lattice_r2c(omega_, N_, spec_[0]));
    k_za_mul<T><<<dim3(Gi_, B_), 256, 0, st_>>>(spec_[0], spec_[1], spec_[2], spec_[3], np_, amp_, maxn2_,
                                                inv_kfp_, lis, (T)0);
    PMGB_CK(cudaGetLastError());
    C* bufs[3] = {spec_[1], spec_[2], spec_[3]};
    PMGB_RET(lattice_c2r(bufs, 3));
    k_ic_state<T><<<dim3(Gi_, B_), 256, 0, st_>>>(rmesh(1), rmesh(2), rmesh(3), 2 * lis, N_, d1_, gd_, s1_, s_, p_);
    PMGB_CK(cudaGetLastError());
    if (lpt2_) PMGB_RET(lpt2_state());
    if (fx_.u) {
      k_fix_init<T><<<dim3(256, B_), 256, 0, st_>>>(s_, p_, fx_, fix_to_u_, 3 * N_);
      PMGB_CK(cudaGetLastError());
    }
    return PM_OK;
  }

  // 2LPT (Sec. 2.1, Eqs. 2-4) from Omega^ in spec_[0]: the Hessian of the first-order
  // potential in two groups of three (diagonal, mixed) through spec_[1..3], the source S
  // accumulated in the real view of spec_[4], s2_c = IDFT[i k_c / k^2 S^] / n^3 through
  // spec_[1..3], then s += D2 s2, p += G_D2 s2.  18 launches.
  int lpt2_state() {
    const long long lis = spec_len_cx(np_);
    C* h[3] = {spec_[1], spec_[2], spec_[3]};
    for (int g = 0; g < 2; ++g) {
      k_lpt_hess<T><<<dim3(Gi_, B_), 256, 0, st_>>>(spec_[0], h[0], h[1], h[2], np_, amp_, maxn2_, lis, g);
      PMGB_CK(cudaGetLastError());
      PMGB_RET(lattice_c2r(h, 3));
      k_lpt_source<T><<<dim3(Gi_, B_), 256, 0, st_>>>(rmesh(1), rmesh(2), rmesh(3), 2 * lis, N_, rmesh(4), 2 * lis,
                                                      g);
      PMGB_CK(cudaGetLastError());
    }
    PMGB_RET(lattice_r2c(rmesh(4), 2 * lis, spec_[4]));
    k_za_mul<T><<<dim3(Gi_, B_), 256, 0, st_>>>(spec_[4], h[0], h[1], h[2], np_, nullptr, maxn2_, inv_kfp_, lis,
                                                unit_);
    PMGB_CK(cudaGetLastError());
    PMGB_RET(lattice_c2r(h, 3));
    k_ic_state2<T><<<dim3(Gi_, B_), 256, 0, st_>>>(rmesh(1), rmesh(2), rmesh(3), 2 * lis, N_, d2_, gd2_, s2_, s_,
                                                   p_);
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // Back-propagation through s2 (the transpose of lpt2_state): sbar2 = D2 xi_0 + G_D2 pi_0
  // and the partials xi_0.s2, pi_0.s2; S_bar = sum_c IDFT[conj(i k_c / k^2) DFT sbar2_c] / n^3
  // (real view of spec_[4]); per Hessian group phi_bar = dS/dphi S_bar, and
  // sum_ij k_i k_j / k^2 amp DFT phi_bar_ij accumulated in spec_[5], where the Zel'dovich
  // transpose adds its part.  Leaves Omega^ in spec_[0].  27 launches.
  int lpt2_adjoint() {
    const long long lis = spec_len_cx(np_);
    k_ic_adj_prep<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(xi_, pi_, s2_, N_, d2_, gd2_, rmesh(1), rmesh(2),
                                                             rmesh(3), 2 * lis, part_, part_ + (long long)B_ * Go_);
    PMGB_CK(cudaGetLastError());
    k_sum_partials<<<2 * B_, 256, 0, st_>>>(part_, Go_, scal_ + 9 * B_, 1.0);
    PMGB_CK(cudaGetLastError());
    RowJob<T> job{};
    for (int c = 0; c < 3; ++c) job.b[c] = RowBuf<T>{rmesh(1 + c), 2 * lis, spec_[1 + c]};
    job.b[3] = RowBuf<T>{omega_, N_, spec_[0]};
    PMGB_RET(fft_x_r2c<T>(np_, job, 4, B_ * np_ * np_, tw_, st_));
    PMGB_CK(cudaGetLastError());
    C* bufs[4] = {spec_[1], spec_[2], spec_[3], spec_[0]};
    PMGB_RET(cols(np_, -1, false, bufs, 4, false));
    PMGB_RET(cols(np_, -1, true, bufs, 4, false));
    k_za_adj_mul<T><<<dim3(Gz_, B_), kPtclThreads, 0, st_>>>(spec_[1], spec_[2], spec_[3], nullptr, nullptr, spec_[4],
                                                             np_, nullptr, unit_, nullptr, maxn2_, inv_kfp_, lis,
                                                             nullptr);
    PMGB_CK(cudaGetLastError());
    C* sb[1] = {spec_[4]};
    PMGB_RET(lattice_c2r(sb, 1));
    C* h[3] = {spec_[1], spec_[2], spec_[3]};
    for (int g = 0; g < 2; ++g) {
      k_lpt_hess<T><<<dim3(Gi_, B_), 256, 0, st_>>>(spec_[0], h[0], h[1], h[2], np_, amp_, maxn2_, lis, g);
      PMGB_CK(cudaGetLastError());
      PMGB_RET(lattice_c2r(h, 3));
      k_lpt_source_adj<T><<<dim3(Gi_, B_), 256, 0, st_>>>(rmesh(1), rmesh(2), rmesh(3), 2 * lis, N_, rmesh(4),
                                                          2 * lis, g);
      PMGB_CK(cudaGetLastError());
      RowJob<T> jh{};
      for (int c = 0; c < 3; ++c) jh.b[c] = RowBuf<T>{rmesh(1 + c), 2 * lis, spec_[1 + c]};
      PMGB_RET(fft_x_r2c<T>(np_, jh, 3, B_ * np_ * np_, tw_, st_));
      PMGB_CK(cudaGetLastError());
      PMGB_RET(cols(np_, -1, false, h, 3, false));
      PMGB_RET(cols(np_, -1, true, h, 3, false));
      k_lpt_hess_adj<T><<<dim3(Gi_, B_), 256, 0, st_>>>(spec_[1], spec_[2], spec_[3], spec_[5], np_, amp_, maxn2_,
                                                        lis, g);
      PMGB_CK(cudaGetLastError());
    }
    return PM_OK;
  }
  int lattice_r2c(const T* in, long long in_is, C* out) {
    RowJob<T> job{};
    job.b[0] = RowBuf<T>{(void*)in, in_is, out};
    PMGB_RET(fft_x_r2c<T>(np_, job, 1, B_ * np_ * np_, tw_, st_));
    C* bufs[1] = {out};
    PMGB_RET(cols(np_, -1, false, bufs, 1, false));
    PMGB_RET(cols(np_, -1, true, bufs, 1, false));
    return PM_OK;
  }
  int lattice_c2r(C* const* bufs, int nb) {
    PMGB_RET(cols(np_, +1, true, bufs, nb, false));
    PMGB_RET(cols(np_, +1, false, bufs, nb, false));
    RowJob<T> jc{};
    for (int q = 0; q < nb; ++q) jc.b[q] = RowBuf<T>{bufs[q], 2 * spec_len_cx(np_), bufs[q]};
    PMGB_RET(fft_x_c2r<T>(np_, jc, nb, B_ * np_ * np_, tw_, st_));
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  // Back-propagation through the ICs (Eq. 51): sbar = D1 xi_0 + G_D pi_0, omega_bar =
  // sum_c B_c^T sbar_c, and the theta terms of P_lin, D1(a0), G_D(a0).
  int ic_adjoint(void* djdw) {
    const long long lis = spec_len_cx(np_);
    if (lpt2_) PMGB_RET(lpt2_adjoint());
    k_ic_adj_prep<T><<<dim3(Go_, B_), kPtclThreads, 0, st_>>>(xi_, pi_, s1_, N_, d1_, gd_, rmesh(1), rmesh(2),
                                                             rmesh(3), 2 * lis, part_, part_ + (long long)B_ * Go_);
    PMGB_CK(cudaGetLastError());
    k_sum_partials<<<2 * B_, 256, 0, st_>>>(part_, Go_, scal_ + 2 * B_, 1.0);
    PMGB_CK(cudaGetLastError());
    // 3 R2C of sbar (in place: real input in the same buffer) and the R2C of omega
    RowJob<T> job{};
    for (int c = 0; c < 3; ++c) job.b[c] = RowBuf<T>{rmesh(1 + c), 2 * lis, spec_[1 + c]};
    job.b[3] = RowBuf<T>{omega_, N_, spec_[0]};
    PMGB_RET(fft_x_r2c<T>(np_, job, 4, B_ * np_ * np_, tw_, st_));
    PMGB_CK(cudaGetLastError());
    C* bufs[4] = {spec_[1], spec_[2], spec_[3], spec_[0]};
    PMGB_RET(cols(np_, -1, false, bufs, 4, false));
    PMGB_RET(cols(np_, -1, true, bufs, 4, false));
    k_za_adj_mul<T><<<dim3(Gz_, B_), kPtclThreads, 0, st_>>>(spec_[1], spec_[2], spec_[3], spec_[0],
                                                             lpt2_ ? spec_[5] : nullptr, spec_[5], np_, amp_, (T)0,
                                                             hdl_, maxn2_, inv_kfp_, lis, part_);
    PMGB_CK(cudaGetLastError());
    k_sum_partials<<<5 * B_, 256, 0, st_>>>(part_, Gz_, scal_ + 4 * B_, 1.0);
    PMGB_CK(cudaGetLastError());
    C* ob[1] = {spec_[5]};
    PMGB_RET(cols(np_, +1, true, ob, 1, false));
    PMGB_RET(cols(np_, +1, false, ob, 1, false));
    RowJob<T> jc{};
    jc.b[0] = RowBuf<T>{djdw ? djdw : (void*)rmesh(5), djdw ? N_ : 2 * lis, spec_[5]};
    PMGB_RET(fft_x_c2r<T>(np_, jc, 1, B_ * np_ * np_, tw_, st_));
    PMGB_CK(cudaGetLastError());
    return PM_OK;
  }

  pm_config cfg_{};
  cudaStream_t st_ = 0;
  int B_ = 1, np_ = 0, nm_ = 0, n_ = 0, lgN_ = 0, e_d_ = 0, G_ = 1, Go_ = 1, Gm_ = 1, Gz_ = 1, nck_ = 0, maxn2_ = 0;
  int Gf_ = 1, Gc_ = 1, Gb1_ = 1, Gb4_ = 1, Gof_ = 1, Goa_ = 1, Gpm_ = 1, Gi_ = 1;   // grids of the particle loops

  // Grid of a particle loop over `work` items of each instance: the blocks that the kernel keeps
  // resident on all SMs, for each instance, or where an instance is no more than kMaxRedBlocks
  // blocks of particles, for the batch; with `sums` always for each instance, so that sums of
  // doubles are grouped alike in a batch and alone, and their bits the same.  (Several whole waves
  // scatter the blocks in flight over the lattice as they drift apart: adjoint gather with three
  // waves 112, 769 and 6323 us at 256^3, 512^3 and 1024^3, with one 102, 742 and 5962; forward gather
  // 73, 506 and 4551 with two, 71, 497 and 4470 with one.  One wave over 16 instances of 128^3 mixes
  // their meshes in the L2: adjoint gather 1204 us against 836 with one each.)
  int wave_grid(const void* fn, long long work, bool sums = false) const {
    const long long need = (work + kPtclThreads - 1) / kPtclThreads;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kPtclThreads, 0) != cudaSuccess || occ < 1) {
      (void)cudaGetLastError();
      occ = 1;
    }
    long long blocks = std::min<long long>((long long)occ * nsm_, kMaxRedBlocks);
    if (!sums && need <= kMaxRedBlocks) blocks /= B_;
    return (int)std::max<long long>(1, std::min(need, blocks));
  }
  long long N_ = 0, M_ = 0, bytes_ = 0;
  T mass_ = 1, inv_kfp_ = 1;
  Geo<T> geo_{};
  std::vector<void*> allocs_;
  T *tgt_ = nullptr, *djdd_ = nullptr, *gw_ = nullptr;
  unsigned long long* pw_acc_ = nullptr;
  unsigned* pw_max_ = nullptr;
  unsigned long long* pw_modes_ = nullptr;   // modes and sum of |n| of each power bin
  double* pw_out_ = nullptr;
  double* pl_buf_ = nullptr;   // power objective: target, weights, g, loss
  std::vector<int> snap_of_;   // observed states: step -> snapshot index (-1: none)
  T* snap_mom_ = nullptr;      // momenta of the observed states (forward output)
  const T* snap_gmom_ = nullptr;   // their cotangents (adjoint input)
  struct InterpObs { int j; };  // an observed scale factor in step j + 1 = (a_j, a_{j+1}]
  std::vector<InterpObs> interp_;
  std::vector<double> interp_a_, theta_host_;
  T *interp_disp_ = nullptr, *interp_dens_ = nullptr;
  const T *interp_gdisp_ = nullptr, *interp_gdens_ = nullptr;
  T *obs_c_ = nullptr, *obs_fac_ = nullptr, *obs_cf_ = nullptr;
  double *obs_w_ = nullptr, *obs_sums_ = nullptr, *obs_part_ = nullptr;
  long long obs_fac_n_ = 0, obs_cf_n_ = 0, obs_w_n_ = 0, obs_sums_n_ = 0;
  T *snap_disp_ = nullptr, *snap_dens_ = nullptr;
  const T *snap_gdisp_ = nullptr, *snap_gdens_ = nullptr;
  bool have_dens_ = false;
  cudaGraphExec_t graph_exec_ = nullptr;
  const void* graph_args_[4] = {nullptr, nullptr, nullptr, nullptr};
  T *s_ = nullptr, *p_ = nullptr, *a_ = nullptr, *xi_ = nullptr, *pi_ = nullptr, *s1_ = nullptr, *omega_ = nullptr;
  BinGeo bg1_{}, bg4_{};
  BinGeo bgf1_{}, bgf4_{};   // whole-row tiles of the deposit fused with the R2C x pass
  bool fused1_ = false, fused4_ = false;
  double fused_ms_[4] = {};   // autotuner: separate and fused deposit times (density, density + pi)
  bool counted_ = false;   // the last gather counted the bins of the next deposit
  pm_tuning tune_{};
  pm_tuning tune0_{};            // the default shapes
  long long* sacc_ = nullptr;    // integer mesh of the small deposits, zero between calls
  long long max_bins_ = 0;       // length of bcount_, bstart_ and bcursor_
  unsigned *bkeys_ = nullptr, *bcount_ = nullptr, *bstart_ = nullptr, *bcursor_ = nullptr, *bsums_ = nullptr;
  V4<T> *brec0_ = nullptr, *brec1_ = nullptr;
  C* spec_[7] = {};
  T* dens_ = nullptr;
  V4<T>* fvec_ = nullptr;
  T *ck_s_ = nullptr, *ck_p_ = nullptr;
  T *fkA_ = nullptr, *fkB_ = nullptr, *fdr_ = nullptr, *rkA_ = nullptr, *rkB_ = nullptr, *rdr_ = nullptr;
  double *wpa_ = nullptr, *wxp_ = nullptr, *dd1_ = nullptr, *dgd_ = nullptr, *dd2_ = nullptr, *dgd2_ = nullptr;
  T *s2_ = nullptr, *d2_ = nullptr, *gd2_ = nullptr, unit_ = 0;
  bool lpt2_ = false;
  T *d1_ = nullptr, *gd_ = nullptr, *gcoef_ = nullptr, *amp_ = nullptr, *dtab_ = nullptr;
  double* hdl_ = nullptr;
  C* tw_ = nullptr;
  unsigned* pimax_ = nullptr;
  int* e_pi_ = nullptr;
  double *part_ = nullptr, *steps_ = nullptr, *scal_ = nullptr, *theta_out_ = nullptr;
  bool have_fwd_ = false;
  long long *fix_u_ = nullptr, *fix_w_ = nullptr;   // fixed-point state (cfg.fixed_state)
  FixState<T> fx_{};
  T fix_to_u_ = 0;
  Prof prof_;
  bool use_tma_ = false;
  int nsm_ = 1;   // SM count
  bool hf_ = false;        // pm_config.half_force: the FP16 [cell][4] force mesh (FP32 path)
  int* fexp_ = nullptr;    // its int8 exponent quadruples, one int per mesh row [B][n][n]
  // the gathers of the force mesh in its stored form (OP: the operators' form)
  template <bool OP = false> decltype(&k_gather_fwd<T, false, false>) gather_fwd_fn() const {
    if constexpr (sizeof(T) == 4)
      if (hf_) return &k_gather_fwd<T, true, OP>;
    return &k_gather_fwd<T, false, OP>;
  }
  template <bool OP = false> decltype(&k_gather_adj<T, false, false>) gather_adj_fn() const {
    if constexpr (sizeof(T) == 4)
      if (hf_) return &k_gather_adj<T, true, OP>;
    return &k_gather_adj<T, false, OP>;
  }
  cudaStream_t cp_st_ = nullptr;                       // copy stream of pm_gradient's target
  cudaEvent_t cp_in_ = nullptr, cp_done_ = nullptr;     // its order after st_, its completion
  int* err_host_ = nullptr;   // set by a bounded device wait that gave up (host memory)
  int* dev_err_ = nullptr;    // its device address
  int first_wait_ = -1;   // spin limit of the TMA passes' first wait (test hook)
  CUtensorMap tmy_[7], tmz_[7], tmf_[7];   // y, z and fused z passes of spec_[q]
};

template <typename T>
int make_engine_t(const pm_config* cfg, const double* theta, const void* omega, cudaStream_t st, EngineBase** out) {
  Engine<T>* e = new Engine<T>();
  const int r = e->init(cfg, theta, omega, st);
  if (r != PM_OK) {
    delete e;
    return r;
  }
  *out = e;
  return PM_OK;
}

}  // namespace pmgb
