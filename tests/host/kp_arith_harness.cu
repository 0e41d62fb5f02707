// Host-only harness of the loop kernel's arithmetic rules (kp_arith.cuh), for
// CPU tests: the functions that the kernel calls, compiled for the host.
#include "../../paper_2409_06807_gb300/csrc/kp_arith.cuh"
#include "../../paper_2409_06807_gb300/csrc/kp_layout.h"

using namespace kp;

extern "C" {

void kpt_key_quot(int lam, const int* keys, int n, int* out) {
  const KeyDiv kd(lam);
  for (int i = 0; i < n; ++i) out[i] = kd.quot(keys[i]);
}

int kpt_bias(int gx, int gy, int gz) {
  const int32_t g[3] = {gx, gy, gz};
  return bp_bias_of(g);
}

void kpt_within(const float* d, int n, int q, unsigned char* out) {
  for (int i = 0; i < n; ++i) out[i] = within_clearance(d[i], q) ? 1 : 0;
}

void kpt_threshold_of(const double* p, int n, uint64_t* out) {
  for (int i = 0; i < n; ++i) out[i] = threshold_of(p[i]);
}

// The thresholds of scores under a sum, as the kernel takes them (1 / sum where
// it has one) and always by the division; returns whether it has one.
int kpt_thresholds(const double* score, int n, double sum, double eps, uint64_t* fast, uint64_t* slow) {
  const ScoreSum s = score_sum_of(sum, eps);
  for (int i = 0; i < n; ++i) {
    fast[i] = accept_threshold(score[i], s.sum, s.inv, eps);
    slow[i] = accept_threshold(score[i], s.sum, 0.0, eps);
  }
  return s.inv != 0.0;
}

// Draws w[i] against score[i]: the answer, and whether it was decided in FP32.
void kpt_draws(const uint32_t* w, const double* score, int n, double sum, double eps,
               unsigned char* out, unsigned char* decided) {
  const ScoreSum s = score_sum_of(sum, eps);
  for (int i = 0; i < n; ++i) {
    bool below;
    out[i] = draw_accepted(w[i], score[i], s, eps) ? 1 : 0;
    decided[i] = draw_decided(w[i], score[i], s, &below) ? 1 : 0;
  }
}

}  // extern "C"
