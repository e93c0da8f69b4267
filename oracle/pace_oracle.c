/*
 * PACE oracle: a plain, slow, fp64 CPU statement of what the PACE hot path
 * computes.  TEST INFRASTRUCTURE ONLY: it exists so that the test-suite, the
 * smoke check and the CPU-baseline leg of the benchmark can compare the CUDA
 * library against an independent reading of the paper.  Nothing in the
 * product path may call it, and it shares no code, header or constant table
 * with the CUDA library.
 *
 * Paper: "Where Does Staleness Accumulate? Pool Aware Effective Staleness
 * Control for Asynchronous RL in LLM Post-Training" (PACE).
 *
 * Each function cites the passage it follows.  Arithmetic is IEEE fp64 with
 * FP contraction disabled at build time (-ffp-contract=off), so every product
 * and sum is rounded once, in the order written here.
 *
 * Parity status of each function (what pins it, see tests/test_oracle_*.py):
 *   oracle_policy_lag, oracle_staleness   Lemma 1 integer identity, hand pool
 *   oracle_ecdf, oracle_sharpen           hand pool fractions, closed forms
 *   oracle_score_pool                     hand pool (all three modes)
 *   oracle_budget                         hand pool, EMA example, r = 0 case,
 *                                         rational-arithmetic sweep
 *   oracle_select                         brute-force k-subset enumeration
 *   oracle_token_logprob                  fp64 log_softmax of a library, W = 0
 *                                         closed form, one-hot hidden rows
 *   oracle_group_advantages               closed forms (two-member groups)
 *   oracle_surrogate                      hand-worked clip branches, ratio-1
 *                                         on-policy identity
 *   oracle_stale_k                        hand pool kbar column, threshold
 *                                         boundaries (kbar == k is admitted)
 *   oracle_histogram                      hand-counted bins, totals, clamping
 *   oracle_quantile_admit                 hand-worked window / draw sequences,
 *                                         numpy inverted-CDF quantile
 *   oracle_surrogate_grad                 central finite differences of
 *                                         oracle_surrogate away from its kinks
 *   oracle_lmhead_backward                fp64 autograd of a library on small
 *                                         shapes, vocabulary-sum-zero identity
 *   oracle_lmhead_backward_magnitude      |G| from fp64 autograd of a library
 *                                         times |W| and |H|; bounds |dH|, |dW|
 *   oracle_prefix_score                   hand-worked prefixes, zero / constant
 *                                         drift identities, min-token and cap
 *                                         boundaries
 * No function is "parity unpinned".
 */
#include <math.h>
#include <pthread.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

/* Status codes of the oracle (numbering chosen to read the same as the
 * library's public codes, so tests can compare them directly). */
enum {
  OR_OK = 0,
  OR_ERR_INVALID_ARG = 1,
  OR_ERR_VERSION_ORDER = 2, /* v_t > c(tau) or c(tau) > j: Lemma 1 premise */
  OR_ERR_NAN_INPUT = 3,
};

enum { OR_MODE_EFF = 0, OR_MODE_RAW = 1, OR_MODE_GEN = 2 };
enum { OR_AGG_TOKEN_MEAN = 0, OR_AGG_SEQ_MEAN_TOKEN_MEAN = 1 };

/* A per-token version tag of -1 marks a token not generated by the policy
 * (tool output in multi-turn rollouts); it carries no policy version and is
 * left out of every staleness sum. */
#define OR_NO_VERSION (-1)

static int check_offsets(const int64_t* offsets, int64_t n_traj, int64_t n_tokens) {
  if (n_traj < 0) return OR_ERR_INVALID_ARG;
  if (offsets[0] != 0) return OR_ERR_INVALID_ARG;
  for (int64_t i = 0; i < n_traj; ++i)
    if (offsets[i + 1] < offsets[i]) return OR_ERR_INVALID_ARG;
  if (n_tokens >= 0 && offsets[n_traj] != n_tokens) return OR_ERR_INVALID_ARG;
  return OR_OK;
}

/* Eq. 1 (Sec. 2, "Trajectory Lifecycle and Policy Lag"): the token-weighted
 * policy lag  kbar(tau; j) = (1/T) * sum_t (j - v_t)  over the response tokens
 * that carry a policy version.  T = 0 gives 0.  Used by the tests to check the
 * Lemma 1 identity; not part of the hot path. */
int oracle_policy_lag(const int32_t* tags, const int64_t* offsets, int64_t n_traj,
                      int32_t j, int64_t* lag_sum, int64_t* n_policy_tokens, double* kbar) {
  int st = check_offsets(offsets, n_traj, -1);
  if (st) return st;
  for (int64_t i = 0; i < n_traj; ++i) {
    int64_t s = 0, t_count = 0;
    for (int64_t t = offsets[i]; t < offsets[i + 1]; ++t) {
      if (tags[t] == OR_NO_VERSION) continue;
      s += (int64_t)j - (int64_t)tags[t];
      t_count += 1;
    }
    lag_sum[i] = s;
    n_policy_tokens[i] = t_count;
    kbar[i] = t_count > 0 ? (double)s / (double)t_count : 0.0;
  }
  return OR_OK;
}

/* Lemma 1 / Eq. 2 (Sec. 2, "Staleness Decomposition"):
 *   K_gen(tau)    = (1/T) * sum_t (c(tau) - v_t)
 *   K_wait(tau;j) = j - c(tau)
 * under the premise v_t <= c(tau) <= j.  The numerator is summed exactly in
 * 64-bit integers and divided once.  Violating the premise is an error
 * (OR_ERR_VERSION_ORDER); a tag below -1 or a negative c is invalid. */
int oracle_staleness(const int32_t* tags, const int64_t* offsets, const int32_t* c_version,
                     int64_t n_traj, int64_t n_tokens, int32_t j,
                     int64_t* gen_sum, int64_t* n_policy_tokens, double* kgen, double* kwait) {
  int st = check_offsets(offsets, n_traj, n_tokens);
  if (st) return st;
  int err = OR_OK;
  for (int64_t i = 0; i < n_traj; ++i) {
    const int64_t c = c_version[i];
    if (c < 0) return OR_ERR_INVALID_ARG;
    int64_t s = 0, t_count = 0;
    for (int64_t t = offsets[i]; t < offsets[i + 1]; ++t) {
      const int64_t v = tags[t];
      if (v == OR_NO_VERSION) continue;
      if (v < 0) return OR_ERR_INVALID_ARG;
      if (v > c && !err) err = OR_ERR_VERSION_ORDER;
      s += c - v;
      t_count += 1;
    }
    if (c > (int64_t)j && !err) err = OR_ERR_VERSION_ORDER;
    gen_sum[i] = s;
    n_policy_tokens[i] = t_count;
    kgen[i] = t_count > 0 ? (double)s / (double)t_count : 0.0;
    kwait[i] = (double)((int64_t)j - c);
  }
  return err;
}

/* Eq. 9 (Sec. 3.2, "Effective Staleness"): empirical percentile rank of a
 * prefix score within the window W^pre of recent prefix scores.  The ECDF is
 * taken right-continuous: the count of window values w with w <= s, compared
 * in float32 (the precision scores are stored in), divided by |W|. */
double oracle_ecdf(const float* window, int64_t window_len, float s) {
  int64_t cnt = 0;
  for (int64_t i = 0; i < window_len; ++i)
    if (window[i] <= s) cnt += 1;
  return (double)cnt / (double)window_len;
}

/* Eq. 10 (Sec. 3.2): temperature sharpening
 *   phi_gamma(q) = q^gamma / (q^gamma + (1 - q)^gamma),  gamma >= 1,
 * for integer gamma, each power formed by repeated multiplication from the
 * left (q, q*q, (q*q)*q, ...). */
double oracle_sharpen(double q, int32_t gamma) {
  double a = q;
  double one_minus_q = 1.0 - q;
  double b = one_minus_q;
  for (int32_t g = 1; g < gamma; ++g) {
    a = a * q;
    b = b * one_minus_q;
  }
  return a / (a + b);
}

/* Whole-pool scoring, Eqs. 2, 7, 8, 9, 10 (Sec. 3.2) and the group
 * aggregation of the experimental settings ("mean aggregation within
 * groups"):
 *   EFF (PACE):            M = K_wait + F * K_gen      (w1 = 1, w2 = F)
 *   RAW (Raw Staleness):   M = K_wait + K_gen          (w1 = 1, w2 = 1)
 *   GEN (Gen. Staleness):  M = F * K_gen               (w1 = 0, w2 = F)
 * with F = phi_gamma(ECDF_W(s_pre)).  F = f_missing when s_pre is NaN (no
 * prefix was rescored), and F = 1 for every trajectory when the window holds
 * fewer than min_obs observations.  The unit score of group u is the sum of
 * its G member scores, taken from the lowest id upward, divided by G. */
int oracle_score_pool(const int32_t* tags, const int64_t* offsets, const int32_t* c_version,
                      const float* s_pre, int64_t n_traj, int64_t n_tokens, int32_t j,
                      const float* window, int64_t window_len, int32_t mode, int32_t gamma,
                      int32_t min_obs, double f_missing, int32_t group_size,
                      double* kgen, double* kwait, double* weight, double* score,
                      double* unit_score) {
  if (n_traj < 0 || group_size < 1 || gamma < 1 || window_len < 0) return OR_ERR_INVALID_ARG;
  if (mode != OR_MODE_EFF && mode != OR_MODE_RAW && mode != OR_MODE_GEN) return OR_ERR_INVALID_ARG;
  if (n_traj % group_size != 0) return OR_ERR_INVALID_ARG;
  for (int64_t w = 0; w < window_len; ++w)
    if (isnan(window[w])) return OR_ERR_NAN_INPUT;

  int64_t* gen_sum = (int64_t*)malloc(sizeof(int64_t) * (size_t)(n_traj > 0 ? n_traj : 1));
  int64_t* t_count = (int64_t*)malloc(sizeof(int64_t) * (size_t)(n_traj > 0 ? n_traj : 1));
  int st = oracle_staleness(tags, offsets, c_version, n_traj, n_tokens, j, gen_sum, t_count, kgen, kwait);
  free(gen_sum);
  free(t_count);
  if (st) return st;

  const int window_ready = window_len >= (int64_t)min_obs && window_len > 0;
  for (int64_t i = 0; i < n_traj; ++i) {
    double f;
    if (!window_ready) f = 1.0;
    else if (isnan(s_pre[i])) f = f_missing;
    else f = oracle_sharpen(oracle_ecdf(window, window_len, s_pre[i]), gamma);
    weight[i] = f;
    if (mode == OR_MODE_EFF) score[i] = kwait[i] + f * kgen[i];
    else if (mode == OR_MODE_RAW) score[i] = kwait[i] + kgen[i];
    else score[i] = f * kgen[i];
  }
  const int64_t n_units = n_traj / group_size;
  for (int64_t u = 0; u < n_units; ++u) {
    double acc = 0.0;
    for (int32_t g = 0; g < group_size; ++g) acc = acc + score[u * group_size + g];
    unit_score[u] = acc / (double)group_size;
  }
  return OR_OK;
}

/* Eq. 3 and Eq. 4 (Sec. 3.1) with the maximum rejection budget of the
 * experimental settings:
 *   r_j     = clip((N_j - N_tar) / max(N_j, 1), 0, 1)
 *   rhat_j  = beta * rhat_{j-1} + (1 - beta) * r_j,   beta in [0, 1)
 *   r_eff   = min(rhat_j, r_max)
 * The number of units to reject is floor(r_eff * U + 1e-9), at most U.  The
 * 1e-9 nudge makes the floor land on the exact integer when r_eff * U is an
 * integer that fp64 rounding left just below it (e.g. N = 47, N_tar = 35). */
int oracle_budget(int64_t n_traj, int64_t n_target, double beta, double r_max,
                  double r_hat_prev, int64_t n_units, double* r_out, double* r_hat_out,
                  int64_t* k_out) {
  if (n_traj < 0 || n_target < 0 || n_units < 0) return OR_ERR_INVALID_ARG;
  if (!(beta >= 0.0 && beta < 1.0)) return OR_ERR_INVALID_ARG;
  if (!(r_max >= 0.0 && r_max <= 1.0)) return OR_ERR_INVALID_ARG;
  if (!(r_hat_prev >= 0.0 && r_hat_prev <= 1.0)) return OR_ERR_INVALID_ARG;
  const int64_t denom = n_traj > 1 ? n_traj : 1;
  double r = (double)(n_traj - n_target) / (double)denom;
  if (r < 0.0) r = 0.0;
  if (r > 1.0) r = 1.0;
  const double r_hat = beta * r_hat_prev + (1.0 - beta) * r;
  const double r_eff = r_hat < r_max ? r_hat : r_max;
  int64_t k = (int64_t)floor(r_eff * (double)n_units + 1e-9);
  if (k > n_units) k = n_units;
  if (k < 0) k = 0;
  *r_out = r;
  *r_hat_out = r_hat;
  *k_out = k;
  return OR_OK;
}

/* Rejection of the k highest-scored units (Sec. 3.1 quantile rule, read as
 * "reject the upper r-hat fraction of the current pool"; Algorithm 1, trainer
 * side).  Units are ordered by score, largest first, and equal scores by unit
 * id, smallest first; the first k in that order are rejected.  Unit u stands
 * for trajectories u*G .. u*G+G-1.  Outputs are trajectory ids in ascending
 * order. */
typedef struct {
  double score;
  int64_t id;
} unit_key;

static int unit_key_cmp(const void* pa, const void* pb) {
  const unit_key* a = (const unit_key*)pa;
  const unit_key* b = (const unit_key*)pb;
  if (a->score > b->score) return -1;
  if (a->score < b->score) return 1;
  return (a->id < b->id) ? -1 : (a->id > b->id) ? 1 : 0;
}

int oracle_select(const double* unit_score, int64_t n_units, int32_t group_size, int64_t k,
                  int32_t* accepted_ids, int32_t* rejected_ids, uint8_t* traj_accepted) {
  if (n_units < 0 || group_size < 1 || k < 0 || k > n_units) return OR_ERR_INVALID_ARG;
  for (int64_t u = 0; u < n_units; ++u)
    if (isnan(unit_score[u])) return OR_ERR_NAN_INPUT;
  unit_key* keys = (unit_key*)malloc(sizeof(unit_key) * (size_t)(n_units > 0 ? n_units : 1));
  uint8_t* rejected = (uint8_t*)calloc((size_t)(n_units > 0 ? n_units : 1), 1);
  for (int64_t u = 0; u < n_units; ++u) {
    keys[u].score = unit_score[u];
    keys[u].id = u;
  }
  qsort(keys, (size_t)n_units, sizeof(unit_key), unit_key_cmp);
  for (int64_t r = 0; r < k; ++r) rejected[keys[r].id] = 1;
  int64_t na = 0, nr = 0;
  for (int64_t u = 0; u < n_units; ++u) {
    for (int32_t g = 0; g < group_size; ++g) {
      const int64_t id = u * group_size + g;
      if (rejected[u]) rejected_ids[nr++] = (int32_t)id;
      else accepted_ids[na++] = (int32_t)id;
      if (traj_accepted) traj_accepted[id] = rejected[u] ? 0 : 1;
    }
  }
  free(keys);
  free(rejected);
  return OR_OK;
}

/* bf16 storage to a real number: the 16 bits are the top half of an IEEE
 * binary32; the widening to fp64 is exact. */
static double bf16_to_double(uint16_t bits) {
  uint32_t w = (uint32_t)bits << 16;
  float f;
  memcpy(&f, &w, sizeof f);
  return (double)f;
}

/* Per-token log-probability under the current policy (Sec. 2: the policy
 * factorises over tokens; the update consumes log pi_theta_j(y_t | x, y_<t);
 * training temperature 1.0 in the shared settings):
 *   z_v   = h_r . W_v                   (fp64 dot product, k ascending)
 *   lse   = log sum_v exp(z_v / tau)    (two passes: maximum, then sum)
 *   lp_r  = z_{y_r} / tau - lse
 * on the bf16 values of the hidden row h_r and vocabulary rows W_v.  Rows are
 * split across n_threads worker threads; each row is computed by one thread
 * in the order above. */
typedef struct {
  const uint16_t* hidden;
  const uint16_t* w;
  const int32_t* targets;
  const int64_t* row_ids;
  int64_t r_begin, r_end;
  int32_t H, V;
  double tau;
  double* logprob;
  double* lse;
  int status;
} lp_job;

static void* lp_worker(void* arg) {
  lp_job* jb = (lp_job*)arg;
  double* z = (double*)malloc(sizeof(double) * (size_t)jb->V);
  double* h = (double*)malloc(sizeof(double) * (size_t)jb->H);
  for (int64_t r = jb->r_begin; r < jb->r_end; ++r) {
    const int64_t row = jb->row_ids ? jb->row_ids[r] : r;
    const uint16_t* hr = jb->hidden + (size_t)row * (size_t)jb->H;
    for (int32_t k = 0; k < jb->H; ++k) h[k] = bf16_to_double(hr[k]);
    for (int32_t v = 0; v < jb->V; ++v) {
      const uint16_t* wv = jb->w + (size_t)v * (size_t)jb->H;
      double acc = 0.0;
      for (int32_t k = 0; k < jb->H; ++k) acc = acc + h[k] * bf16_to_double(wv[k]);
      z[v] = acc / jb->tau;
    }
    double m = -INFINITY;
    for (int32_t v = 0; v < jb->V; ++v)
      if (z[v] > m) m = z[v];
    double s = 0.0;
    for (int32_t v = 0; v < jb->V; ++v) s = s + exp(z[v] - m);
    const double lse = m + log(s);
    const int32_t y = jb->targets[row];
    if (y < 0 || y >= jb->V) {
      jb->status = OR_ERR_INVALID_ARG;
      jb->logprob[r] = NAN;
    } else {
      jb->logprob[r] = z[y] - lse;
    }
    if (jb->lse) jb->lse[r] = lse;
  }
  free(z);
  free(h);
  return NULL;
}

int oracle_token_logprob(const uint16_t* hidden, const uint16_t* w_vocab, const int32_t* targets,
                         const int64_t* row_ids, int64_t n_rows, int32_t H, int32_t V,
                         double temperature, double* logprob, double* lse, int32_t n_threads) {
  if (n_rows < 0 || H < 1 || V < 1 || !(temperature > 0.0)) return OR_ERR_INVALID_ARG;
  if (n_threads < 1) n_threads = 1;
  if (n_threads > 256) n_threads = 256;
  if ((int64_t)n_threads > n_rows) n_threads = n_rows > 0 ? (int32_t)n_rows : 1;
  lp_job jobs[256];
  pthread_t th[256];
  const int64_t per = (n_rows + n_threads - 1) / n_threads;
  for (int32_t t = 0; t < n_threads; ++t) {
    lp_job* jb = &jobs[t];
    jb->hidden = hidden;
    jb->w = w_vocab;
    jb->targets = targets;
    jb->row_ids = row_ids;
    jb->r_begin = (int64_t)t * per < n_rows ? (int64_t)t * per : n_rows;
    jb->r_end = jb->r_begin + per < n_rows ? jb->r_begin + per : n_rows;
    jb->H = H;
    jb->V = V;
    jb->tau = temperature;
    jb->logprob = logprob;
    jb->lse = lse;
    jb->status = OR_OK;
  }
  for (int32_t t = 1; t < n_threads; ++t) pthread_create(&th[t], NULL, lp_worker, &jobs[t]);
  lp_worker(&jobs[0]);
  for (int32_t t = 1; t < n_threads; ++t) pthread_join(th[t], NULL);
  for (int32_t t = 0; t < n_threads; ++t)
    if (jobs[t].status) return jobs[t].status;
  return OR_OK;
}

/* GRPO within-group standardisation (experimental settings: "GRPO with
 * within-group standardization"): for the accepted members of each prompt
 * group (sequences g*G .. g*G+G-1),
 *   A_i = (R_i - mean_g) / (std_g + eps)
 * with the sample standard deviation (divisor n - 1) when unbiased != 0 and
 * the population one otherwise.  A member whose reward equals the group mean
 * gets A = 0 even when std + eps is 0 (one accepted member, or all rewards
 * equal with eps = 0), instead of 0/0.  Rejected members get A = 0. */
int oracle_group_advantages(const float* reward, const uint8_t* seq_accepted, int64_t n_seq,
                            int32_t group_size, double eps, int32_t unbiased, double* adv) {
  if (n_seq < 0 || group_size < 1 || n_seq % group_size != 0) return OR_ERR_INVALID_ARG;
  for (int64_t g0 = 0; g0 < n_seq; g0 += group_size) {
    int64_t n = 0;
    double sum = 0.0;
    for (int64_t i = g0; i < g0 + group_size; ++i) {
      if (seq_accepted && !seq_accepted[i]) continue;
      sum = sum + (double)reward[i];
      n += 1;
    }
    const double mean = n > 0 ? sum / (double)n : 0.0;
    double ss = 0.0;
    for (int64_t i = g0; i < g0 + group_size; ++i) {
      if (seq_accepted && !seq_accepted[i]) continue;
      const double d = (double)reward[i] - mean;
      ss = ss + d * d;
    }
    const int64_t div = unbiased ? n - 1 : n;
    const double sd = div > 0 ? sqrt(ss / (double)div) : 0.0;
    for (int64_t i = g0; i < g0 + group_size; ++i) {
      if (seq_accepted && !seq_accepted[i]) adv[i] = 0.0;
      else {
        const double d = (double)reward[i] - mean;
        adv[i] = d == 0.0 ? 0.0 : d / (sd + eps);
      }
    }
  }
  return OR_OK;
}

/* The policy objective the trainer applies to the accepted batch (shared
 * experimental settings: asymmetric clipping 0.20 / 0.28, dual-clip
 * coefficient 10, token-mean loss aggregation; the ratio uses the recorded
 * rollout log-probabilities as behaviour reference):
 *   rho_t = exp(clamp(lp_t - l^mu_t, -20, 20))
 *   L_t   = max(-A rho_t, -A clip(rho_t, 1 - eps_low, 1 + eps_high))
 *   L_t   = min(L_t, -c A)                      when A < 0 (dual clip)
 * TOKEN_MEAN:              loss = sum_t m_t L_t / sum_t m_t
 * SEQ_MEAN_TOKEN_MEAN:     loss = mean over sequences with tokens of
 *                                 (sum_t m_t L_t / sum_t m_t) per sequence
 * A row is in the loss when its mask byte is non-zero and its sequence is
 * accepted; an empty loss is 0.  Sums run over rows in ascending order. */
int oracle_surrogate(const double* logprob, const double* behav_lp, const uint8_t* mask,
                     const int64_t* seq_offsets, const uint8_t* seq_accepted, int64_t n_seq,
                     const double* adv, double eps_low, double eps_high, double dual_clip,
                     int32_t agg, double* loss, double* ratio_out, double* term_out) {
  if (n_seq < 0) return OR_ERR_INVALID_ARG;
  if (agg != OR_AGG_TOKEN_MEAN && agg != OR_AGG_SEQ_MEAN_TOKEN_MEAN) return OR_ERR_INVALID_ARG;
  int st = check_offsets(seq_offsets, n_seq, -1);
  if (st) return st;
  double tot = 0.0, cnt = 0.0, seq_tot = 0.0;
  int64_t n_seq_used = 0;
  for (int64_t i = 0; i < n_seq; ++i) {
    const int seq_in = seq_accepted ? seq_accepted[i] != 0 : 1;
    const double a = adv[i];
    double s_tot = 0.0, s_cnt = 0.0;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1]; ++r) {
      const int in = seq_in && (mask ? mask[r] != 0 : 1);
      double d = logprob[r] - behav_lp[r];
      if (d < -20.0) d = -20.0;
      if (d > 20.0) d = 20.0;
      const double rho = exp(d);
      double rc = rho;
      if (rc < 1.0 - eps_low) rc = 1.0 - eps_low;
      if (rc > 1.0 + eps_high) rc = 1.0 + eps_high;
      const double p1 = -a * rho;
      const double p2 = -a * rc;
      double l = p1 > p2 ? p1 : p2;
      if (a < 0.0) {
        const double p3 = -dual_clip * a;
        if (p3 < l) l = p3;
      }
      if (ratio_out) ratio_out[r] = in ? rho : 0.0;
      if (term_out) term_out[r] = in ? l : 0.0;
      if (!in) continue;
      tot = tot + l;
      cnt = cnt + 1.0;
      s_tot = s_tot + l;
      s_cnt = s_cnt + 1.0;
    }
    if (s_cnt > 0.0) {
      seq_tot = seq_tot + s_tot / s_cnt;
      n_seq_used += 1;
    }
  }
  if (agg == OR_AGG_TOKEN_MEAN) *loss = cnt > 0.0 ? tot / cnt : 0.0;
  else *loss = n_seq_used > 0 ? seq_tot / (double)n_seq_used : 0.0;
  return OR_OK;
}

/* Prefix Forgetting Score, Eq. 6 (Sec. 3.2), with the collection rules of the
 * admission settings (scores need at least min_tokens eligible tokens; only
 * the first cap_tokens eligible response tokens are scored):
 *   s_pre = (1/m) * sum_{t <= m} | log pi_u(y_t | x, y_<t) - l^mu_t |
 * over the first m = min(#eligible, cap_tokens) eligible rows of each prefix
 * (rows with a non-zero mask byte, in row order), or NaN when the prefix has
 * fewer than min_tokens eligible rows.  logprob holds log pi_u of each row
 * (from oracle_token_logprob under the rescoring policy u). */
int oracle_prefix_score(const double* logprob, const double* behav_lp, const uint8_t* mask,
                        const int64_t* seq_offsets, int64_t n_seq, int32_t min_tokens,
                        int32_t cap_tokens, double* s_pre) {
  if (n_seq < 0 || min_tokens < 1 || cap_tokens < 1) return OR_ERR_INVALID_ARG;
  int st = check_offsets(seq_offsets, n_seq, -1);
  if (st) return st;
  for (int64_t i = 0; i < n_seq; ++i) {
    int64_t eligible = 0;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1]; ++r)
      if (!mask || mask[r]) eligible += 1;
    if (eligible < min_tokens) {
      s_pre[i] = NAN;
      continue;
    }
    const int64_t m = eligible < cap_tokens ? eligible : cap_tokens;
    double sum = 0.0;
    int64_t used = 0;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1] && used < m; ++r) {
      if (mask && !mask[r]) continue;
      sum = sum + fabs(logprob[r] - behav_lp[r]);
      used += 1;
    }
    s_pre[i] = sum / (double)m;
  }
  return OR_OK;
}

/* Stale-k admission (Sec. 2, "Controlled Stale-k Analysis", the prior-work
 * baseline): a trajectory is admitted when its token-weighted policy lag
 * kbar(tau; j) of Eq. 1 is at most k_max.  kbar is returned too; a trajectory
 * with no policy tokens has kbar = 0 and is admitted. */
int oracle_stale_k(const int32_t* tags, const int64_t* offsets, int64_t n_traj, int32_t j,
                   double k_max, double* kbar, uint8_t* admitted) {
  int64_t* s = (int64_t*)malloc(sizeof(int64_t) * (size_t)(n_traj > 0 ? n_traj : 1));
  int64_t* t = (int64_t*)malloc(sizeof(int64_t) * (size_t)(n_traj > 0 ? n_traj : 1));
  int st = oracle_policy_lag(tags, offsets, n_traj, j, s, t, kbar);
  free(s);
  free(t);
  if (st) return st;
  for (int64_t i = 0; i < n_traj; ++i) admitted[i] = kbar[i] <= k_max ? 1 : 0;
  return OR_OK;
}

/* Staleness diagnostics (the retained-vs-rejected histograms of the admission
 * analysis): counts of values in n_bins equal-width bins over [lo, hi), values
 * below lo in the first bin and at or above hi in the last; hist[0..n_bins) for
 * rejected entries (flag 0), hist[n_bins..2 n_bins) for accepted (flag != 0).
 * The bin of x is floor((x - lo) / (hi - lo) * n_bins), computed in fp64; where hi - lo
 * overflows that is bin 0 (the quotient is 0, or NaN where x - lo overflows too). */
int oracle_histogram(const double* values, const uint8_t* flags, int64_t n, double lo,
                     double hi, int32_t n_bins, uint32_t* hist) {
  if (n < 0 || n_bins < 1 || !(hi > lo)) return OR_ERR_INVALID_ARG;
  for (int32_t b = 0; b < 2 * n_bins; ++b) hist[b] = 0;
  for (int64_t i = 0; i < n; ++i) {
    const double x = values[i];
    if (isnan(x)) return OR_ERR_NAN_INPUT;
    int64_t b;
    if (x < lo) b = 0;
    else if (x >= hi) b = n_bins - 1;
    else {
      const double f = floor((x - lo) / (hi - lo) * (double)n_bins);
      b = !(f > 0.0) ? 0 : (f > (double)(n_bins - 1) ? n_bins - 1 : (int64_t)f);
    }
    hist[(flags && flags[i] ? n_bins : 0) + b] += 1;
  }
  return OR_OK;
}

static int double_cmp(const void* pa, const void* pb) {
  const double a = *(const double*)pa, b = *(const double*)pb;
  return a < b ? -1 : (a > b ? 1 : 0);
}

/* The literal admission rule of Sec. 3.1 and Algorithm 1 (trainer side):
 *   kappa = Quantile_{1 - r}(W^M)   over the window of recently observed scores
 * with the inverted-CDF (type-1) quantile: the k-th smallest window value,
 * k = max(ceil((1 - r) |W| - 1e-9), 1) (the nudge keeps an exact product such as
 * 0.75 * 512 from rounding up to the next rank).  Candidates are drawn in the
 * given order; a candidate with score > kappa is rejected (decision 0), the
 * others are retained (1) until batch_units are retained; candidates after that
 * are not drawn (2).  With fewer than min_obs scores in the window there is no
 * threshold (kappa = +inf) and every drawn candidate is retained.  batch_units
 * <= 0 draws every candidate.  Every drawn score, retained or rejected, then
 * enters the window (a ring of `capacity` slots: count, head = next slot). */
int oracle_quantile_admit(const double* score, int64_t n_cand, double r, int64_t batch_units,
                          int32_t min_obs, double* window, int64_t capacity, int64_t* count,
                          int64_t* head, uint8_t* decision, double* kappa_out) {
  if (n_cand < 0 || capacity < 1 || !(r >= 0.0 && r <= 1.0) || *count < 0 || *count > capacity ||
      *head < 0 || *head >= capacity)
    return OR_ERR_INVALID_ARG;
  for (int64_t i = 0; i < n_cand; ++i)
    if (isnan(score[i])) return OR_ERR_NAN_INPUT;
  const int64_t n = *count;
  double kappa = INFINITY;
  if (n > 0 && n >= (int64_t)min_obs) {
    double* sorted = (double*)malloc(sizeof(double) * (size_t)n);
    /* the window's n most recent values are the n slots before head */
    for (int64_t t = 0; t < n; ++t) sorted[t] = window[(*head - n + t + capacity) % capacity];
    qsort(sorted, (size_t)n, sizeof(double), double_cmp);
    int64_t k = (int64_t)ceil((1.0 - r) * (double)n - 1e-9);
    if (k < 1) k = 1;
    if (k > n) k = n;
    kappa = sorted[k - 1];
    free(sorted);
  }
  int64_t retained = 0, drawn = 0;
  for (int64_t i = 0; i < n_cand; ++i) {
    if (batch_units > 0 && retained >= batch_units) {
      decision[i] = 2;
      continue;
    }
    drawn += 1;
    if (score[i] > kappa) decision[i] = 0;
    else {
      decision[i] = 1;
      retained += 1;
    }
  }
  for (int64_t i = 0; i < drawn; ++i) {
    window[*head] = score[i];
    *head = (*head + 1) % capacity;
    if (*count < capacity) *count += 1;
  }
  *kappa_out = kappa;
  return OR_OK;
}

/* Derivative of the surrogate loss of oracle_surrogate with respect to each
 * row's log-probability (the input the LM-head backward consumes):
 *   dL_t/dlp_t = -A rho_t   when the unclipped term is the active maximum
 *                           (p1 >= p2) and the dual clip is not active,
 *              = 0          when the clipped term or the dual clip (-c A < max,
 *                           A < 0) is active, or lp - l^mu is clamped (|.| >= 20),
 * then scaled by the aggregation: 1 / sum_t m_t (TOKEN_MEAN), or
 * 1 / (#sequences with tokens * #tokens of the row's sequence) (SEQ_MEAN).
 * Rows outside the loss get 0. */
int oracle_surrogate_grad(const double* logprob, const double* behav_lp, const uint8_t* mask,
                          const int64_t* seq_offsets, const uint8_t* seq_accepted, int64_t n_seq,
                          const double* adv, double eps_low, double eps_high, double dual_clip,
                          int32_t agg, double* dlp) {
  if (n_seq < 0) return OR_ERR_INVALID_ARG;
  if (agg != OR_AGG_TOKEN_MEAN && agg != OR_AGG_SEQ_MEAN_TOKEN_MEAN) return OR_ERR_INVALID_ARG;
  int st = check_offsets(seq_offsets, n_seq, -1);
  if (st) return st;
  double n_tok = 0.0;
  int64_t n_seq_used = 0;
  for (int64_t i = 0; i < n_seq; ++i) {
    const int seq_in = seq_accepted ? seq_accepted[i] != 0 : 1;
    int64_t c = 0;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1]; ++r)
      if (seq_in && (mask ? mask[r] != 0 : 1)) c += 1;
    n_tok += (double)c;
    if (c > 0) n_seq_used += 1;
  }
  for (int64_t i = 0; i < n_seq; ++i) {
    const int seq_in = seq_accepted ? seq_accepted[i] != 0 : 1;
    const double a = adv[i];
    int64_t c = 0;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1]; ++r)
      if (seq_in && (mask ? mask[r] != 0 : 1)) c += 1;
    for (int64_t r = seq_offsets[i]; r < seq_offsets[i + 1]; ++r) {
      const int in = seq_in && (mask ? mask[r] != 0 : 1);
      if (!in) {
        dlp[r] = 0.0;
        continue;
      }
      const double d = logprob[r] - behav_lp[r];
      double dc = d;
      if (dc < -20.0) dc = -20.0;
      if (dc > 20.0) dc = 20.0;
      const double rho = exp(dc);
      double rc = rho;
      if (rc < 1.0 - eps_low) rc = 1.0 - eps_low;
      if (rc > 1.0 + eps_high) rc = 1.0 + eps_high;
      const double p1 = -a * rho;
      const double p2 = -a * rc;
      const double l = p1 > p2 ? p1 : p2;
      double g = 0.0;
      if (d > -20.0 && d < 20.0 && p1 >= p2) g = -a * rho;
      if (a < 0.0 && -dual_clip * a < l) g = 0.0;
      const double scale =
          agg == OR_AGG_TOKEN_MEAN ? 1.0 / n_tok : 1.0 / ((double)n_seq_used * (double)c);
      dlp[r] = g * scale;
    }
  }
  return OR_OK;
}

/* Backward of the per-row log-probability through the LM head (Sec. 2's
 * token factorisation): with p = softmax(z / tau), z_v = h . W_v and
 * g_r = dLoss/dlp_r,
 *   G_rv  = (g_r / tau) (1[v = y_r] - p_rv)
 *   dH_r  = sum_v G_rv W_v            (fp64, v ascending)
 *   dW_v  = sum_r G_rv h_r            (fp64, rows ascending)
 * Rows with g_r = 0 contribute nothing.  dW may be NULL (row gradients only).
 * Worker threads take contiguous row ranges; each keeps its own dW sum and the
 * sums are added in thread order. */
typedef struct {
  const uint16_t* hidden;
  const uint16_t* w;
  const int32_t* targets;
  const double* g;
  int64_t r_begin, r_end;
  int32_t H, V;
  double tau;
  double* dh;
  double* dw;  /* private [V][H] or NULL */
  int magnitude; /* 1: sum |G_rv| |W_vk| and |G_rv| |h_rk| instead (error scale) */
  int status;
} bw_job;

static void* bw_worker(void* arg) {
  bw_job* jb = (bw_job*)arg;
  const int32_t H = jb->H, V = jb->V;
  double* z = (double*)malloc(sizeof(double) * (size_t)V);
  double* h = (double*)malloc(sizeof(double) * (size_t)H);
  for (int64_t r = jb->r_begin; r < jb->r_end; ++r) {
    double* dhr = jb->dh + (size_t)r * (size_t)H;
    for (int32_t k = 0; k < H; ++k) dhr[k] = 0.0;
    const double gr = jb->g[r];
    if (gr == 0.0) continue;
    const int32_t y = jb->targets[r];
    if (y < 0 || y >= V) {
      jb->status = OR_ERR_INVALID_ARG;
      continue;
    }
    const uint16_t* hr = jb->hidden + (size_t)r * (size_t)H;
    for (int32_t k = 0; k < H; ++k) h[k] = bf16_to_double(hr[k]);
    for (int32_t v = 0; v < V; ++v) {
      const uint16_t* wv = jb->w + (size_t)v * (size_t)H;
      double acc = 0.0;
      for (int32_t k = 0; k < H; ++k) acc = acc + h[k] * bf16_to_double(wv[k]);
      z[v] = acc / jb->tau;
    }
    double m = -INFINITY;
    for (int32_t v = 0; v < V; ++v)
      if (z[v] > m) m = z[v];
    double s = 0.0;
    for (int32_t v = 0; v < V; ++v) s = s + exp(z[v] - m);
    const double lse = m + log(s);
    for (int32_t v = 0; v < V; ++v) {
      const double p = exp(z[v] - lse);
      const double G = (gr / jb->tau) * ((v == y ? 1.0 : 0.0) - p);
      const uint16_t* wv = jb->w + (size_t)v * (size_t)H;
      if (jb->magnitude) {
        const double Ga = fabs(G);
        for (int32_t k = 0; k < H; ++k) dhr[k] = dhr[k] + Ga * fabs(bf16_to_double(wv[k]));
        if (jb->dw) {
          double* dwv = jb->dw + (size_t)v * (size_t)H;
          for (int32_t k = 0; k < H; ++k) dwv[k] = dwv[k] + Ga * fabs(h[k]);
        }
        continue;
      }
      for (int32_t k = 0; k < H; ++k) dhr[k] = dhr[k] + G * bf16_to_double(wv[k]);
      if (jb->dw) {
        double* dwv = jb->dw + (size_t)v * (size_t)H;
        for (int32_t k = 0; k < H; ++k) dwv[k] = dwv[k] + G * h[k];
      }
    }
  }
  free(z);
  free(h);
  return NULL;
}

static int lmhead_backward_run(const uint16_t* hidden, const uint16_t* w_vocab,
                               const int32_t* targets, const double* g, int64_t n_rows,
                               int32_t H, int32_t V, double temperature, double* dh, double* dw,
                               int32_t n_threads, int magnitude) {
  if (n_rows < 0 || H < 1 || V < 1 || !(temperature > 0.0)) return OR_ERR_INVALID_ARG;
  if (n_threads < 1) n_threads = 1;
  if (n_threads > 64) n_threads = 64;
  if ((int64_t)n_threads > n_rows) n_threads = n_rows > 0 ? (int32_t)n_rows : 1;
  bw_job jobs[64];
  pthread_t th[64];
  const int64_t per = (n_rows + n_threads - 1) / n_threads;
  const size_t wsz = (size_t)V * (size_t)H;
  for (int32_t t = 0; t < n_threads; ++t) {
    bw_job* jb = &jobs[t];
    jb->hidden = hidden;
    jb->w = w_vocab;
    jb->targets = targets;
    jb->g = g;
    jb->r_begin = (int64_t)t * per < n_rows ? (int64_t)t * per : n_rows;
    jb->r_end = jb->r_begin + per < n_rows ? jb->r_begin + per : n_rows;
    jb->H = H;
    jb->V = V;
    jb->tau = temperature;
    jb->dh = dh;
    jb->dw = dw ? (double*)calloc(wsz, sizeof(double)) : NULL;
    jb->magnitude = magnitude;
    jb->status = OR_OK;
  }
  for (int32_t t = 1; t < n_threads; ++t) pthread_create(&th[t], NULL, bw_worker, &jobs[t]);
  bw_worker(&jobs[0]);
  for (int32_t t = 1; t < n_threads; ++t) pthread_join(th[t], NULL);
  int status = OR_OK;
  if (dw) {
    for (size_t i = 0; i < wsz; ++i) dw[i] = 0.0;
    for (int32_t t = 0; t < n_threads; ++t) {
      for (size_t i = 0; i < wsz; ++i) dw[i] = dw[i] + jobs[t].dw[i];
      free(jobs[t].dw);
    }
  }
  for (int32_t t = 0; t < n_threads; ++t)
    if (jobs[t].status) status = jobs[t].status;
  return status;
}

int oracle_lmhead_backward(const uint16_t* hidden, const uint16_t* w_vocab,
                           const int32_t* targets, const double* g, int64_t n_rows, int32_t H,
                           int32_t V, double temperature, double* dh, double* dw,
                           int32_t n_threads) {
  return lmhead_backward_run(hidden, w_vocab, targets, g, n_rows, H, V, temperature, dh, dw,
                             n_threads, 0);
}

/* Error scale of the backward above (a test aid, not part of the method): the
 * same sums with every term replaced by its magnitude,
 *   mh_rk = sum_v |G_rv| |W_vk|,     mw_vk = sum_r |G_rv| |h_rk|.
 * A relative error of at most e in each G_rv (for instance from holding G in a
 * narrower format) moves dH_rk by at most e * mh_rk and dW_vk by at most
 * e * mw_vk, so these give element-wise tolerances. */
int oracle_lmhead_backward_magnitude(const uint16_t* hidden, const uint16_t* w_vocab,
                                     const int32_t* targets, const double* g, int64_t n_rows,
                                     int32_t H, int32_t V, double temperature, double* mh,
                                     double* mw, int32_t n_threads) {
  return lmhead_backward_run(hidden, w_vocab, targets, g, n_rows, H, V, temperature, mh, mw,
                             n_threads, 1);
}
