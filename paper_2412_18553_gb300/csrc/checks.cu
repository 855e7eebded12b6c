// Device-side checks of the input values, launched at the head of every call
// on the caller's stream (no host synchronisation):
//  * every entry of the seven arrays is finite;
//  * max(eps_o) < min(eps_v), so that every denominator D of Eq. D is
//    negative (the orbital energies need not be sorted).
// A violation sets ERR_BAD_INPUT in the handle's error word with the site
// (1..7: the array, in the order eps_o, eps_v, ovvv, ooov, ovov, t1, t2;
// 8: the ordering of the orbital energies; 9, 10: the density-fitting
// factors Bov, Bvv) and the cluster index; te_sync
// reports it as TE_EINVAL.  The kernels that follow still run (they never
// fault on such values); their results are then unspecified.
//
// The pass is the one that finds the largest magnitudes the exact-slice modes
// scale by (k_absmax, prep_tc.cu): an entry is not finite exactly when its
// high word, sign taken off, reaches 0x7FF00000, and the integer maximum of
// those words carries both answers, so the inputs are read once for the two.
#include "prep_tc.h"

namespace te {

cudaError_t launch_check_inputs(const te_cluster* c, int64_t cluster, unsigned int* err, int num_sms,
                                cudaStream_t s, const te_df* df, const MaxOut* out) {
  const int64_t o = c->nocc, v = c->nvir, P = df ? df->naux : 0;
  const MaxOut none{};
  const MaxOut& m = out ? *out : none;
  const bool grp = m.groups;
  // with density-fitting factors, ovvv is not read: Bov and Bvv instead
  const MaxArray all[MAX_ARRAYS] = {
      {c->ovvv, df ? 0 : (grp ? o : 1), grp ? v * v * v : o * v * v * v, grp ? -1 : 0, m.ovvv, nullptr, 0, 3u},
      {c->t2, grp ? o * o : 1, grp ? v * v : o * o * v * v, grp ? -1 : 0, m.t2, m.t2L, grp ? (int)o : 0, 7u},
      {c->ooov, grp ? o * o * o : 1, grp ? v : o * o * o * v, grp ? (int)o : 0, m.ooov, nullptr, 0, 4u},
      {df ? df->Bov : nullptr, df ? 1 : 0, P * o * v, 0, m.bov, nullptr, 0, 9u},
      {df ? df->Bvv : nullptr, df ? 1 : 0, P * v * v, 0, m.bvv, nullptr, 0, 10u},
      {c->ovov, 1, o * v * o * v, 0, nullptr, nullptr, 0, 5u},
      {c->t1, 1, o * v, 0, nullptr, nullptr, 0, 6u},
      {c->eps_o, 1, o, 0, nullptr, nullptr, 0, 1u},
      {c->eps_v, 1, v, 0, nullptr, nullptr, 0, 2u}};
  MaxArray a[MAX_ARRAYS];
  int n = 0;
  for (const MaxArray& x : all) {
    if (!err && !x.out) continue;  // largest magnitudes only
    a[n] = x;
    if (!err) a[n].site = 0;
    ++n;
  }
  return launch_absmax(a, n, err ? c->eps_o : nullptr, (int)o, c->eps_v, (int)v, (unsigned int)cluster, err, num_sms,
                       s);
}

// The MP2 step's inputs: eps_o (site 1), eps_v (site 2), the DF factor's ov
// block (site 9), and the eps ordering (site 8).
cudaError_t launch_check_mp2(const double* eps_o, int64_t o, const double* eps_v, int64_t v, const double* Bov,
                             int64_t nB, int64_t cluster, unsigned int* err, int num_sms, cudaStream_t s,
                             unsigned int* max_bov) {
  const MaxArray a[3] = {{Bov, 1, nB, 0, max_bov, nullptr, 0, 9u},
                         {eps_o, 1, o, 0, nullptr, nullptr, 0, 1u},
                         {eps_v, 1, v, 0, nullptr, nullptr, 0, 2u}};
  return launch_absmax(a, 3, eps_o, (int)o, eps_v, (int)v, (unsigned int)cluster, err, num_sms, s);
}

}  // namespace te
