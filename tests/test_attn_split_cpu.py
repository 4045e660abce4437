"""The split of full attention's last round (csrc/attn_split.h), which two kernels work out separately:
the same S whatever the compiler's floating-point options, and the minimum of the stated cost with ties
to the smaller S (no GPU needed)."""
from fractions import Fraction

from host_build import host_lib

SOURCE = """
#include "attn_split.h"
extern "C" int best_split(int T, int P, int n_kv) {
  int best = 1;
  for (int S = 2; S <= vp::kMaxParts; ++S)
    if (vp::split_allowed(T, n_kv, S) && vp::split_cost(T, P, n_kv, S) < vp::split_cost(T, P, n_kv, best))
      best = S;
  return best;
}
extern "C" unsigned cost(int T, int P, int n_kv, int S) { return vp::split_cost(T, P, n_kv, S); }
"""


def stated_cost(T, P, n_kv, S):
    """Rounds of parts, in key tiles; below 41 key tiles in groups (3 % of a group per part)."""
    rounds = -(-T * S // P)
    if n_kv < 41:
        return Fraction(1) if S == 1 else rounds * (Fraction(1, S) + Fraction(3, 100))
    return rounds * (Fraction(n_kv, S) + 7) + (S if S > 1 else 0)


def test_split_is_the_minimum_of_its_cost(tmp_path):
    libs = []
    for i, flags in enumerate((("-O0", "-ffp-contract=off"), ("-O3", "-ffast-math"))):
        (tmp_path / str(i)).mkdir()
        libs.append(host_lib(tmp_path / str(i), SOURCE, flags))
    for P in (152, 148, 7):
        for T in sorted({t for t in (1, 2, 3, 8, 54, 87, 115, 130, P - 1) if t < P}):
            for n_kv in (1, 2, 17, 40, 41, 42, 172, 687, 2147, 500_000, 2 ** 25):
                allowed = [S for S in range(1, 65)
                           if S == 1 or (S <= n_kv and T * S <= (512 if n_kv < 41 else 682))]
                n = min(n_kv, 2 ** 19 - 1024)
                costs = {S: stated_cost(T, P, n, S) for S in allowed}
                got = [lib.best_split(T, P, n_kv) for lib in libs]
                assert got[0] == got[1] and got[0] in costs, (T, P, n_kv, got)
                # A cost rounds down by less than one unit a round, and no smaller S may cost less.
                slack = Fraction(64, 4096) if n_kv >= 41 else 0
                assert costs[got[0]] <= min(costs.values()) + slack, (T, P, n_kv, got)
                assert all(costs[S] > costs[got[0]] - slack for S in allowed if S < got[0]), (T, P, n_kv, got)
                for S in allowed:  # no overflow of 32 bits
                    unit = Fraction(1, 4096) if n_kv >= 41 else Fraction(1, 100 * 2 ** 16)
                    assert 0 <= costs[S] - libs[0].cost(T, P, n_kv, S) % 2 ** 32 * unit <= 64 * unit
