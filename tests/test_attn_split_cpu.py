"""The split of full attention's last round (csrc/attn_split.h), which two kernels work out separately: the
same S whatever the compiler's floating-point options, the minimum of the stated cost with ties to the
smaller S, and never fewer parts than the share rule's, which would round more large weights (no GPU needed)."""
from fractions import Fraction

from host_build import host_lib

SOURCE = """
#include "attn_split.h"
using namespace vp;
extern "C" int least_split(int T, int P, int n_kv) {
  int best = 1;
  for (int S = 2; S <= kMaxParts; ++S)
    if (share_cost(T, P, n_kv, S) < share_cost(T, P, n_kv, best)) best = S;
  return best;
}
extern "C" int best_split(int T, int P, int n_kv) {
  const int least = least_split(T, P, n_kv);
  int best = least;
  for (int S = 1; S <= kMaxParts; ++S)
    if (split_cost(T, P, n_kv, S, least) < split_cost(T, P, n_kv, best, least)) best = S;
  return best;
}
extern "C" unsigned cost(int T, int P, int n_kv, int S) { return split_cost(T, P, n_kv, S, 1); }
"""


def share_rule(T, P, n_kv):
    """The cheapest S at 3 % of a group per part."""
    costs = {1: Fraction(1)}
    for S in range(2, 65):
        if S <= n_kv and T * S <= 512:
            costs[S] = -(-T * S // P) * (Fraction(1, S) + Fraction(3, 100))
    return min(costs, key=lambda S: (costs[S], S))


def stated_cost(T, P, n_kv, S):
    """The last round in key tiles."""
    return -(-T * S // P) * (Fraction(n_kv, S) + 7) + (S if S > 1 else 0)


def test_split_is_the_minimum_of_its_cost(tmp_path):
    libs = []
    for i, flags in enumerate((("-O0", "-ffp-contract=off"), ("-O3", "-ffast-math"))):
        (tmp_path / str(i)).mkdir()
        libs.append(host_lib(tmp_path / str(i), SOURCE, flags))
    for P in (152, 148, 7):
        for T in sorted({t for t in (1, 2, 3, 7, 8, 54, 87, 115, 130, P - 1) if t < P}):
            for n_kv in (1, 2, 17, 40, 41, 42, 77, 172, 687, 2147, 500_000, 2 ** 25):
                least = share_rule(T, P, n_kv)
                got = [lib.best_split(T, P, n_kv) for lib in libs]
                assert got[0] == got[1], (T, P, n_kv, got)
                assert [lib.least_split(T, P, n_kv) for lib in libs] == [least, least], (T, P, n_kv)
                allowed = [S for S in range(least, 65) if S == 1 or (S <= n_kv and T * S <= 682)]
                n = min(n_kv, 2 ** 19 - 1024)
                costs = {S: stated_cost(T, P, n, S) for S in allowed}
                # A cost rounds down by less than one unit a round, and no smaller S may cost less.
                slack = Fraction(64, 4096)
                assert costs[got[0]] <= min(costs.values()) + slack, (T, P, n_kv, got)
                assert all(costs[S] > costs[got[0]] - slack for S in allowed if S < got[0]), (T, P, n_kv, got)
                for S in allowed:  # no overflow of 32 bits
                    assert 0 <= costs[S] - Fraction(libs[0].cost(T, P, n_kv, S) % 2 ** 32, 4096) <= slack


def test_no_fewer_parts_than_the_share_rule(tmp_path):
    lib = host_lib(tmp_path, SOURCE)
    for T in (1, 3, 7, 8, 12, 13, 41, 54, 115):
        for n_kv in [*range(1, 61, 4), *range(61, 400, 9)]:
            got, least = lib.best_split(T, 152, n_kv), share_rule(T, 152, n_kv)
            assert got == least if n_kv <= 60 else got >= least, (T, n_kv)
