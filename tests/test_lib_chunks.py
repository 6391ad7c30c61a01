"""Term chunks against their byte budget, on the host.

The plan cuts the operator-table into runs of consecutive terms, as long as
their intermediates fit the budget.  Restated here from the environment's own
task table: a run is closed when the next term would not fit, and the term that
opens the next run counts with everything it needs there, also what it shared
with the closed run.  With the fewest bytes that the intermediates can take (each
(right block, psi block) product once, each (left block, output block) sum once),
this gives the fewest chunks the budget allows.
"""
import numpy as np
import pytest

import synth

L_ = pytest.importorskip("paper_2309_16724_gb300._lib")

KB = 1 << 10


@pytest.fixture(scope="module")
def hctx():
    import paper_2309_16724_gb300 as P
    return P.Context(-1)


def term_sets(env, sec):
    """Per term: {key: bytes} of its T blocks, its T' sums and its operator blocks."""
    rows, _ = env.tasks()
    ta, td, _, _ = env.terms()
    B = sec.blocks
    T, S, O = ([{} for _ in range(len(ta))] for _ in range(3))
    for f, term, e, ao, ai, bo, bi, flags in rows.tolist():
        if not flags & 2:
            T[term][(int(td[term]), bo, bi, e)] = (B[e][6] * sec.right[bo][2] + 1) // 2 * 2 * 8
            O[term][(1, int(td[term]), bo, bi)] = (sec.right[bo][2] * sec.right[bi][2] + 1) // 2 * 2 * 8
        left = (0, B[e][0]) if flags & 1 else (int(ta[term]), ao, ai)
        S[term][left, f] = 12 * B[e][6] * B[f][7]
        if not flags & 1:
            O[term][(0, int(ta[term]), ao, ai)] = (sec.left[ao][2] * sec.left[ai][2] + 1) // 2 * 2 * 8
    return T, S, O


def runs(n_terms, budget, measures):
    """Number of runs when every measure (a list of per-term {key: bytes} lists, weighted) of a run stays within the budget."""
    n, held = 1, [[{} for _ in m] for m in measures]

    def total(sets, ti):
        return [sum(w * sum({**h, **d[ti]}.values()) for h, (w, d) in zip(hs, m)) for hs, m in zip(sets, measures)]

    for ti in range(n_terms):
        if any(h for hs in held for h in hs) and max(total(held, ti)) > budget:
            n += 1
            held = [[{} for _ in m] for m in measures]
        for hs, m in zip(held, measures):
            for h, (_, d) in zip(hs, m):
                h.update(d[ti])
    return n


@pytest.mark.parametrize("L,D,model,budget_kb", [(10, 60, "ab_initio", 60), (12, 100, "skeleton", 120),
                                                 (12, 100, "skeleton", 700), (12, 300, "skeleton", 4000)])
def test_chunks_are_no_fewer_than_the_budget_allows(hctx, L, D, model, budget_kb):
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("chunks", synth.SPATIAL_ORBITAL, L, L, 0, D, 9)
    m = P.SU2_MODEL_AB_INITIO if model == "ab_initio" else P.SU2_MODEL_QC_SKELETON
    budget = budget_kb * KB
    sec, env = workload.build(hctx, cfg, model=m, t_budget_bytes=budget)
    T, S, O = term_sets(env, sec)
    least = runs(env.info["n_terms"], budget, [[(1, T)]])
    assert least > 2 and env.info["n_chunks"] >= least
    if max(sum(t.values()) for t in T) <= budget:
        assert env.info["t_chunk_bytes"] <= budget
    _, oc = workload.build(hctx, cfg, model=m, t_budget_bytes=budget, resident_bytes=1)
    least = runs(env.info["n_terms"], budget, [[(1, T), (1, S)], [(1, O)]])
    assert least > 2 and oc.info["n_io_chunks"] >= least
