"""What the out-of-core planner lets into a chunk, on the host.

The split path keeps a chunk's products as dense stacks: T' holds all left blocks
of an output sector (and its identity) times all output columns of that sector,
12 bytes an element (six slices), columns rounded up to 16; T holds all psi rows
of a right sector (each block's rounded up to 8) times the rows of all its right
blocks, 8 bytes an element.  Tasks with every dimension at most 16 take no part.
Restated here, a greedy cut of consecutive terms with these sizes gives the
fewest chunks that stay within the budget.
"""
import pytest

import synth

L_ = pytest.importorskip("paper_2309_16724_gb300._lib")

MB = 1 << 20


@pytest.fixture(scope="module")
def hctx():
    import paper_2309_16724_gb300 as P
    return P.Context(-1)


def needs(env, sec):
    """Per term: the left blocks (with their output sector) and the right blocks its larger tasks read."""
    rows, _ = env.tasks()
    ta, td, _, _ = env.terms()
    B = sec.blocks
    left, right = ([set() for _ in range(len(ta))] for _ in range(2))
    for f, term, e, ao, ai, bo, bi, flags in rows.tolist():
        if max(B[f][6], B[f][7], B[e][6], B[e][7]) <= 16:
            continue
        a = B[f][0]
        left[term].add((a, 0, a) if flags & 1 else (ao, int(ta[term]), ai))
        if not flags & 2:
            right[term].add((bi, int(td[term]), bo))
    return left, right


def dense_bytes(sec, left, right):
    B = sec.blocks
    cols, rows = {}, {}
    for b in B:
        cols[b[0]] = cols.get(b[0], 0) + b[7]
        rows[b[3]] = rows.get(b[3], 0) + (b[6] + 7) // 8 * 8
    total = 0
    for a, _, ai in left:
        total += 12 * ((cols[a] + 15) // 16 * 16) * ((sec.left[ai][2] + 7) // 8 * 8)
    for bi, _, bo in right:
        total += 8 * rows[bi] * sec.right[bo][2]
    return total


@pytest.mark.parametrize("L,D,model,budget", [(12, 300, "skeleton", 8 * MB), (12, 300, "skeleton", 16 * MB),
                                              (14, 500, "skeleton", 64 * MB), (12, 150, "ab_initio", 2 * MB)])
def test_dense_stacks_of_a_chunk_fit_the_budget(hctx, L, D, model, budget):
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("dense", synth.SPATIAL_ORBITAL, L, L, 0, D, 9)
    m = P.SU2_MODEL_AB_INITIO if model == "ab_initio" else P.SU2_MODEL_QC_SKELETON
    sec, env = workload.build(hctx, cfg, model=m, t_budget_bytes=budget, resident_bytes=1)
    left, right = needs(env, sec)
    least, hl, hr = 1, set(), set()
    for x, y in zip(left, right):
        if (hl or hr) and dense_bytes(sec, hl | x, hr | y) > budget:
            least, hl, hr = least + 1, set(), set()
        hl |= x
        hr |= y
    assert least > 2 and env.info["n_io_chunks"] >= least
