"""Edges of the stacked products of H.psi (both precisions) and of the
Rayleigh-Ritz step, at the sizes where they can go wrong: sectors just below
and above a 64-row (FP64) or 128-row (split) tile and a 192-K drain chunk,
stacks of one block, K that is no multiple of 8, one and many term chunks,
K-split and whole tiles, odd chains and open shells, every slice count.
"""
import numpy as np
import pytest

import synth

from gpu_common import oracle_apply, oracle_problem, rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2309_16724_gb300 as P
    return P.Context(0, stream=torch.cuda.current_stream())


def run(ctx, env, psi, prec):
    import paper_2309_16724_gb300 as P
    x = torch.from_numpy(psi).cuda()
    y = torch.full_like(x, float("nan"))  # every element has to be written
    P.apply_heff(ctx, env, x, y, prec)
    assert ctx.status() == 0
    return y.cpu().numpy()


# (L, N, twoS, D): largest sectors of 19, 30, about 65, 75, 129, 175 and 261 rows
SIZES = [(10, 10, 0, 58), (13, 12, 0, 120), (16, 16, 0, 258), (11, 11, 1, 260), (16, 16, 0, 513), (14, 14, 0, 760),
         (15, 15, 1, 1030)]


@pytest.mark.parametrize("L,N,twoS,D", SIZES)
def test_split_and_fp64_agree_at_tile_edges(ctx, L, N, twoS, D):
    """The two paths share no kernel: their difference is the split error (bar
    1e-10), and cutting the terms into chunks moves neither."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("edge", synth.SPATIAL_ORBITAL, L, N, twoS, D, 17)
    sec, env = workload.build(ctx, cfg, prepare_split=True)
    psi = synth.gaussian_psi(sec.psi_len, 3)
    F = run(ctx, env, psi, P.SU2_FP64)
    G = run(ctx, env, psi, P.SU2_SPLIT_BF16)
    assert rel_err(G, F) <= 1e-10
    _, cut = workload.build(ctx, cfg, prepare_split=True, t_budget_bytes=max(1 << 16, int(env.info["t_chunk_bytes"]) // 7))
    assert cut.info["n_chunks"] > 1
    assert rel_err(run(ctx, cut, psi, P.SU2_FP64), F) <= 1e-13
    assert rel_err(run(ctx, cut, psi, P.SU2_SPLIT_BF16), F) <= 1e-10


@pytest.mark.parametrize("S,tol", [(2, 1e-3), (3, 1e-5), (4, 1e-7), (5, 1e-10), (6, 1e-11)])
def test_slice_counts_on_mixed_tiles(ctx, S, tol):
    """Every slice count (each has its own grouping of MMAs) on sectors of 1 to
    37 rows, against the oracle."""
    from paper_2309_16724_gb300 import workload
    import paper_2309_16724_gb300 as P
    cfg = synth.Config("mix", synth.SPATIAL_ORBITAL, 12, 11, 1, 150, 23)
    p = oracle_problem(cfg)
    psi = synth.gaussian_psi(p["n"], 8)
    F = oracle_apply(p, psi)
    _, env = workload.build(ctx, cfg, prepare_split=True, n_slices=S)
    assert rel_err(run(ctx, env, psi, P.SU2_SPLIT_BF16), F) <= tol
    assert rel_err(run(ctx, env, psi, P.SU2_FP64), F) <= 1e-12


@pytest.mark.parametrize("L,N,twoS,D", [(6, 6, 0, 3), (8, 7, 1, 20), (9, 9, 1, 33), (10, 10, 0, 58)])
def test_small_task_class_matches_oracle(ctx, L, N, twoS, D):
    """Environments of small tasks only (the first three) run in FP64 on either path."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("small", synth.SPATIAL_ORBITAL, L, N, twoS, D, 29)
    p = oracle_problem(cfg)
    psi = synth.gaussian_psi(p["n"], 2)
    F = oracle_apply(p, psi)
    _, env = workload.build(ctx, cfg, prepare_split=True)
    tol = 1e-12 if max(max(b.rows, b.cols) for b in p["blocks"]) <= 16 else 1e-10
    assert rel_err(run(ctx, env, psi, P.SU2_SPLIT_BF16), F) <= tol
    assert rel_err(run(ctx, env, psi, P.SU2_FP64), F) <= 1e-12


@pytest.mark.parametrize("max_sub,use_graph", [(3, False), (8, True), (17, False), (24, True), (32, False), (32, True)])
def test_rayleigh_ritz_at_every_subspace_size(ctx, max_sub, use_graph):
    """Odd and even subspaces up to the limit (32), eager and as a graph, reach
    the lowest eigenvalue of the dense H_eff (residual 1e-9: the eigenvalue is
    then good to 1e-12)."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("dav", synth.SPATIAL_ORBITAL, 7, 6, 0, 14, 31)
    p = oracle_problem(cfg)
    n = p["n"]
    H = np.stack([oracle_apply(p, e) for e in np.eye(n)], axis=1)
    _, env = workload.build(ctx, cfg)
    x = torch.from_numpy(synth.gaussian_psi(n, 5)).cuda()
    dav = P.Davidson(ctx, env, x, tol=1e-9, max_sub=max_sub, max_iter=2000, use_graph=use_graph)
    th, _, _, ok = dav.solve()
    assert ok and abs(th - np.linalg.eigvalsh(0.5 * (H + H.T))[0]) <= 1e-11
    v = torch.empty_like(x)
    dav.vector(v)
    v = v.cpu().numpy()
    assert np.linalg.norm(H @ v - th * v) <= 1e-8
    dav.close()
