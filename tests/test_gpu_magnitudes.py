"""The split path on operators of different magnitude.

H.psi is linear in the integrals, so neither a change of their unit nor a
constant on the diagonal of h may cost relative accuracy: the first makes the
complementary operators (which carry integrals) large beside the bare ones, the
second the block Hamiltonian beside the identity.  Neighbouring left blocks
share exponents in the split path, and which ones are neighbours depends on the
term chunks, hence the budgets: from one term a chunk to all in one.

Bound: five slices hold an operand to 2^-40 of its largest entry, 1e-12; the
same windows with integrals of order 1 and one exponent set per task give
1.3e-12 from K2 alone (the same slices in NumPy on these operators).  Four times
that for both products.
"""
import numpy as np
import pytest

import synth

from gpu_common import rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 5e-12


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2309_16724_gb300 as P
    return P.Context(0, stream=torch.cuda.current_stream())


@pytest.mark.parametrize("unit,shift", [(1.0, 0.0), (1.0, -10.0), (1.0, -50.0), (1e5, 0.0), (1e-4, 0.0)])
@pytest.mark.parametrize("resident", [0, 1])
def test_split_accuracy_does_not_depend_on_unit_or_shift(ctx, unit, shift, resident):
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("mag", synth.SPATIAL_ORBITAL, 10, 10, 0, 220, 1002)
    h, eri = synth.integrals(cfg.L, cfg.seed)
    h[np.diag_indices(cfg.L)] += shift
    kw = dict(model=P.SU2_MODEL_AB_INITIO, h=unit * h, eri=unit * eri, prepare_split=True, n_slices=5,
              resident_bytes=resident)
    F, worst = None, {}
    for budget in [0] + [3 << k for k in range(14, 24)]:
        sec, env = workload.build(ctx, cfg, t_budget_bytes=budget, **kw)
        x = torch.from_numpy(synth.gaussian_psi(sec.psi_len, 3)).cuda()
        y, z = torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
        P.apply_heff(ctx, env, x, y, P.SU2_SPLIT_BF16)
        if F is None:
            P.apply_heff(ctx, env, x, z, P.SU2_FP64)
            F = z.cpu().numpy()
        assert ctx.status() == 0
        worst[budget] = rel_err(y.cpu().numpy(), F)
        env.close()
    assert max(worst.values()) <= TOL, worst


def test_six_slices_lose_nothing_in_the_accumulator(ctx):
    """With six slices the rounding of a chunk's tail (2^-38 of the chunk) is
    what is left of the error; the tile accumulator must not add to it over the
    chunks of a long K axis.  The same slices and drain in NumPy give 1.01e-12
    for K2 and 0.81e-12 for K1, 1.29e-12 together; a pair that is normalised
    every fourth chunk 1.60e-12.  The bound is the geometric mean of the two."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("six", synth.SPATIAL_ORBITAL, 12, 12, 0, 300, 1002)
    sec, env = workload.build(ctx, cfg, model=P.SU2_MODEL_AB_INITIO, prepare_split=True, n_slices=6)
    x = torch.from_numpy(synth.gaussian_psi(sec.psi_len, 3)).cuda()
    y, z = torch.empty_like(x), torch.empty_like(x)
    P.apply_heff(ctx, env, x, y, P.SU2_SPLIT_BF16)
    P.apply_heff(ctx, env, x, z, P.SU2_FP64)
    assert ctx.status() == 0
    assert rel_err(y.cpu().numpy(), z.cpu().numpy()) <= 1.44e-12


@pytest.mark.parametrize("power", [-60, 60])
def test_split_is_homogeneous_in_psi(ctx, power):
    """A power of two on psi passes through every cut and scale exactly."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("pow", synth.SPATIAL_ORBITAL, 12, 11, 1, 150, 23)
    sec, env = workload.build(ctx, cfg, prepare_split=True)
    x = torch.from_numpy(synth.gaussian_psi(sec.psi_len, 3)).cuda()
    y, z = torch.empty_like(x), torch.empty_like(x)
    P.apply_heff(ctx, env, x, y, P.SU2_SPLIT_BF16)
    P.apply_heff(ctx, env, x * 2.0 ** power, z, P.SU2_SPLIT_BF16)
    assert torch.equal(z, y * 2.0 ** power)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_nan_or_infinity_in_psi_reaches_the_result(ctx, bad):
    """Where the FP64 path returns something that is not finite, so does the split path."""
    import paper_2309_16724_gb300 as P
    from paper_2309_16724_gb300 import workload
    cfg = synth.Config("nan", synth.SPATIAL_ORBITAL, 12, 11, 1, 150, 23)
    sec, env = workload.build(ctx, cfg, prepare_split=True)
    x = torch.from_numpy(synth.gaussian_psi(sec.psi_len, 3)).cuda()
    big = max(sec.blocks, key=lambda b: b[6] * b[7])
    x[big[8] + big[6] * (big[7] // 2) + big[6] // 3] = bad
    y, z = torch.empty_like(x), torch.empty_like(x)
    P.apply_heff(ctx, env, x, y, P.SU2_SPLIT_BF16)
    P.apply_heff(ctx, env, x, z, P.SU2_FP64)
    assert ctx.status() == 0
    lost = ~torch.isfinite(z)
    assert bool(lost.any()) and not bool(torch.isfinite(y[lost]).any())
