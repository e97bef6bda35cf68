"""The Legendre sums beside kept maps: what else runs on the plan leaves them, or they are formed again, so that the
ring-mode linear term of a retained call equals that of modal_cubic bit for bit."""
import numpy as np
import pytest
import torch

import simgen

pytestmark = pytest.mark.gpu

L, P, R, NPHI, NB = 24, 6, 25, 64, 3


def _setup(prec, tmp_path):
    """A plan in ring mode, its state and a pixel-mode state on files, three maps and their coefficients in ring mode."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1105_2791_gb300 as M
    basis, cl = simgen.shifted_legendre_basis(L, P), simgen.cl_model(L)
    make = lambda: M.Plan(L, P, basis, cl, R, NPHI, prec=prec, ring_mask=simgen.band_mask(R, 20.0))
    sims = torch.from_numpy(simgen.gaussian_alm(cl, 6, seed=81).astype(np.complex64)).cuda()
    a = torch.from_numpy(simgen.gaussian_alm(cl, NB, seed=82).astype(np.complex64)).cuda()
    plan, files = make(), {}
    for mode in ("pixel", "ring"):
        plan.set_linear_mode(mode)
        plan.linear_term(sims, finalize=True)
        files[mode] = str(tmp_path / mode)
        plan.save_state(files[mode])
    ref = plan.cubic(a, use_linear=True)
    plan.close()
    return make(), files, sims, a, ref


@pytest.mark.parametrize("prec", ["fp32", "fp16x3", "3xtf32"])
@pytest.mark.parametrize("table", ["own means", "means of earlier maps", "loaded state"])
def test_pair_mean_table_leaves_the_kept_sums(prec, table, tmp_path):
    """The per-pixel means' harmonic table, however it comes to be built after the maps were kept."""
    plan, files, sims, a, ref = _setup(prec, tmp_path)
    plan.set_retain_maps(True)
    if table == "own means":
        plan.linear_term(a, finalize=True)
    elif table == "means of earlier maps":
        plan.linear_term(sims)
        plan.cubic(a)
        plan.linear_term(None, finalize=True)
    else:
        plan.cubic(a)
        plan.load_state(files["pixel"])
    plan.set_linear_mode("ring")
    plan.load_state(files["ring"])
    assert torch.equal(plan.cubic_retained(a, use_linear=True), ref)
    plan.sync()
    plan.close()


@pytest.mark.parametrize("prec", ["fp32", "fp16x3"])
@pytest.mark.parametrize("others", [1, NB, 7])
def test_synthesis_of_other_maps_between(prec, others, tmp_path):
    """modal_synthesize writes the caller's maps and leaves the kept ones, but goes through the Legendre sums."""
    plan, files, sims, a, ref = _setup(prec, tmp_path)
    plan.set_retain_maps(True)
    b = torch.from_numpy(simgen.gaussian_alm(simgen.cl_model(L), others, seed=5).astype(np.complex64)).cuda()
    plan.load_state(files["pixel"])
    plan.cubic(a)
    maps = plan.synthesize(b)
    plan.cubic_retained(a, use_linear=True)                # per pixel: needs the maps alone
    plan.set_linear_mode("ring")
    plan.load_state(files["ring"])
    for _ in range(2):
        assert torch.equal(plan.cubic_retained(a, use_linear=True), ref)
    assert torch.equal(plan.synthesize(b), maps)
    plan.sync()
    plan.close()


@pytest.mark.parametrize("schedule", ["streams", "shared_cubic"])
def test_replayed_batch_replaces_the_kept_maps(schedule, tmp_path):
    """A replay of a batch's graph writes its members' maps like the call that captured it: what another call kept before
    is gone, what the batch synthesised is kept."""
    plan, files, sims, a, ref = _setup("fp16x3", tmp_path)
    import paper_1105_2791_gb300 as M
    other = M.Plan(16, P, simgen.shifted_legendre_basis(16, P), simgen.cl_model(16), 17, NPHI)
    c = torch.from_numpy(simgen.gaussian_alm(simgen.cl_model(16), 2, seed=6).astype(np.complex64)).cuda()
    for p in (plan, other):
        p.set_retain_maps(True)
    batch = M.Batch([plan, other], schedule=schedule)
    alms = [sims, c]
    want = [b.clone() for b in batch.cubic(alms)]
    assert torch.equal(plan.cubic_retained(sims), want[0])
    plan.cubic(a)
    for b, w in zip(batch.cubic(alms), want):              # the captured graph again
        assert torch.equal(b, w)
    with pytest.raises(M.ModalError) as e:
        plan.cubic_retained(a)
    assert e.value.status == M.MODAL_ESTATE
    assert torch.equal(plan.cubic_retained(sims), want[0]) and torch.equal(other.cubic_retained(c), want[1])
    plan.sync()
    batch.close()
    plan.close()
    other.close()
