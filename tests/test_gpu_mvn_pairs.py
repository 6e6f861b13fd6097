"""Sample counts around the rules that give each lane of the Monte Carlo kernel
two samples per turn (from 225, saddles from 513) and around those turns (64 a
warp): identical streams to the oracle's, hits equal up to its near ties."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ucp():
    from paper_2407_18015_gb300 import build
    build.build()
    from paper_2407_18015_gb300 import ucp as u
    return u


@pytest.mark.parametrize("S", [224, 225, 255, 256, 257, 287, 289, 512, 513, 543, 545,
                               576, 577])
@pytest.mark.parametrize("shape", [(5, 7), (1, 9)])
def test_sample_counts(ucp, orc, S, shape):
    from paper_2407_18015_gb300 import synth
    ens = synth.ensemble_iid(*shape, 12, seed=S)
    ctx = ucp.Context(0)
    desc = ucp.make_desc("mvn", mc_samples=S, seed=0xABCDEF0123, field_id=9)
    params = ctx.fit(torch.from_numpy(ens).cuda(), desc)
    pmin, pmax, _ = ctx.probability_from_params(params, desc)
    sad, _ = ctx.saddle_from_params(params, desc)
    torch.cuda.synchronize()
    idx = np.arange(shape[0] * shape[1])
    hmin, hmax, ties, _, hsad = orc.mvn_mc_at(params.double().cpu().numpy(), idx, S, 0xABCDEF0123,
                                              field=9, with_saddle=True)
    for g, h in ((pmin, hmin), (pmax, hmax), (sad, hsad)):
        assert (np.abs(g.cpu().numpy().ravel() * S - h) <= ties + 1e-3).all()
