"""FP32 adjoint steps of fields whose rows are no 16-byte multiple: the saved states and the
gradients from the row-padded working copy against the same from the plain kernels
(BIOFVM_PITCHED=0).  Bound: both are FP32 solves of one step (1e-5 normwise each)."""
import numpy as np
import pytest

from paper_2602_05017_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("shape", [(37, 23, 19, 3), (5, 40, 33, 1), (101, 7, 50, 2)],
                         ids=lambda s: "x".join(map(str, s)))
def test_saved_states_and_gradients_match_plain_kernels(shape, dirichlet, monkeypatch):
    import torch
    from paper_2602_05017_gb300 import binding
    rng = np.random.default_rng(shape[0])
    w = inputs.random_problem(rng, *shape, n_agents=60, dirichlet=dirichlet)
    gout = torch.tensor(rng.normal(size=w.shape), dtype=torch.float32, device="cuda")
    results = []
    for pitched in ("1", "0"):
        monkeypatch.setenv("BIOFVM_PITCHED", pitched)
        sim = binding.BioFVM.from_workload(w, precision="fp32")
        saved = torch.empty(4 * sim.n_elem, dtype=torch.float32, device="cuda")
        sim.step_save(saved)
        g = torch.empty_like(gout)
        dD, dl = (torch.zeros(w.ns, dtype=torch.float64, device="cuda") for _ in range(2))
        ds, du = (torch.zeros(60 * w.ns, dtype=torch.float64, device="cuda") for _ in range(2))
        sim.adjoint_step(gout, g, dD, dl, ds, saved, dupt=du)
        sim.sync()
        results.append([saved, sim.field_tensor().clone(), g, dD, dl, ds, du])
        sim.close()
    for a, b in zip(*results):
        a, b = a.double(), b.double()
        assert (a - b).abs().max() <= 2e-5 * b.abs().max()
