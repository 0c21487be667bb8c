"""The ADMM graphs a handle keeps: what is changed on the handle between calls reaches the next one."""

import numpy as np
import pytest

from gpu_common import CASES, device_kernel
from paper_2101_11680_gb300 import ctof

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def measurement(name, seed=1):
    kw = CASES[name]
    rng = np.random.default_rng(seed)
    return torch.tensor(rng.uniform(0.0, 1.0, (kw["nt"], kw["n"], kw["n"])), dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("batched", [False, True])
def test_wait_limit_takes_effect_after_the_first_call(batched):
    k, m, prm = device_kernel("admm16"), measurement("admm16"), ctof.admm_params(4)
    solve = lambda: ctof.reconstruct_batch([k], [m], prm)[0] if batched else k.reconstruct(m, prm)
    want = solve()
    k.sync_status()
    try:
        k.set_wait_limit(0)
        solve()
        with pytest.raises(ctof.CtofError) as e:
            k.sync_status()
        assert e.value.status == ctof.ETIMEOUT
    finally:
        k.set_wait_limit(1 << 24)
    assert torch.equal(solve(), want)
    k.sync_status()
