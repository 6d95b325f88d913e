"""lbm_batch_step returns before its work is done: nothing that the work reads
may go back to the caller's allocator before the handle is destroyed."""
import numpy as np
import pytest

from lbm_workloads import fields
from lbm_workloads.mechanism import h2_air_synthetic
from paper_2108_07605_gb300 import lbm

pytestmark = pytest.mark.gpu


class _Allocator:
    """Caller's allocation hooks that record what is given back."""

    def __init__(self):
        import torch
        self.live, self.freed = {}, []

        def alloc(nbytes, user):
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        def free(ptr, user):
            self.freed.append(ptr)      # (kept alive in self.live)

        self.alloc, self.free = lbm.ALLOC_FN(alloc), lbm.FREE_FN(free)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batch_step_frees_nothing(precision):
    mech = h2_air_synthetic()
    hooks, handles, ref, keep = _Allocator(), [], [], []
    for k in range(2):
        w = fields.perturbed_box((8, 6, 5), "D3Q27", seed=k, mech=mech)
        kw = dict(lattice=w["lattice"], shape=w["shape"], dx=w["dx"], precision=precision)
        args = [np.ascontiguousarray(w[n]).reshape(-1) for n in ("P", "u", "T", "Y")]
        cfg, kept = lbm.make_config(mech, use_torch_allocator=False, **kw)
        cfg.dev_alloc, cfg.dev_free = hooks.alloc, hooks.free
        keep.append((cfg, kept))
        handles.append(lbm.lbm_create(cfg))
        lbm.lbm_init_fields_pressure(handles[-1], *args)
        ref.append(lbm.Solver(mech, **kw))
        ref[-1].init_fields_pressure(w["P"], w["u"], w["T"], w["Y"])
    before = len(hooks.freed)
    lbm.lbm_batch_step(handles[:1], 2)
    lbm.lbm_batch_step(handles[:1], 1)
    assert len(hooks.freed) == before
    lbm.lbm_batch_step(handles, 4)              # a larger batch
    for h, r, n in zip(handles, ref, (7, 4)):
        r.step(n)
        want = r.populations()
        got = np.empty(want.size)
        lbm.lbm_get_populations(h, got)
        assert np.abs(got - want.reshape(-1)).max() <= 1e-6 * np.abs(want).max()
        lbm.lbm_destroy(h)
        r.close()
