"""M, M^dagger and M M^dagger on a field passed with the call: the kernels form
the phases themselves, or build only the table they read, and give bit for bit
what they give on the loaded field's tables; also where out lies on the field."""
import pytest

import workloads as W

from gpu_util import ctx_for, dev, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ms", [0.0, 0.3])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("shape", [(1, 2, 3), (6, 6, 16), (25, 3, 17), (51, 51, 64)])
def test_call_field_equals_loaded_field(shape, prec, ms):
    need_gpu()
    w = W.small(*shape, seed=2300 + sum(shape))
    dt = torch.complex128 if prec == 64 else torch.complex64
    b = dev(w.b).to(dt)
    phi = dev(w.phi)
    with ctx_for(w.lat) as ctx:
        for variant in (0, 1, 2):
            ctx.set_apply_variant(variant)
            calls = [lambda f, o: ctx.apply_M(f, ms, b, out=o), lambda f, o: ctx.apply_Mdag(f, ms, b, out=o),
                     lambda f, o: ctx.apply_MMdag(f, ms, b, sigma=0.2, out=o)]
            for call in calls:
                ctx.load_field(phi)
                ref = call(None, torch.empty_like(b)).clone()
                assert torch.equal(call(phi, torch.empty_like(b)), ref)
                if prec == 64:  # out on top of the field: read before it is written
                    out = torch.empty_like(b)
                    f = out.view(torch.float64)[: w.lat.nsites]
                    f.copy_(phi)
                    assert torch.equal(call(f, out), ref)
        assert ctx.check_guards() == 0
