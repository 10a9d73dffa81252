"""GPU parity of the chunked kernel with 16-token chunks and two blocks per SM, which launches with more than 1.7 tiles per SM
take at Dk = 64, against the fp64 CPU oracle: partial chunks, one chunk alone, a partial column slice, and sequences cut
between blocks."""
import pytest
import torch

from paper_2609_39034_b200 import workloads as wl
from tests._gpu_util import assert_close, gpu_forward, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    from paper_2609_39034_b200 import binding as b

    return b


def _w(H, T, J=4, Dv=64):
    return wl.Workload(f"h{H}_t{T}_j{J}_v{Dv}", 1, B=1, H=H, T=T, Dk=64, Dv=Dv, J=J, io_dtype="bf16")


@pytest.mark.parametrize("w0,var", [
    (_w(130, 16), dict()), (_w(130, 47), dict()), (_w(90, 99, Dv=72), dict()), (_w(70, 70, J=8), dict()), (_w(40, 66, J=16), dict()),
    (_w(160, 290), dict()), (_w(130, 83), dict(gated=True, granularity=wl.GRAN_PER_OUT)),
    (_w(160, 290), dict(gated=True, granularity=wl.GRAN_SCALAR, post_decay=True))], ids=lambda x: x.name if isinstance(x, wl.Workload) else "+".join(x) or "plain")
def test_two_blocks_per_sm_match_oracle(binding, oracle, w0, var):
    w = w0.variant(**var)
    inp = wl.make_inputs(w, stress=True)
    ref = oracle.forward_inputs(inp, flags=w.flags, gran=w.gate_granularity)
    dev = to_dev(inp)
    got = gpu_forward(binding, w, dev, algo=binding.ALGO_CHUNK)
    binding.device_status()
    assert_close(w, got, ref, w.name)
    if not w.gated and w.J <= 8:  # the auxiliary instantiation: same outputs, and r
        aux = gpu_forward(binding, w, dev, algo=binding.ALGO_CHUNK, want_r=True)
        binding.device_status()
        assert torch.equal(aux["o"], got["o"]) and torch.equal(aux["W"], got["W"])
        assert_close(w, aux, oracle.forward_inputs(inp, want_r=True), w.name)
