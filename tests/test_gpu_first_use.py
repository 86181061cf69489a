"""The first call that launches work with a code copies its tables to the
device. That call may come on any stream, also on one that does not wait for
the legacy stream, and the tables' place may have belonged to another code."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_parity import dev, packed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


def test_first_use_on_a_non_blocking_stream_reads_its_own_tables():
    """Codes of different sizes come and go, each first used by a syndrome on
    a side stream: every one has the oracle's syndrome."""
    side = torch.cuda.Stream()
    makers = (synth.rate010_code, synth.rate002_code, synth.rate005_code)
    for rep in range(30):
        d = makers[rep % 3]((64, 37, 512, 9)[rep % 4])
        ocode = oracle.Code.from_dict(d)
        bits = np.random.default_rng(rep).integers(0, 2, (1, ocode.n)).astype(np.uint8)
        bits_dev = dev(packed(bits).view(np.int32).reshape(-1))
        syn = torch.zeros((ocode.m + 31) // 32, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        code = q.create_code_from(d)
        q.qcldpc_syndrome(code, bits_dev, syn, 1, side)
        torch.cuda.synchronize()
        got = synth.unpack_bits(syn.cpu().numpy().view(np.uint32), ocode.m)
        np.testing.assert_array_equal(got, oracle.syndrome(ocode, bits[0]))
        q.qcldpc_destroy_code(code)
