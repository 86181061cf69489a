"""Syndromes of codes with short rows: one thread per check or per word of 32
checks, chosen by row length, row weight and the number of checks."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402
from test_gpu_parity import gpu_syndrome  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


def short_rows(mb, Z, deg):
    """mb rows of deg heavy circulants in distinct ones of 16 columns and a
    degree-1 circulant each."""
    rng = np.random.default_rng(Z * deg)
    heavy = np.stack([rng.choice(16, deg, replace=False) for _ in range(mb)])
    row = np.repeat(np.arange(mb), deg + 1)
    col = np.concatenate([heavy, 16 + np.arange(mb)[:, None]], 1).reshape(-1)
    return dict(mb=mb, nb=16 + mb, Z=Z, row=row, col=col, shift=rng.integers(0, Z, row.size))


@pytest.mark.parametrize("deg", [2, 6])
@pytest.mark.parametrize("Z", [1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 15, 16, 17, 20, 24, 31, 33])
def test_short_rows_match_the_oracle(Z, deg):
    d = short_rows(67, Z, deg)
    code = oracle.Code.from_dict(d)
    bits = np.random.default_rng(Z).integers(0, 2, (3, code.n)).astype(np.uint8)
    got = gpu_syndrome(q.create_code_from(d), bits)
    np.testing.assert_array_equal(got, np.stack([oracle.syndrome(code, b) for b in bits]))


@pytest.mark.parametrize("maker, Z", [(synth.rate002_code, 8), (synth.met_code, 9), (synth.rate010_code, 7)])
def test_frame_counts_on_both_sides_of_a_million_checks(maker, Z):
    """The frames of a call above 2^20 checks have the syndromes that calls
    below give them."""
    code = q.create_code_from(maker(Z))
    wn, wm = (code.n + 31) // 32, (code.m + 31) // 32
    F = (1 << 20) // code.m + 2
    g = torch.Generator(device="cuda")
    g.manual_seed(Z)
    bits = torch.randint(-2 ** 31, 2 ** 31, (F * wn,), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    many, few = (torch.full((F * wm,), 7, dtype=torch.int32, device="cuda") for _ in range(2))
    q.qcldpc_syndrome(code, bits, many, F)
    half = F // 2
    q.qcldpc_syndrome(code, bits[:half * wn], few[:half * wm], half)
    q.qcldpc_syndrome(code, bits[half * wn:], few[half * wm:], F - half)
    torch.cuda.synchronize()
    assert torch.equal(many, few)
