"""Layered decoding: row groups whose check pass updates the posteriors itself
give the bits of the check pass followed by the posterior pass."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from bench import layered_launches

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import build  # noqa: E402
from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402
from test_gpu_kernel_edges import odd_code  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


def with_unfused_rows(d):
    """d's rows, each followed by a row on columns of its own that meets one of
    them twice: a group of the two rows cannot update the posteriors in its
    check pass, and d's part of the decode is untouched by the other rows."""
    mb, nb, Z = d["mb"], d["nb"], d["Z"]
    own = np.arange(mb)
    row = np.concatenate([2 * d["row"]] + [2 * own + 1] * 3)
    col = np.concatenate([d["col"], np.full(2 * mb, nb), nb + 1 + own])
    shift = np.concatenate([d["shift"], np.zeros(mb, int), np.full(mb, Z // 2), np.zeros(mb, int)])
    return dict(mb=2 * mb, nb=nb + 1 + mb, Z=Z, row=row.astype(np.int32), col=col.astype(np.int32),
                shift=shift.astype(np.int32))


def decode(d, llr, syn, iters, soft, **params):
    F = llr.shape[0]
    code = q.create_code_from(d)
    p = q.qcldpc_params_init(schedule=1, et_start=iters + 1, **params)
    dec = q.Decoder(code, F, p, soft=soft)
    dec.decode(torch.from_numpy(llr.reshape(-1)).cuda(),
               torch.from_numpy(synth.pack_bits(syn).view(np.int32).reshape(-1)).cuda(), iters)
    torch.cuda.synchronize()
    return (dec.keys.cpu().numpy().reshape(F, -1),
            dec.posterior.cpu().numpy().reshape(F, -1) if soft else None)


@pytest.mark.parametrize("fmt, step", [(0, 0.0), (1, 0.0), (2, 0.0), (2, 0.011), (2, 0.37)])
@pytest.mark.parametrize("maker, Z", [(odd_code, 5), (synth.rate002_code, 33), (synth.rate002_code, 257),
                                      (synth.rate002_code, 1025)])
def test_fused_groups_have_the_bits_of_the_separate_update(maker, Z, fmt, step):
    """The quantum 0.011 saturates most int8 codes, 0.37 leaves few levels."""
    d = maker(Z)
    both = with_unfused_rows(d)
    mb, n, F = d["mb"], d["nb"] * Z, 2
    assert layered_launches(d, mb) < 2 + 2 * mb and layered_launches(both, mb) == 2 + 2 * mb
    rng = np.random.default_rng(Z + fmt)
    llr = rng.normal(0.3, 1.0, (F, both["nb"] * Z)).astype(np.float32)
    syn = rng.integers(0, 2, (F, 2 * mb * Z)).astype(np.uint8)
    own = np.ascontiguousarray(syn.reshape(F, mb, 2, Z)[:, :, 0].reshape(F, -1))
    for iters in (1, 2, 5):
        keys, post = decode(d, llr[:, :n].copy(), own, iters, True, msg_format=fmt, msg_step=step)
        _, ref = decode(both, llr, syn, iters, True, msg_format=fmt, msg_step=step, layers=mb)
        np.testing.assert_array_equal(post.view(np.int32), ref[:, :n].copy().view(np.int32))
        hard, _ = decode(d, llr[:, :n].copy(), own, iters, False, msg_format=fmt, msg_step=step)
        np.testing.assert_array_equal(hard, keys)


def test_checks_evaluated_one_at_a_time_update_the_posteriors_too(tmp_path):
    """A build without packed pairs (an option of tuning builds) takes the
    scalar form of the check pass; its fused groups match the oracle."""
    lib = build.build(extra_flags=["-DQCLDPC_CN_PAIR=0"], out_dir=str(tmp_path))
    tests = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-m", "gpu", "-p", "no:cacheprovider",
                        os.path.join(tests, "test_gpu_kernel_edges.py"), os.path.abspath(__file__),
                        "-k", "one_row_groups or separate_update"],
                       env=dict(os.environ, QCLDPC_LIB=lib), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:]
