"""Kernel forms chosen by size, alignment or option, at the edges of their tiles.

Each form is compared with the oracle or with the other form that computes
the same bits: word-wise syndromes (rows that end inside a word, windows that
wrap), the vector form of the d-dimensional maps (unaligned buffers, tails),
the check pass that loads its operands directly against the staged one, and
row groups whose check pass updates the posteriors itself.
"""
import numpy as np
import pytest

import oracle
import synth
from frames import make_frames

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402
from test_gpu_parity import (U32, assert_posteriors_close, decode_soft, dev, gpu_syndrome,  # noqa: E402
                             odd_code, packed)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


@pytest.mark.parametrize("Z", [2, 3, 15, 31, 32, 33, 63, 64, 65, 127, 1000])
def test_syndrome_words_across_rows_and_wraps(Z):
    d = odd_code(Z) if Z < 64 else synth.rate002_code(Z)
    code = oracle.Code.from_dict(d)
    bits = np.random.default_rng(Z).integers(0, 2, (3, code.n)).astype(np.uint8)
    got = gpu_syndrome(q.create_code_from(d), bits)
    np.testing.assert_array_equal(got, np.stack([oracle.syndrome(code, b) for b in bits]))


@pytest.mark.parametrize("offset", [0, 1, 4])
@pytest.mark.parametrize("d, n", [(1, 1), (1, 7), (1, 1030), (2, 2), (2, 6), (2, 1030), (4, 4), (4, 1028)])
def test_maps_of_any_alignment_and_tail(d, n, offset):
    """Buffers `offset` floats past a 16-byte boundary; the bounds are those of
    the dimension test (a block product of d terms in FP32). The words after
    the outputs stay untouched."""
    rng = np.random.default_rng(10 * n + d)
    x, y = rng.standard_normal(n).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    bits = rng.integers(0, 2, n).astype(np.uint8)
    snr = 0.3

    def buf(a=None):
        t = torch.full((n + offset + 8,), 7.0, dtype=torch.float32, device="cuda")
        if a is not None:
            t[offset:offset + n] = dev(a)
        return t, t[offset:offset + n]

    (_, xd), (_, yd), (m_all, m), (l_all, llr) = buf(x), buf(y), buf(), buf()
    q.qcldpc_bob_message(d, yd, dev(packed(bits.reshape(1, -1)).view(np.int32).reshape(-1)), n, m)
    q.qcldpc_llr(d, xd, m, n, snr, llr)
    torch.cuda.synchronize()
    m_gpu = m.cpu().numpy()
    m_ref = oracle.bob_message(y.astype(np.float64), bits, d=d)
    yb = np.repeat(np.linalg.norm(y.reshape(-1, d).astype(np.float64), axis=1), d)
    assert np.all(np.abs(m_gpu - m_ref) <= 16 * U32 * np.sqrt(d) * yb)
    ref = oracle.llr(x.astype(np.float64), m_gpu.astype(np.float64), snr, d=d)
    xb = np.repeat(np.linalg.norm(x.reshape(-1, d).astype(np.float64), axis=1), d)
    mb = np.repeat(np.linalg.norm(m_gpu.reshape(-1, d).astype(np.float64), axis=1), d)
    assert np.all(np.abs(llr.cpu().numpy() - ref) <= 16 * U32 * (2 * snr / d) * xb * mb + 2 * U32 * np.abs(ref))
    for t in (m_all, l_all):
        assert (t[:offset] == 7.0).all() and (t[offset + n:] == 7.0).all()


@pytest.mark.parametrize("fmt", [0, 1, 2])
@pytest.mark.parametrize("maker, Z", [
    (odd_code, 1), (odd_code, 5), (odd_code, 37), (synth.rate002_code, 31), (synth.rate002_code, 33),
    (synth.rate002_code, 127), (synth.rate002_code, 129), (synth.rate002_code, 257),
    (synth.rate005_code, 1023), (synth.rate010_code, 1025), (synth.rate002_code, 2049), (synth.met_code, 41),
])
def test_check_pass_forms_agree(maker, Z, fmt):
    """Key bits, flags and stop iterations are the same whether the check pass
    loads its operands directly or stages them (cn_threads above 128), with
    soft output or without, in one chain or two."""
    fr = make_frames(maker(Z), 0.12 if maker is synth.rate002_code else 0.3, 3, d=2)
    code = q.create_code_from(fr.code_dict)
    llr, syn = dev(fr.q64.astype(np.float32).reshape(-1)), dev(packed(fr.syn).view(np.int32).reshape(-1))
    for max_iter, et_start in ((0, 1), (1, 1), (12, 1), (12, 13), (9, 5)):
        out, post = [], []
        for soft, groups, cn in ((True, 0, 0), (True, 0, 160), (False, 0, 0), (False, 1, 0), (False, 1, 32),
                                 (False, 1, 160), (False, 2, 256)):
            p = q.qcldpc_params_init(msg_format=fmt, et_start=et_start, frame_groups=groups, cn_threads=cn)
            dec = q.Decoder(code, fr.F, p, soft=soft)
            dec.decode(llr, syn, max_iter)
            torch.cuda.synchronize()
            out.append((dec.keys.cpu(), dec.converged.cpu(), dec.iters.cpu()))
            post += [dec.posterior.cpu()] if soft else []
        assert torch.equal(post[0], post[1]), (max_iter, et_start)
        for i, o in enumerate(out[1:]):
            assert all(torch.equal(a, b) for a, b in zip(o, out[0])), (i, max_iter, et_start)


@pytest.mark.parametrize("fmt", [0, 1, 2])
def test_check_pass_forms_agree_on_full_grids(fmt):
    """24 frames at Z = 2049 fill the GPU: eight checks per lane, in one chain
    and in two, and the staged pass; random LLRs and syndromes."""
    code = q.create_code_from(synth.rate002_code(2049))
    F, g = 24, torch.Generator(device="cuda")
    g.manual_seed(5)
    llr = torch.randn(F * code.n, generator=g, device="cuda") * 0.5
    syn = torch.randint(-2 ** 31, 2 ** 31, (F * ((code.m + 31) // 32),), generator=g, device="cuda",
                        dtype=torch.int64).to(torch.int32)
    out = []
    for groups, cn in ((1, 0), (2, 0), (1, 160), (1, 256)):
        dec = q.Decoder(code, F, q.qcldpc_params_init(msg_format=fmt, frame_groups=groups, cn_threads=cn))
        dec.decode(llr, syn, 15)
        torch.cuda.synchronize()
        out.append((dec.keys.cpu(), dec.converged.cpu(), dec.iters.cpu()))
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(o, out[0]))


@pytest.mark.parametrize("maker, Z, groups", [
    (synth.rate002_code, 31, 0), (synth.rate002_code, 33, 0), (synth.rate002_code, 1025, 0), (odd_code, 5, 0),
    (odd_code, 37, 0), (synth.met_code, 41, 0),
])
def test_one_row_groups_match_the_oracle(maker, Z, groups):
    """Rows that meet each heavy column at most once update the posteriors in
    their check pass, the others in a pass of their own; both kinds occur."""
    fr = make_frames(maker(Z), 0.1, 2, d=2)
    code = q.create_code_from(fr.code_dict)
    iters = 6
    layer = oracle.row_layers(fr.code, fr.code.mb)
    _, conv, its, post = decode_soft(code, dev(fr.q64.astype(np.float32).reshape(-1)), fr.syn, fr.F, iters, et_start=iters + 1,
                                     schedule=1, layers=groups)
    for f in range(fr.F):
        ref, _, it, cv = oracle.decode_layered(fr.code, fr.q64[f], fr.syn[f], iters, layer, et_start=iters + 1)
        assert_posteriors_close(post[f], ref, f"Z {Z} frame {f}")
        assert its[f] == it and conv[f] == int(cv)
