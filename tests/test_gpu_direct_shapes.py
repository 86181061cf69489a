"""The check pass that loads its operands directly, over every row shape it has
and at lifting sizes around its tiles (32 lanes, 2 and 8 checks per lane),
against the FP64 oracle and against the staged pass."""
import numpy as np
import pytest

import oracle
from frames import make_frames

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402
from test_gpu_parity import assert_posteriors_close, dev, packed  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


SHAPES = ((1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (4, 1))


def shapes_code(Z, copies=2):
    """`copies` rows of each shape (heavy, degree-1 circulants); heavy circulants
    on four columns, from Z = 2 on some rows meet one of them twice."""
    rng = np.random.default_rng(Z)
    ents, col = [], 4
    for r, (nh, nd) in enumerate(SHAPES * copies):
        cols = rng.choice(4, nh, replace=False)
        if Z > 1 and nh > 1 and r % 2:
            cols[1] = cols[0]
        shifts = rng.choice(Z, nh, replace=Z < nh)
        if nh > 1 and cols[0] == cols[1] and shifts[0] == shifts[1]:
            shifts[1] = (shifts[1] + 1) % Z
        ents += [(r, int(c), int(s)) for c, s in zip(cols, shifts)]
        if nd:
            ents.append((r, col, int(rng.integers(Z))))
            col += 1
    row, cl, sh = (np.array(v) for v in zip(*ents))
    mb = len(SHAPES) * copies
    return dict(mb=mb, nb=max(col, mb) + 2, Z=Z, row=row, col=cl, shift=sh)


def takes_direct_pass(d):
    """Every row has at most four heavy and one degree-1 circulants, at least
    one of each kind or two heavy ones."""
    deg = np.bincount(d["col"], minlength=d["nb"])[d["col"]]
    nh, nd = (np.bincount(d["row"][m], minlength=d["mb"]) for m in (deg > 1, deg == 1))
    return bool(np.all(((nd == 1) & (nh >= 1) & (nh <= 4)) | ((nd == 0) & (nh >= 2) & (nh <= 4))))


def outputs(code, F, llr, syn, iters, soft, **params):
    dec = q.Decoder(code, F, q.qcldpc_params_init(**params), soft=soft)
    dec.decode(llr, syn, iters)
    torch.cuda.synchronize()
    return [dec.keys.cpu(), dec.converged.cpu(), dec.iters.cpu()] + ([dec.posterior.cpu()] if soft else [])


ZS = [1, 2, 5, 31, 32, 33, 37, 63, 64, 65, 95, 127, 129, 255, 256, 257, 1000, 1025]


@pytest.mark.parametrize("Z", ZS)
def test_every_row_shape_matches_the_oracle(Z):
    d = shapes_code(Z)
    assert takes_direct_pass(d)
    fr = make_frames(d, 0.4, 2, d=1)
    code, iters = q.create_code_from(d), 6
    llr, syn = dev(fr.q64.astype(np.float32).reshape(-1)), dev(packed(fr.syn).view(np.int32).reshape(-1))
    post = outputs(code, 2, llr, syn, iters, True, et_start=iters + 1)[3].numpy().reshape(2, -1)
    for f in range(2):
        ref, _, _, _ = oracle.decode(fr.code, fr.q64[f], fr.syn[f], iters, et_start=iters + 1)
        assert_posteriors_close(post[f], ref, f"Z {Z} frame {f}")


@pytest.mark.parametrize("fmt", [0, 1, 2])
@pytest.mark.parametrize("Z", ZS)
def test_direct_and_staged_passes_agree(Z, fmt):
    """cn_threads above 128 takes the staged pass. Three frames run two checks
    per lane; with 24 copies of each shape 70 frames fill the GPU and run eight."""
    for copies, F in ((2, 3), (24, 70)):
        d = shapes_code(Z, copies)
        assert takes_direct_pass(d)
        code = q.create_code_from(d)
        g = torch.Generator(device="cuda")
        g.manual_seed(Z)
        llr = torch.randn(F * code.n, generator=g, device="cuda") + 0.6
        syn = torch.randint(-2 ** 31, 2 ** 31, (F * ((code.m + 31) // 32),), generator=g, device="cuda",
                            dtype=torch.int64).to(torch.int32)
        for iters, et_start in ((1, 1), (7, 1), (7, 8)):
            par = dict(msg_format=fmt, et_start=et_start)
            ref = outputs(code, F, llr, syn, iters, True, cn_threads=256, **par)
            for soft, extra in ((True, {}), (False, {}), (False, dict(frame_groups=1, cn_threads=64))):
                got = outputs(code, F, llr, syn, iters, soft, **par, **extra)
                assert all(torch.equal(a, b) for a, b in zip(got, ref)), (copies, iters, et_start, soft, extra)
