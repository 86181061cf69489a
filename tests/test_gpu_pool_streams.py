"""Pools whose step graphs run at the same time on streams of their own, as a
server steps them: together they fill the GPU many times over, and every frame
keeps the result of a decode alone."""
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1702_07740_gb300 import qcldpc as q  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device visible")
    q.load()


CODES = ((synth.rate002_code, 2000, 12), (synth.rate002_code, 513, 40), (synth.rate005_code, 3001, 16),
         (synth.rate010_code, 257, 60), (synth.rate010_code, 9999, 6), (synth.met_code, 100, 10),
         (synth.met_code, 31, 20), (synth.rate005_code, 64, 64))


@pytest.mark.parametrize("schedule, fmt", [(0, 0), (0, 1), (0, 2), (1, 0)])
def test_pools_stepped_side_by_side_decode_as_alone(schedule, fmt):
    """Random LLRs and syndromes: no frame converges, so every pass of every
    pool runs to the end (layered with 7 row groups)."""
    iters, g = 20, torch.Generator(device="cuda")
    g.manual_seed(3 + fmt)
    par = dict(schedule=schedule, layers=7 * schedule, msg_format=fmt)
    main = torch.cuda.current_stream()
    pools, streams = [], [torch.cuda.Stream() for _ in CODES]
    for maker, Z, F in CODES:
        code = q.create_code_from(maker(Z))
        llr = torch.randn(F * code.n, generator=g, device="cuda") * 0.5
        syn = torch.randint(-2 ** 31, 2 ** 31, (F * ((code.m + 31) // 32),), generator=g, device="cuda",
                            dtype=torch.int64).to(torch.int32)
        ids = torch.arange(F, dtype=torch.int32, device="cuda")
        pool = q.Pool(code, F, iters, q.qcldpc_params_init(**par))
        q.qcldpc_pool_load(pool, F, ids, llr, syn)
        pools.append((code, pool, F, ids, llr, syn))
    for _ in range(-(-(iters + 1) // 3)):
        start = torch.cuda.Event()
        start.record(main)
        for p, s in zip(pools, streams):
            s.wait_event(start)
            q.qcldpc_pool_step(p[1], 3, s)
        for s in streams:
            main.wait_stream(s)
    for code, pool, F, ids, llr, syn in pools:
        keys = torch.empty(F * ((code.k + 31) // 32), dtype=torch.int32, device="cuda")
        conv, its = (torch.full((F,), -2, dtype=torch.int32, device="cuda") for _ in range(2))
        q.qcldpc_pool_collect(pool, F, ids, keys, conv, its)
        alone = q.Decoder(code, F, q.qcldpc_params_init(**par))
        alone.decode(llr, syn, iters)
        torch.cuda.synchronize()
        assert torch.equal(keys, alone.keys) and torch.equal(conv, alone.converged) and torch.equal(its, alone.iters)
