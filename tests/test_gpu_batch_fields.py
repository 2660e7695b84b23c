"""Fields that the batched product cannot use where they are: at addresses no
kernel may read floats from, and outputs that share memory (needs a GB300)."""
import numpy as np
import pytest

from synth import damage_snapshot, random_field

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = [(8, 6), (10, 4, 6), (12, 18), (8, 6)]


@pytest.fixture()
def batch():
    from paper_2207_10657_gb300 import Phase, RVEBatch, build
    build.build()
    pms = [(np.random.default_rng(i).random(tuple(reversed(d))) < 0.3).astype(np.uint8) for i, d in enumerate(DIMS)]
    b = RVEBatch(DIMS, pms, [Phase(1.0, 0.3, True, 1e-4, 1e-3), Phase(10.0, 0.2)])
    for i, pm in enumerate(pms):
        b.set_damage(i, torch.from_numpy(damage_snapshot(pm, dmax=0.9, seed=i)).float().cuda())
    vs = [torch.from_numpy(random_field(6 if len(d) == 3 else 3, d, seed=i)).float().cuda()
          for i, d in enumerate(DIMS)]
    yield b, vs, b.hessp(vs)
    b.close()


@pytest.mark.parametrize("shift", [1, 2, 4])
def test_fields_at_any_address(batch, shift):
    from paper_2207_10657_gb300 import binding as B
    b, vs, want = batch

    def shifted(t):
        raw = torch.zeros(4 * t.numel() + 16, dtype=torch.uint8, device="cuda")
        raw[shift:shift + 4 * t.numel()] = t.reshape(-1).view(torch.uint8)
        return raw
    ins, outs = [shifted(v) for v in vs], [shifted(torch.zeros_like(v)) for v in vs]
    B.rve_batch_hessp(b.h, [t.data_ptr() + shift for t in ins], [t.data_ptr() + shift for t in outs])
    for o, w in zip(outs, want):
        got = o[shift:shift + 4 * w.numel()].clone().view(torch.float32).reshape(w.shape)
        assert torch.equal(got, w)


def test_outputs_that_share_memory_are_written_in_order(batch):
    from paper_2207_10657_gb300 import binding as B
    b, vs, want = batch
    scratch = torch.empty(max(v.numel() for v in vs), device="cuda")
    B.rve_batch_hessp(b.h, [v.data_ptr() for v in vs], [scratch.data_ptr()] * len(vs))
    assert torch.equal(scratch[:want[-1].numel()].reshape(want[-1].shape), want[-1])


def test_product_under_capture(batch):
    """The look at the pointers is legal while the stream captures."""
    from paper_2207_10657_gb300 import Phase, RVEBatch
    from paper_2207_10657_gb300 import binding as B
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    pm = (np.random.default_rng(0).random((6, 8)) < 0.3).astype(np.uint8)
    b = RVEBatch([(8, 6)], [pm], [Phase(1.0, 0.3), Phase(10.0, 0.2)], stream=st)
    v = torch.from_numpy(random_field(3, (8, 6), seed=0)).float().cuda()
    want = b.hessp([v])[0]
    out = torch.zeros_like(v)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        B.rve_batch_hessp(b.h, [v.data_ptr()], [out.data_ptr()])
    torch.cuda.synchronize()
    assert not out.any()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    b.close()
