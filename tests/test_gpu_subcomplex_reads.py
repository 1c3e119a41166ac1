"""AlphaComplex.subcomplex has read the context when it returns, so that a build on another stream may follow at once:
with the current stream held up before every list is copied, the stream is idle when the call returns, and the rows and
values are those of an undisturbed call although the context was built again on another stream."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_a_build_on_another_stream_may_follow(monkeypatch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    c, r = synth.globule(47, 6000, probe=False)
    cx = ac.AlphaComplex(torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda(), 1.0).build()
    want = cx.subcomplex(0.5)
    torch.cuda.synchronize()
    current = ac._current_stream

    def held_up(t, index):
        t.cuda._sleep(10_000_000)  # about 5 ms of the current stream
        return current(t, index)

    other = torch.cuda.Stream()
    monkeypatch.setattr(ac, "_current_stream", held_up)
    got = cx.subcomplex(0.5)
    assert torch.cuda.current_stream().query(), "the reads of the context were still to come"
    cx.build(stream=other)
    for (rows, f), (rows0, f0) in zip(got, want):
        assert torch.equal(rows, rows0) and torch.equal(f, f0)
