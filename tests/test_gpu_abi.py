"""Pointer ownership at the C ABI on a GPU: buffers that are not memory of
the current device (page-locked or pageable host memory) are refused with
APC_EINVAL before anything is enqueued, so the caller's output is left as it
was."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # the CUDA path has no fallback: without a GPU these tests cannot run
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_18178_gb300 as apc  # noqa: E402

N = 4096
SENTINEL = 0x5A5A5A5A


def _device_set():
    d = {k: torch.zeros(N, dtype=torch.float32, device="cuda") for k in "pmv"}
    d["g"] = torch.zeros(N, dtype=torch.int16, device="cuda")
    d["w"] = torch.zeros(N, dtype=torch.int16, device="cuda")
    return d


def _refused(call):
    with pytest.raises(apc.ApcError) as ei:
        call()
    assert ei.value.status == 1, ei.value
    return str(ei.value)


def test_host_pointers_are_refused_before_launch():
    d = _device_set()
    out = torch.full((8,), SENTINEL, dtype=torch.int64, device="cuda")
    pinned = torch.zeros(N, dtype=torch.float32).pin_memory()
    pageable = np.zeros(N, dtype=np.float32)
    for bad in (pinned.data_ptr(), pageable.ctypes.data):
        for field in "pmvgw":
            e = dict(d)
            e[field] = bad
            msg = _refused(lambda: apc.commit_step([apc.TensorEntry(e["p"], e["m"], e["v"], e["g"], e["w"], 0,
                                                                    n=N)], 1, out=out[:4]))
            assert "table[0].%s" % field in msg
        _refused(lambda: apc.digest([apc.BufferEntry(bad, 0, 0, apc.F32, n=N)], 1, out=out[4:5]))
        _refused(lambda: apc.count_nonzero([apc.BufferEntry(bad, 0, 0, apc.F32, n=N)], 1, out=out[5:6]))
    host_out = torch.zeros(4, dtype=torch.int64).pin_memory()
    msg = _refused(lambda: apc.commit_step([apc.TensorEntry(d["p"], d["m"], d["v"], d["g"], d["w"], 0)], 1,
                                           out=host_out.data_ptr()))
    assert "out_digests" in msg
    _refused(lambda: apc.digest(apc.state_buffers(d["p"], d["m"], d["v"], d["w"]), 4, out=host_out.data_ptr()))
    torch.cuda.synchronize()
    assert out.cpu().tolist() == [SENTINEL] * 8      # nothing was zeroed or launched
    assert int(host_out.abs().sum()) == 0


def test_device_pointers_still_pass():
    d = _device_set()
    out = apc.commit_step([apc.TensorEntry(d["p"], d["m"], d["v"], d["g"], d["w"], 0)], 1)
    ver = apc.digest(apc.state_buffers(d["p"], d["m"], d["v"], d["w"]), 4)
    assert apc.digests_to_host(out) == apc.digests_to_host(ver)


def test_output_overlapping_a_buffer_is_refused():
    d = _device_set()
    _refused(lambda: apc.commit_step([apc.TensorEntry(d["p"], d["m"], d["v"], d["g"], d["w"], 0)], 1,
                                     out=d["m"][8:16].view(torch.int64)))
    _refused(lambda: apc.digest(apc.state_buffers(d["p"], d["m"], d["v"], d["w"]), 4,
                                out=d["v"][:8].view(torch.int64)))


@pytest.mark.parametrize("where", ["arena", "interleaved", "separate"])
def test_pointer_ranges_of_long_tables(where):
    """Tables long enough for the checks by allocation: buffers of each kind in
    an arena of their own, all kinds interleaved in one arena, or an allocation
    each.  A host pointer or an overlap anywhere in them is still refused, the
    same table without it still commits."""
    n, k = 264, 40
    if where == "separate":
        get = lambda f, i: torch.zeros(300_000 if i % 7 == 0 else n, dtype=torch.float32 if f in "pmv" else torch.int16,
                                       device="cuda")[:n]
    elif where == "arena":
        arena = {f: torch.zeros(n * k, dtype=torch.float32 if f in "pmv" else torch.int16, device="cuda") for f in "pmvgw"}
        get = lambda f, i: arena[f][i * n:(i + 1) * n]
    else:
        flat = torch.zeros(k * 4 * n, dtype=torch.float32, device="cuda")

        def get(f, i):
            at = (k - 1 - i) * 4 * n + "pmvgw".index(f) * n
            t = flat[at:at + n] if f in "pmv" else flat[at - (n // 2 if f == "w" else 0):][:n // 2].view(torch.int16)
            return t
    e = [apc.TensorEntry(*(get(f, i) for f in "pmvgw"), i * n) for i in range(k)]
    out = torch.full((4,), SENTINEL, dtype=torch.int64, device="cuda")
    pinned = torch.zeros(n, dtype=torch.float32).pin_memory()
    for i, f in ((0, "p"), (17, "v"), (k - 1, "w")):
        bad = [apc.TensorEntry(t.p, t.m, t.v, t.g, t.w, t.global_offset) for t in e]
        setattr(bad[i], f, pinned.data_ptr())
        bad[i].n = n
        assert "table[%d].%s" % (i, f) in _refused(lambda: apc.commit_step(bad, 1, out=out))
        bad[i] = apc.TensorEntry(e[i].p, e[i].m, e[i].v, e[i].g, e[i].w, 0)
        setattr(bad[i], f, getattr(e[(i + 5) % k], f))
        assert "overlap" in _refused(lambda: apc.commit_step(bad, 1, out=out))
    assert out.cpu().tolist() == [SENTINEL] * 4
    apc.commit_step(e, 1, out=out)
    ver = apc.digest([b for t in e for b in apc.state_buffers(t.p, t.m, t.v, t.w, t.global_offset)], 4)
    assert apc.digests_to_host(out) == apc.digests_to_host(ver)
