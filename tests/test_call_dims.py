"""The structure a call takes follows the workspace's memory and the stream, whatever was kept from earlier calls (CPU)."""
import pytest
import torch

from paper_2207_08393_b200 import binding

SHAPE = (2, 4, 1, 2, (1, 48, 40), 0, binding.GLEAM_MASK_FULL)


def fields(d):
    return {k: tuple(getattr(d, k)) if k == "n" else getattr(d, k) for k, _ in binding.gleam_dims._fields_}


def check(kept, ws, stream):
    d = kept.get(ws, stream)
    assert fields(d) == fields(binding.make_dims(*SHAPE, stream=stream, workspace=ws))
    return d


def test_a_kept_structure_is_found_again_and_follows_the_stream():
    kept, ws = binding.CallDims(*SHAPE), torch.zeros(4096, dtype=torch.uint8)
    assert check(kept, ws, 7) is check(kept, ws, 7)
    assert check(kept, ws, 9) is not check(kept, ws, 7)


def test_new_storage_of_the_same_tensor():
    kept, ws = binding.CallDims(*SHAPE), torch.zeros(4096, dtype=torch.uint8)
    first = check(kept, ws, 7).workspace
    ws.set_(torch.zeros(8192, dtype=torch.uint8))
    assert check(kept, ws, 7).workspace != first
    ws.resize_(1 << 20)
    assert check(kept, ws, 7).workspace_bytes == 1 << 20
    ws.resize_(1024)                                       # the same memory, less of it
    assert check(kept, ws, 7).workspace_bytes == 1024


def test_another_tensor_and_the_bound():
    kept = binding.CallDims(*SHAPE)
    a, b = torch.zeros(4096, dtype=torch.uint8), torch.zeros(4096, dtype=torch.uint8)
    for i in range(4 * kept.LIMIT):
        check(kept, a if i % 2 else b, i)
    assert len(kept._known) <= kept.LIMIT


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_the_undocumented_functions(monkeypatch, missing):
    class Stream:
        cuda_stream = 41
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.setattr(torch._C, name, lambda *a: 43, raising=False)
    assert binding._current_stream_handle() == 43
    monkeypatch.delattr(torch._C, missing)
    assert binding._current_stream_handle() == 41
