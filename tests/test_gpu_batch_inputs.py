"""Batched calls on inputs that need no conversion and on inputs that do
(wider types, host memory, other strides and shapes) give the same results,
and refuse the same ones."""
import numpy as np
import pytest
import torch

from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


FORMS = {
    "as is": lambda t: t,
    "int64": lambda t: t.long(),
    "host": lambda t: t.cpu(),
    "numpy": lambda t: t.cpu().numpy(),
    "strided": lambda t: t.repeat_interleave(2, 0)[::2],
    "flat": lambda t: t.reshape(-1),
    "parameter": lambda t: torch.nn.Parameter(t, requires_grad=False),
}


@pytest.mark.parametrize("form", sorted(FORMS))
def test_forms(form):
    from paper_2112_06188_gb300.forest import Forest, erase_batch, insert_batch, knn_batch
    to = FORMS[form]
    pts = [torch.from_numpy(inputs.uniform_points(n, d, n)).cuda() for n, d in ((3_000, 2), (0, 2), (700, 3))]
    fs, ref = ([Forest(p.shape[1]) for p in pts] for _ in range(2))
    got = insert_batch(fs, [to(p) for p in pts])
    for f, p, i in zip(ref, pts, got):
        assert torch.equal(f.insert(p), i)
    gone = [i[::3].contiguous() for i in got]
    assert erase_batch(fs, [to(g) for g in gone]) == [f.erase(g) for f, g in zip(ref, gone)]
    q = [p[:50].contiguous() for p in pts]
    for (a, b), f, x in zip(knn_batch(fs, [to(x) for x in q], 4), ref, q):
        c, d = f.knn(x, 4)
        assert torch.equal(a, c) and torch.equal(b, d)


def test_refusals():
    from paper_2112_06188_gb300.forest import Forest, insert_batch, knn_batch
    f = Forest(2)
    p = torch.from_numpy(inputs.uniform_points(100, 2, 1)).cuda()
    insert_batch([f], [p])
    ok = (torch.empty((100, 3), dtype=torch.int32, device="cuda"), torch.empty((100, 3), dtype=torch.int64, device="cuda"))
    for bad in ((ok[0][:99], ok[1]), (ok[1], ok[1]), (ok[0], ok[0]), (ok[0], ok[1].t().contiguous().t()),
                (ok[0].cpu(), ok[1]), (ok[0], ok[1].cpu())):
        with pytest.raises(ValueError):
            knn_batch([f], [p], 3, out=[bad])
    with pytest.raises((TypeError, ValueError)):
        insert_batch([f], [p.float()])
    with pytest.raises(ValueError):
        insert_batch([f], [p.long() + (1 << 32)])
    knn_batch([f], [p], 3, out=[ok])
    assert np.array_equal(ok[0][:, 0].cpu().numpy(), np.arange(100))
