"""Which k-NN kernel a call took, from the library's launch records."""
import torch


def knn_kernel(call):
    """The k-NN kernel that `call` launched ("k_knn": a thread per query, "k_knn_warp": a warp), and its result."""
    from paper_2112_06188_gb300 import capi
    torch.cuda.synchronize()
    capi.bdl_profile(1)
    got = call()
    torch.cuda.synchronize()
    names = [n for n in capi.bdl_profile_read() if n in ("k_knn", "k_knn_warp")]
    capi.bdl_profile(0)
    assert len(names) == 1, names
    return names[0], got


def crossing(f, q, k):
    """The most leading rows of q that the warp-per-query kernel takes."""
    lo, hi = 1, q.shape[0]
    assert knn_kernel(lambda: f.knn(q[:lo], k))[0] == "k_knn_warp"
    assert knn_kernel(lambda: f.knn(q, k))[0] == "k_knn"
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if knn_kernel(lambda: f.knn(q[:mid], k))[0] == "k_knn_warp":
            lo = mid
        else:
            hi = mid
    return lo
