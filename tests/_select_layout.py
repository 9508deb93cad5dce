"""Where the selection kernels' shares lie (a replay of the dispatch and of the share layouts of csrc/onela_select.cu), so that a
test can crowd candidates into few shares and see on the host that more of them reach the bound than shared memory holds."""
import numpy as np

LIST = 4096          # candidates that reach the bound: room in shared memory


def kernel_of(n: int, k: int) -> str:
    """'one' (one CTA, shares of neighbours), 'cluster' (a cluster, spread shares) or 'threads' (a cluster's own threads)."""
    if n > (16384 if k <= 256 else 32768) and n >= 48 * k:
        return "one" if k <= 256 else "cluster"
    return "threads"


def shares(n: int, k: int) -> np.ndarray:
    """Share of every candidate."""
    i = np.arange(n)
    kind = kernel_of(n, k)
    if kind == "one":
        return i // (64 if n > 262144 else 16)
    if kind == "cluster":
        o = i % 16384
        return i // 16384 * 1024 + (o % 1024 - o // 1024 * 977) % 1024
    span = 1024 * (1 if n <= 4096 else 2 if n <= 32768 else 4 if n <= 65536 else 8)
    return (i % span - i // span * 977) % span


def crowd(n: int, k: int) -> np.ndarray:
    """Candidates of the first k - 1 shares: raised above all others, every one of them reaches any bound that k shares reach."""
    return shares(n, k) < k - 1


def reaching(scores: np.ndarray, k: int) -> int:
    """Candidates that reach the k-th largest of the shares' largest (the kernels' bound leaves these, or a few more)."""
    s = shares(scores.size, k)
    largest = np.full(s.max() + 1, -np.inf, dtype=scores.dtype)
    np.maximum.at(largest, s, scores)
    return int((scores >= np.sort(largest)[-k]).sum())
