"""The channel of a generation call is the first c with u A_K < A_c, A the
sums of the weights in channel order: weights whose sum up to a channel equals
u A_K to the last bit tell an A_c that is one unit off."""
import numpy as np
import pytest

from test_gpu_pass_shapes import problem

pytestmark = pytest.mark.gpu
FIELD = 0x80000000


@pytest.mark.parametrize("K", [2, 24, 32, 33, 100, 300])
def test_channel_at_the_boundary(K):
    from oracle import oracle as O
    from paper_1811_09711_gb300 import vamp as V
    pr = problem(2, 4, K, [[]])
    g, o = V.Vamp(pr), O.Oracle(pr)
    rng = np.random.default_rng(K)
    for call in range(150):
        u = (float(o.eval_call(1, FIELD, call)["words"][pr.d]) + 0.5) * 2.0 ** -32
        at = int(rng.integers(1, K))  # the sum up to and with channel at - 1 will be u, the one of all 1
        a = rng.uniform(0.2, 1.0, K) * (rng.random(K) < 0.7)
        if at > 1:
            a[0] = 0.3
            a[:at - 1] *= u * rng.uniform(0.55, 0.95) / a[:at - 1].sum()
        A = 0.0
        for c in range(at - 1):
            A += a[c]
        a[at - 1] = u - A
        A += a[at - 1]
        a[at:] *= (1.0 - u) * rng.uniform(0.3, 0.9) / max(a[at:].sum(), 1e-9)
        for c in range(at, K - 1):
            A += a[c]
        a[K - 1] = 1.0 - A
        g.set_state(alpha=a)
        o.set_state(alpha=a)
        got, want = g.eval_calls(1, FIELD, call, 1, with_bins=False), o.eval_call(1, FIELD, call, with_bins=False)
        assert a[want["channel"]] > 0.0 and want["channel"] >= at
        assert got["channel"][0] == want["channel"], call
