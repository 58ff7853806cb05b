"""bench.py's byte count of an elementwise target's timed launch."""
import bench


def test_elementwise_launch_bytes():
    C, D, B, K = 100, 10, 50, 150
    row = 4.0 * C * D

    def rows(kernel="k_elementwise_chain", transitions=K, adapt=True, streaming=False, replicas=1):
        return bench.elementwise_launch_bytes(kernel, C, D, transitions, B, K, adapt, streaming, replicas) / row

    assert rows() == 4 + K                                  # the fixed range after an adapting burn-in
    assert rows(transitions=1) == 5                         # ... a launch per transition
    assert rows(adapt=False, transitions=B + K) == 4 + K    # burn-in in the same launch
    assert rows(streaming=True) == 14                       # no samples, five moments in and out
    assert rows(transitions=1, replicas=4) == 4             # samples are another kernel's
    assert rows(kernel="k_funnel_grad", transitions=0.1) == 2
    assert rows(kernel="k_std_normal_grad", transitions=0.1, streaming=True) == 2
