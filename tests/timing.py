"""Device times of calls for the tests that compare two of them: both sides of a comparison run in
the same process on the same GPU, so that a bound on their ratio needs no absolute figure."""
import torch


def best_us(fn, calls=20, reps=5):
    """Smallest time of one fn() in us, from a CUDA graph of `calls` of them."""
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()  # the inputs were made on another stream
    with torch.cuda.stream(stream):
        fn()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(calls):
                fn()
    best = float("inf")
    for _ in range(reps + 2):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        graph.replay()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1) * 1e3 / calls)
    return best


def assert_at_most(fn, other, factor, what):
    """fn() takes at most `factor` times as long as other(), in one of three attempts."""
    seen = []
    for _ in range(3):
        seen.append((best_us(fn), best_us(other)))
        if seen[-1][0] <= factor * seen[-1][1]:
            return
    raise AssertionError(f"{what}: {seen} us, allowed {factor}x")
