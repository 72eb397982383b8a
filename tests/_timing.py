"""Device time of a call: graph replays, the fastest of several."""
import torch


def device_us(f, reps=10, rounds=7):
    """Microseconds of one f() among others, launches captured in a graph."""
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        f()  # allocates its workspace
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            for _ in range(reps):
                f()
        best = float("inf")
        for _ in range(rounds):
            graph.replay()
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record(side)
            for _ in range(3):
                graph.replay()
            end.record(side)
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 1e3 / (3 * reps))
    return best
