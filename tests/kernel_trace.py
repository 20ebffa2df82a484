"""Which kernels a call launches, from a trace of the device's activity: name, grid, block, registers, shared memory."""
import json

from torch.profiler import ProfilerActivity, profile


def kernels(ffm, M, call, tmp_path):
    """The kernels of one call on matcher M, launched one by one (with the library's profile on, graphs are off)."""
    ffm.ff_profile_enable(M.ctx, True)
    for i in range(2):  # the first trace of a process may come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            M.sync()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        events = json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
        out = [(e["name"], e["args"]) for e in sorted((e for e in events if e.get("cat") == "kernel"),
                                                      key=lambda e: e["ts"])]
        if out:
            break
    ffm.ff_profile_enable(M.ctx, False)
    assert out, "no kernels in the trace"
    return out
