"""Names of the kernels that a call enqueues, in order of first appearance: the
call is captured into a CUDA graph (which runs nothing) and the graph is
written out as text."""
import gc
import re
import warnings


def kernels(torch, stream, call, path):
    """call() enqueues on `stream` only; its tables and buffers must be there
    already (make the same call uncaptured before)."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    torch.cuda.synchronize()
    gc.collect()  # lattices of earlier tests free their buffers, which ends a capture
    gc.disable()
    try:
        with torch.cuda.graph(g, stream=stream):
            call()
    finally:
        gc.enable()
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        g.debug_dump(str(path))
    names = {}
    for mangled in re.findall(r"_ZN\w+", path.read_text()):
        for m in re.finditer(r"\d+", mangled):  # <length><identifier>
            for k in range(m.start(), m.end()):
                name = mangled[m.end():m.end() + int(mangled[k:m.end()])]
                if name.endswith("_kernel") and name.isidentifier() and len(name) == int(mangled[k:m.end()]):
                    names[name] = None
    return list(names)
