"""What the tensor-core kernels wait for when they give up (csrc/tc05.cuh ring_drain, csrc/flow_tile.cuh pair_drain): the
last fill of every stage of a ring has landed, for every number of fills, whichever of the copies have.  The wait's
stage and parity expressions are taken from the sources and run against barriers as PTX defines them: a wait for parity
p passes when the phase of parity p before the current one has completed, and the first phase has parity 0."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_19048_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _expressions():
    """(parity of stage i from next and phase; next and phase after n fills of two slots; of one slot)."""
    ring = re.search(r"void ring_drain\(.*?\{(.*?)\n\}", _read("tc05.cuh"), re.S).group(1)
    lt, ge = re.search(r"\(uint32_t\)i < next \? (.*?) : (.*?), limit", ring).groups()
    tile = _read("flow_tile.cuh")
    pair = re.search(r"ring_drain\(full, 2, (.*?), (.*?), limit\)", tile).groups()
    one = re.search(r"ring_drain\(rg\.full \+ 2, 1, 0u, (.*?), F_WAIT\)", tile).group(1).replace("rg.fills[1]", "n")
    py = lambda e: re.sub(r"(\d)u\b", r"\1", e)  # noqa: E731
    return py(lt), py(ge), [py(e) for e in pair], py(one)


class Barrier:
    def __init__(self):
        self.completed = 0

    def passes(self, parity):   # the phase before the current one is `completed - 1`; before any, it has parity 1
        return (self.completed - 1) & 1 == parity


@pytest.mark.parametrize("stages", [1, 2, 3, 4, 6, 8])
def test_drain_waits_for_the_last_fill_of_every_stage(stages):
    lt, ge, pair, one = _expressions()
    for fills in range(5 * stages + 1):
        nxt, phase = fills % stages, 1 - (fills // stages) % 2   # the producer's stage and parity, flipped at each wrap
        if stages == 2:
            assert (eval(pair[0], {"n": fills}), eval(pair[1], {"n": fills})) == (nxt, phase)
        if stages == 1:
            assert eval(one, {"n": fills}) == phase
        for i in range(stages):
            mine = fills // stages + (1 if i < nxt else 0)
            parity = eval(lt if i < nxt else ge, {"phase": phase})
            landed, flying = Barrier(), Barrier()
            landed.completed, flying.completed = mine, mine - 1
            assert landed.passes(parity)
            assert mine == 0 or not flying.passes(parity)


def test_every_kernel_with_a_ring_drains_it():
    for unit in ("k_gemm.cu", "k_flow_train.cu", "flow_tile.cuh"):
        s = _read(unit)
        for m in re.finditer(r"atomicExch\((&g_gemm_status|&g_train_status|status), 1\);\n(.*?)tcgen05\.dealloc", s, re.S):
            body = m.group(2)
            if "fwd_drain(rg)" in body:
                body = re.search(r"void fwd_drain\(.*?\n\}", s, re.S).group(0)
            assert re.search(r"(ring|pair)_drain\(", body) and "mma_drain(" in body and "__syncthreads()" in body
    assert len(re.findall(r"mma_drain\(&", "".join(_read(u) for u in ("k_gemm.cu", "k_flow_train.cu", "flow_tile.cuh")))) == 3
