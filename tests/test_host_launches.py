"""What the library's host code launches, with the CUDA runtime replaced by a stand-in (no GPU)."""
import pytest

from host_runtime import run

CHAINS = {
    "int8": "batch([mc.ising((64, 64), 0.44, 1), mc.ising((620, 170), 0.4, 2)])",
    "int8_runs": "batch([mc.ising((2000, 1100), 0.44, 1)])",
    "msc": "batch([mc.ising((256, 64), 0.44, 1)], layout=1)",
    "su2": "batch([mc.su2((4, 4, 4, 4), 2.3, 1)])",
}


@pytest.mark.parametrize("kind", list(CHAINS))
def test_first_kernel_of_a_chunk_starts_after_the_advance(kind):
    """The sweep kernels read the run state before they wait for their predecessor, so the first kernel after the one
    that advances it (between the chunks of a call, and between calls) must not start early; the others are chained."""
    log = run(f"""
b = {CHAINS[kind]}
assert lib.mc_set_mode(b, 1, 0) == 0
launches()
assert lib.mc_sweep(b, 300, 3) == 0      # 255 and 45 sweeps, launched one by one
assert lib.mc_sweep(b, 7, 0) == 0
result = launches()
""")
    runs, state_changed = [], True
    for entry in log:
        if entry[0] in ("wait", "graph", "end"):
            continue
        if "k_advance" in entry[0]:
            state_changed = True
        else:
            if state_changed:
                runs.append([])
            runs[-1].append(entry[3])
            state_changed = False
    assert len(runs) == 3
    for r in runs:
        assert r[0] == "plain"
        assert set(r[1:]) == {"programmatic"}
