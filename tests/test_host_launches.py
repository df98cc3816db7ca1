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


@pytest.mark.parametrize("call", ["lib.mc_sweep(b, 4, 1)", "lib.mc_group_sweep(g, 4, 1)", "lib.mc_group_sweep(p, 4, 1)"])
def test_sweeps_are_refused_on_a_capturing_stream(call):
    """Before a graph of theirs is recorded as well as after: nothing is launched or counted."""
    result = run(f"""
st = stream()
b = batch([mc.ising((64, 64), 0.44, 1)], st=st)
g, p = group([b], st), group([b], st)
assert lib.mc_group_configure(p, 4, 256, 0.0) == 0
out = []
for warm in range(3):
    launches()
    before = swept(b)
    assert fake.cudaStreamBeginCapture(st, 1) == 0
    status = {call}
    h = ctypes.c_void_p()
    fake.cudaStreamEndCapture(st, ctypes.byref(h))
    out.append([status, lib.mc_last_error().decode(), swept(b) - before, launches()])
    assert {call} == 0
result = [mc.MC_ECUDA, out]
""")
    for status, message, counted, log in result[1]:
        assert status == result[0] and "captured" in message
        assert counted == 0 and log == []


def test_host_counters_follow_what_was_launched():
    """A launch that fails in a later chunk, or in a later member of a group: the sweeps launched before are counted (the
    device's counter has advanced by them), those of the failed chunk are not, and nothing follows them."""
    result = run("""
b = batch([mc.ising((64, 64), 0.44, 1)])
lib.mc_set_mode(b, 1, 0)
fake.fake_fail_launch(2 * 256 + 1 + 5)        # within the second chunk
one = [lib.mc_sweep(b, 300, 1), swept(b)]
two = batch([mc.ising((64, 64), 0.44, 1)]), batch([mc.ising((128, 64), 0.44, 1)])
for c in two:
    lib.mc_set_mode(c, 1, 0)
g = group(two)
launches()
fake.fake_fail_launch(2 * 4 + 1 + 2)          # within the second member
st = lib.mc_group_sweep(g, 4, 1)
advanced = sum("k_advance" in e[0] for e in launches())
rec = (mc.mc_record * 4)()
n = ctypes.c_int64()
assert lib.mc_read_series(two[0], rec, 4, ctypes.byref(n)) == 0
result = [one, [st, swept(two[0]), swept(two[1]), advanced, n.value]]
""")
    assert result == [[-3, 256], [-3, 4, 0, 1, 4]]


def test_group_launches_what_its_split_cost_asks_for():
    """MC_GROUP_SIDE_BY_SIDE: the members' own kernels, and nothing of the persistent launch (no schedule, so that a cluster
    size the device cannot place does not matter).  MC_GROUP_FAIR_SHARE, anything below it and costs >= 0: one
    persistent kernel a call, also after a member's overrelaxation count has changed."""
    result = run("""
a = batch([mc.ising((64, 64), 0.44, 1)])
b = batch([mc.su2((4, 4, 4, 4), 2.3, 1)])
g = group([a, b])
nc, nr = ctypes.c_int32(), ctypes.c_int32()

def schedule():
    st = lib.mc_group_schedule(g, ctypes.byref(nc), ctypes.byref(nr))
    return [st, nc.value > 0, nr.value > 0]

def call(split, n=1):
    out = []
    for _ in range(n):
        launches()
        st = lib.mc_group_sweep(g, 2, 1)
        names = {e[0] for e in launches()} - {"wait", "graph", "end"}
        out.append([st, any("7k_groupE" in s for s in names), any("k_phase" in s for s in names)])
    return out

result = {}
for split in (-1.0, -0.5, mc.MC_GROUP_FAIR_SHARE, -9.0, 0.0, 1e300):
    assert lib.mc_group_configure(g, 4, 256, split) == 0
    before = schedule()
    result[str(split)] = [before, call(split, 2), schedule()]
assert lib.mc_group_configure(g, 4, 256, mc.MC_GROUP_FAIR_SHARE) == 0
assert lib.mc_su2_set_overrelax(b, 2) == 0
result["overrelax"] = call(-2.0, 2)
fake.fake_set_clusters(0)
result["no cluster"] = []
for split in (-1.0, -2.0):
    assert lib.mc_group_configure(g, 16, 256, split) == 0
    result["no cluster"].append(call(split))
""")
    ok = [0, True, True]
    for split in ("-1.0", "-0.5"):
        assert result[split] == [[0, False, False], [[0, False, True]] * 2, ok]
    for split in ("-2.0", "-9.0", "0.0", "1e+300"):
        assert result[split] == [[0, False, False], [[0, True, False]] * 2, ok]
    assert result["overrelax"] == [[0, True, False]] * 2
    assert result["no cluster"][0] == [[0, False, True]]
    assert result["no cluster"][1][0][0] == -3


@pytest.mark.parametrize("L,depth,pipe", [(8, 3, True), (8, 6, True), (10, 5, True), (6, 6, False), (2, 3, False), (8, 7, False)])
def test_sampler_rule(L, depth, pipe):
    """k_sample_pipe from L = 8 and for up to four hidden layers where it has exactly the registers its split is written
    for (a split of more than the launch's registers would wait for ever); else k_sample."""
    result = run(f"""
result = []
for regs in (128, 126):
    fake.fake_set_regs(regs)
    st, w = van({L}, 32, {depth})
    assert st == 0
    launches()
    assert lib.mc_van_sample(w, 32, 0, None, None, None) == 0
    result.append([e[0] for e in launches() if "k_sample" in e[0]])
""")
    assert [len(r) for r in result] == [1, 1]
    assert ["k_sample_pipe" in r[0] for r in result] == [pipe, False]
