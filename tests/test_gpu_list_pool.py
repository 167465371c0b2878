"""Lists built and freed one after another re-use device memory of their context's pool.

Results must not depend on what a block held before, a list may outlive its context and the
stream it was built on, and lists of several threads share no block.
"""

from __future__ import annotations

import threading

import numpy as np
import pytest

from synth import fcc_box, make_model, water_box

pytestmark = pytest.mark.gpu


def _evaluate(pot, s, times=1):
    import torch

    sy = pot.system(s.pos, s.species, s.cell)
    for _ in range(times):
        sy.evaluate(virial=True)
    sy.check()
    out = float(sy.energy), sy.forces.cpu().numpy().copy(), sy.virial.cpu().numpy().copy()
    sy.close()
    return out


def _same(a, b):
    return a[0] == b[0] and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_reused_memory_gives_the_same_results():
    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=3)
    boxes = [water_box(64, seed=1), fcc_box(8, seed=2), water_box(400, seed=3), fcc_box(3, seed=4)]
    alone = []
    for s in boxes:
        pot = Potential(spec)
        alone.append(_evaluate(pot, s))
        pot.close()
    pot = Potential(spec)
    for order in ([0, 1, 2, 3], [3, 2, 1, 0], [2, 0, 3, 1]):
        for k in order:
            assert _same(_evaluate(pot, boxes[k]), alone[k]), k
    pot.close()


def test_list_outlives_its_context_and_stream():
    import torch

    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=2)
    s = water_box(100, seed=5)
    other = Potential(spec)
    want = _evaluate(other, s)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        pot = Potential(spec, stream=stream)
        sy = pot.system(s.pos, s.species, s.cell)
    pot.close()
    del stream
    sy.pot = other  # evaluate the list on another context
    sy.evaluate(virial=True)
    sy.check()
    assert _same((float(sy.energy), sy.forces.cpu().numpy(), sy.virial.cpu().numpy()), want)
    sy.close()
    other.close()


@pytest.mark.parametrize("close_first", [False, True])
def test_captured_calls_belong_to_their_context(close_first):
    # a list's replayed rebuild, evaluation, host callback and MD step hold their context's weights
    import torch

    from paper_2505_06711_gb300 import Potential
    from synth import MASS_AMU, maxwell_boltzmann

    s = water_box(64, seed=6)
    mass = torch.as_tensor(MASS_AMU[s.species], device="cuda")
    vel0 = torch.as_tensor(maxwell_boltzmann(MASS_AMU[s.species], 300.0, seed=1), device="cuda")

    def calls(sy, host, vel):
        e, f = np.zeros(1), np.zeros((s.n_atoms, 3), np.float32)
        pos0 = sy.pos.clone()
        for _ in range(3):  # direct, captured, replayed
            sy.rebuild()
            sy.evaluate(virial=True)
            sy.evaluate_host(host, e, f, rebuild=True)
        out = [x.cpu().numpy().copy() for x in (sy.energy, sy.forces, sy.virial)] + [e.copy(), f.copy()]
        for _ in range(2):
            sy.pos.copy_(pos0)
            vel.copy_(vel0)
            e_pot, e_kin = sy.md(vel, mass, 0.25, 6)
            out += [x.cpu().numpy().copy() for x in (e_pot, e_kin, sy.pos)]
        sy.check()
        sy.pos.copy_(pos0)
        return out

    first, second = (Potential(make_model(T=2, seed=k)) for k in (11, 12))
    sy = second.system(s.pos, s.species, s.cell)
    want = calls(sy, s.pos, vel0.clone())
    sy.close()
    sy = first.system(s.pos, s.species, s.cell)
    vel = vel0.clone()
    other = calls(sy, s.pos, vel)
    assert not np.array_equal(other[0], want[0])
    if close_first:
        first.close()
    sy.pot = second
    got = calls(sy, s.pos, vel)
    for k, (x, y) in enumerate(zip(got, want)):
        assert np.array_equal(x, y), k
    sy.close()
    first.close()
    second.close()


def test_lists_refuse_models_they_were_not_sized_for():
    import torch

    from paper_2505_06711_gb300 import Potential, binding

    s = water_box(32, seed=7)  # elements 0 and 1
    pot = Potential(make_model(T=2))
    sy = pot.system(s.pos, s.species, s.cell)
    sy.evaluate()
    vel, mass = torch.zeros_like(sy.pos), torch.ones(s.n_atoms, dtype=torch.float64, device="cuda")
    e, f = np.zeros(1), np.zeros((s.n_atoms, 3), np.float32)
    for spec in (make_model(T=2, pairs=True), make_model(T=2, n_elem=1), make_model(T=3)):
        other = Potential(spec)
        sy.pot = other
        for call in (lambda: sy.evaluate(), lambda: sy.evaluate(virial=True), lambda: sy.evaluate_host(s.pos, e, f),
                     lambda: sy.md(vel, mass, 0.25, 1)):
            with pytest.raises(binding.ReannError) as err:
                call()
            assert err.value.code == binding.REANN_E_MISMATCH
        other.close()
    fits = Potential(make_model(T=2, n_elem=2))  # the elements that the list holds
    sy.pot = fits
    sy.evaluate()
    sy.check()
    sy.close()
    fits.close()
    pot.close()


def test_threads_build_and_free_together():
    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=2)
    boxes = [water_box(50 + 13 * k, seed=k) for k in range(4)]
    pot = Potential(spec)
    want = [_evaluate(pot, s) for s in boxes]
    pot.close()
    bad = []

    def work(k):
        import torch

        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            mine = Potential(spec, stream=stream)
            for _ in range(6):
                got = _evaluate(mine, boxes[k], 4)  # direct, captured, replayed: while others free
                if not _same(got, want[k]):
                    bad.append(k)
            mine.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_freeing_while_another_thread_captures():
    # freeing a list must neither invalidate the capture nor keep the list's memory
    import torch

    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=3)
    s = fcc_box(20, seed=8)  # 32,000 atoms: about 0.4 GB in blocks of the pool and larger ones
    warm = Potential(spec)
    _evaluate(warm, fcc_box(3, seed=4))
    warm.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    pot = Potential(spec)
    sy = pot.system(s.pos, s.species, s.cell)
    sy.evaluate()
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    begun, freed, errors = threading.Event(), threading.Event(), []
    graph = torch.cuda.CUDAGraph()

    def capture():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                graph.capture_begin(capture_error_mode="thread_local")
                x.add_(1.0)
                begun.set()
                freed.wait(60)
                x.mul_(2.0)
                graph.capture_end()
        except Exception as exc:  # pragma: no cover - the fault this test is for
            errors.append(exc)
            begun.set()

    t = threading.Thread(target=capture)
    t.start()
    begun.wait(60)
    sy.close()
    freed.set()
    t.join()
    assert not errors, errors
    graph.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 2000.0
    pot.close()
    del sy, graph, x
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] >= before - (64 << 20)


def test_freeing_behind_work_in_flight():
    # nothing waits on the host between a list's work, its release and the next list in the same blocks
    import torch

    from paper_2505_06711_gb300 import Potential
    from synth import MASS_AMU

    spec = make_model(T=3)
    boxes = [water_box(400, seed=9), fcc_box(7, seed=10)]
    pot = Potential(spec)

    def run(s, steps):
        sy = pot.system(s.pos, s.species, s.cell)
        mass = torch.as_tensor(MASS_AMU[s.species], device="cuda")
        vel = torch.zeros_like(sy.pos)
        sy.evaluate(virial=True)
        e_pot, _ = sy.md(vel, mass, 0.25, steps)
        sy.evaluate()
        out = e_pot, sy.energy, sy.forces, sy.virial, sy.pos
        sy.close()
        return out

    want = []
    for s in boxes:
        got = run(s, 40)
        torch.cuda.synchronize()
        want.append([t.cpu().numpy() for t in got])
    got = [run(s, 40) for _ in range(4) for s in boxes]
    for k, g in enumerate(got):
        assert all(np.array_equal(t.cpu().numpy(), w) for t, w in zip(g, want[k % 2])), k
    pot.close()


def test_list_in_a_callers_graph():
    # replays of a caller's own graph are not known to the list: freeing it waits for the device
    import torch

    from paper_2505_06711_gb300 import Potential

    spec = make_model(T=2)
    s = water_box(300, seed=11)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        pot = Potential(spec, stream=stream)
        want = _evaluate(pot, s)
        sy = pot.system(s.pos, s.species, s.cell)
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        graph.capture_begin(capture_error_mode="thread_local")
        sy.evaluate()
        graph.capture_end()
        for _ in range(20):
            graph.replay()
        energy, forces = sy.energy, sy.forces
        sy.close()
        other = pot.system(s.pos[::-1].copy(), s.species[::-1].copy(), s.cell)
        other.evaluate()
        torch.cuda.synchronize()
        assert float(energy) == want[0] and np.array_equal(forces.cpu().numpy(), want[1])
        other.close()
        pot.close()


def test_edge_records_leave_room():
    # with little device memory left a list keeps fewer edge records: its later calls, and others, find room, and
    # the results are the same
    import torch

    from paper_2505_06711_gb300 import Potential
    from synth import MASS_AMU

    spec = make_model(T=2)
    s = fcc_box(24, seed=12)  # 55,296 atoms, about 0.25 GB of edge records
    mass = torch.as_tensor(MASS_AMU[s.species], device="cuda")

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    def calls(sy):
        out = []
        for _ in range(3):
            sy.evaluate(virial=True)
        out += [x.cpu().numpy().copy() for x in (sy.energy, sy.forces, sy.virial)]
        e, f = np.zeros(1), np.zeros((s.n_atoms, 3), np.float32)
        sy.evaluate_host(s.pos, e, f)
        e_pot, _ = sy.md(torch.zeros_like(sy.pos), mass, 0.25, 3)
        sy.check()
        return out + [e, f, e_pot.cpu().numpy()]

    for _ in range(2):  # (the first list also loads the kernels)
        pot = Potential(spec)
        start = free()
        sy = pot.system(s.pos, s.species, s.cell)
        used = start - free()
        want = calls(sy)
        sy.close()
        pot.close()
    pot = Potential(spec)
    fill = torch.empty(free() - used - (40 << 20), dtype=torch.uint8, device="cuda")
    try:
        sy = pot.system(s.pos, s.species, s.cell)
        left = free()
        print(f"[room] used {used >> 20} MiB, left {left >> 20} MiB")
        assert left >= 100 << 20
        for k, (x, y) in enumerate(zip(calls(sy), want)):
            assert np.array_equal(x, y), k
        sy.close()
    finally:
        del fill
        torch.cuda.empty_cache()
        pot.close()
