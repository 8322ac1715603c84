"""Launch graphs of repeated host calls into pageable memory: a replay's result is the device
call's, and keys that do not come back, or more keys in turn than graphs are kept, cost no
captures."""
import numpy as np
import pytest

from paper_1810_11359_gb300 import ism

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, T, TDIFF = 16000.0, 0.2, 0.1


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _room(i):
    L = [3.2 + 0.01 * i, 3.7, 2.9]
    return (L, [0.8, 0.7, 0.75, 0.8, 0.6, 0.7]), (ism.ism_nb_img_from_t(TDIFF, L, 343.0, 4e-3), T, FS)


def _positions(rng, n_rcv=2):
    return (rng.uniform(0.4, 2.4, (n, 3)).astype(np.float32) for n in (1, n_rcv))


def test_replay_with_new_positions_equals_the_device_call():
    rng = np.random.default_rng(5)
    ws, (walls, sizes) = ism.Workspace(), _room(0)
    out = np.empty((1, 2, ism.ism_rir_length(T, FS)), np.float32)
    before = ism.ism_launch_graph_counts()[1]
    for _ in range(100):   # (longer than any graph of other calls is kept against this one's)
        ps, pr = _positions(rng)
        out[:] = np.nan
        ism.ism_simulate_host(*walls, ps, pr, *sizes, Tdiff=TDIFF, seed=7, out=out, workspace=ws)
        dev = ism.ism_simulate(*walls, torch.from_numpy(ps).cuda(), torch.from_numpy(pr).cuda(), *sizes, Tdiff=TDIFF, seed=7)
        assert np.array_equal(dev.cpu().numpy().view(np.uint32), out.view(np.uint32))
    assert ism.ism_launch_graph_counts()[1] > before + 20


def test_keys_that_come_three_times_are_not_captured():
    rng = np.random.default_rng(6)
    ps, pr = _positions(rng)
    before = ism.ism_launch_graph_counts()
    for i in range(20):
        walls, sizes = _room(100 + i)
        for _ in range(3):
            ism.ism_simulate_host(*walls, ps, pr, *sizes, Tdiff=TDIFF)
    assert ism.ism_launch_graph_counts() == before


def test_more_keys_in_turn_than_graphs():
    """20 rooms in turn: 16 graphs, captured once, and then replayed for as long as it goes on."""
    rng = np.random.default_rng(7)
    ps, pr = _positions(rng)
    rooms = [_room(200 + i) for i in range(20)]
    c0 = ism.ism_launch_graph_counts()[0]
    for cycle in range(16):
        r0 = ism.ism_launch_graph_counts()[1]
        for walls, sizes in rooms:
            ism.ism_simulate_host(*walls, ps, pr, *sizes, Tdiff=TDIFF)
    c1, r1 = ism.ism_launch_graph_counts()
    assert c1 - c0 == 16 and r1 - r0 == 16
