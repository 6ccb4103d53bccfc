"""Counts whose independent passes run on the calling thread's side streams: several threads with graphs of their
own, handles taken in turn by one thread, batches captured in between."""
import threading

import pytest

import graphgen
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRAPHS = [graphgen.ba(2000, 4, 1), graphgen.rmat(11, 12, seed=2), graphgen.er(5000, 14.0, 3), graphgen.ba(300, 9, 4)]


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_12074_gb300 import harp as H
    H.lib()
    return H, [O.count4_combo(g.n, g.src, g.dst).tolist() for g in GRAPHS]


def test_threads_and_handles_in_turn(setup):
    H, want = setup
    wrong = []

    def work(k):
        own = [H.harp_build_csr(GRAPHS[i].n, GRAPHS[i].src, GRAPHS[i].dst) for i in (k, (k + 1) % 4)]
        for turn in range(40):
            i = turn % 2
            if H.harp_count4(own[i]).tolist() != want[(k + i) % 4]:
                wrong.append((k, turn))
            if turn % 10 == 9:
                b = H.harp_batch_create(own)
                if H.harp_batch_count(b).tolist() != [want[k], want[(k + 1) % 4]]:
                    wrong.append((k, "batch"))
                b.close()
        for g in own:
            g.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
