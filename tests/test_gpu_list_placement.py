"""Which list placement ordered queries for k > 16 use and report: one set on
the tree, never one tuned for the state machine."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kdt():
    from paper_2210_12859_gb300 import build

    build.build_library()
    from paper_2210_12859_gb300 import kdt as k

    return k


@pytest.mark.parametrize("placement", ["GLOBAL", "GROUP4", "GROUP8"])
def test_tuned_placement(kdt, tmp_path, placement):
    tuned = getattr(kdt, "KDT_LIST_" + placement)

    def load(value):
        path = tmp_path / "t.json"
        gpu = torch.cuda.get_device_name()
        path.write_text('[\n  {"gpu": "%s", "D": 2, "k_bucket": 5, "log2n": 9, "stage_levels": 0, "claim_steps": 64, '
                        '"inline_depth": 2, "light_run": 1, "large_k_list": %d}\n]\n' % (gpu, value))
        kdt.kdt_tuning_load(str(path))

    g = torch.Generator(device="cuda").manual_seed(9)
    tree = kdt.kdt_build(torch.rand((700, 2), generator=g, device="cuda"))
    q = torch.rand((300, 2), generator=g, device="cuda")
    want = kdt.kdt_knn(tree, q, 30)
    load(tuned)
    try:
        assert kdt.kdt_large_k_list(tree, 30) == kdt.KDT_LIST_SHARED
        for flags in (0, kdt.KDT_UNORDERED):
            got = kdt.kdt_knn(tree, q, 30, flags=flags)
            assert torch.equal(got[0], want[0]) and torch.equal(got[1].view(torch.int32), want[1].view(torch.int32))
        kdt.kdt_set_large_k_list(tree, tuned)
        assert kdt.kdt_large_k_list(tree, 30) == tuned
        assert torch.equal(kdt.kdt_knn(tree, q, 30)[0], want[0])
    finally:
        load(kdt.KDT_LIST_SHARED)


def test_ordered_autotune_takes_no_light_run(kdt):
    """Ordered calls are judged by their counts of processed nodes, whose
    kernel has no light runs: none may be picked by noise (and then slow down
    unordered queries)."""
    g = torch.Generator(device="cuda").manual_seed(10)
    q = torch.rand((2000, 3), generator=g, device="cuda")
    tree = kdt.kdt_build(torch.rand((611, 3), generator=g, device="cuda"))
    for _ in range(20):
        kdt.kdt_autotune(tree, q, 3, 0)
        assert kdt.kdt_tuned_params(tree, 3)[3] == 1
