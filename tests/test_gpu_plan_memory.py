"""Plans give back all of their device memory: forty made and destroyed one after the
other leave no less free than the first one did (a megabyte or two of driver slack)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision,survey", [(800, "f32", False), (512, "f32", False), (192, "f64", False),
                                                (100, "f32", False), (480, "f32", True)])
def test_destroyed_plans_leave_nothing(N, precision, survey):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1712_05834_gb300 as pk
    pk.build()

    def once():
        if survey:
            cfg = pk.make_survey_config(1000.0, (0.0, 0.0, 0.0), N, "tsc", True, dk=0.01, omega_m=0.31, zmax=1.0,
                                        capacity=1000)
            pk.ConvolvedFFTPower(cfg).close()
        else:
            pk.pk_destroy(pk.pk_plan(pk.make_config(1000.0, N, "tsc", interlaced=True, dk=0.01, nmu=5, precision=precision,
                                                    capacity=1000)))
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    once()
    before = once()
    for _ in range(40):
        after = once()
    assert before - after < 4 << 20, before - after
