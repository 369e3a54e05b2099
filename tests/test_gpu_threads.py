"""Plans solved from several host threads at once, each on its own stream (the foreign call
gives up the interpreter lock, so the launches interleave)."""
import threading

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes,dtype", [([(24, 24, 1000), (24, 24, 200)], "f32"),
                                          ([(24, 24, 1000), (24, 24, 200)], "f64"),
                                          ([(60, 60, 10), (50, 50, 10), (54, 60, 10)], "f32")])
def test_threads_of_different_sizes(shapes, dtype):
    """Plans of different sizes share kernels but not their shared memory (the z pass of 1000
    points takes 144 KB, that of 200 points 54 KB; plane kernels of 60 x 60 and 50 x 50): a
    launch must not meet the limit that another thread set for a smaller one, and every solve
    gives the bits of one made alone."""
    torch = pytest.importorskip("torch")
    from paper_1612_01799_gb300 import Plan, build
    build.build()
    plans, rhos, refs, outs = [], [], [], []
    for n in shapes:
        p = Plan(n, tuple(0.5 * q for q in n), 1e-6 if dtype == "f32" else 1e-12, dtype)
        if dtype == "f64":
            p.arith = "df"
        torch.manual_seed(sum(n))
        r = torch.rand(n[2], n[1], n[0], dtype=p.torch_dtype, device="cuda")
        plans.append(p)
        rhos.append(r)
        refs.append(p.solve(r))
        outs.append(torch.empty_like(r))
    torch.cuda.synchronize()
    errors, gate = [], threading.Barrier(len(plans))

    def work(i):
        s = torch.cuda.Stream()
        try:
            gate.wait(60)
            for _ in range(1500):
                plans[i].solve(rhos[i], out=outs[i], stream=s)
            s.synchronize()
        except Exception as e:
            errors.append((shapes[i], repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(plans))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    torch.cuda.synchronize()
    for r, o in zip(refs, outs):
        assert torch.equal(r, o)
    for p in plans:
        p.close()
