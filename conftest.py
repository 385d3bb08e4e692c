import pytest


def pytest_configure(config):
    if "s" not in config.option.reportchars:   # a skipped test states its reason
        config.option.reportchars += "s"


@pytest.fixture(scope="session", autouse=True)
def blas_workspaces_first(request):
    """torch keeps the workspace of its first matrix product on a stream for good.  Made between two tests it may lie
    in the freed block of a large one (51.5 GB after n = 15), which can then not be given back, and the n = 16 test
    finds too little memory: 243.7 of 292.1 GB, whatever the library holds."""
    if any(item.get_closest_marker("gpu") for item in request.session.items):
        import torch
        if torch.cuda.is_available():
            for dtype in (torch.complex128, torch.float64, torch.float32, torch.bfloat16):
                a = torch.ones((64, 64), dtype=dtype, device="cuda")
                a @ a
    yield
