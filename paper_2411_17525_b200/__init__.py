"""B200 (sm_100a) implementation of the HIGGS quantized linear layer.

The product is the CUDA shared library built from ``csrc/`` behind the C ABI of
``include/higgs.h``; this package is its ctypes binding (``binding.py``), whose
names are re-exported here on first use.  Using any of them fails loudly when the
library has not been built (``python -m paper_2411_17525_b200.build``): there is
no fallback path.
"""
import importlib
import types

_BINDING = None
_TAKEN = {}          # callables of the binding that are attributes of the package by now


class _Binding(types.ModuleType):
    """The binding's module: replacing one of its names takes what the package took over back, so it shows through the package."""

    def __setattr__(self, name, value):
        super().__setattr__(name, value)
        _forget()

    def __delattr__(self, name):
        super().__delattr__(name)
        _forget()


def _forget():
    while _TAKEN:
        name, value = _TAKEN.popitem()
        if globals().get(name) is value:          # (not what a caller has set on the package itself)
            del globals()[name]


def __getattr__(name):
    global _BINDING
    if name.startswith("__"):
        raise AttributeError(name)
    if _BINDING is None:
        _BINDING = importlib.import_module(".binding", __name__)
        _BINDING.__class__ = _Binding
    try:
        value = getattr(_BINDING, name)
    except AttributeError:
        raise AttributeError(f"module {__name__!r} has no attribute {name!r}") from None
    if callable(value):
        globals()[name] = _TAKEN[name] = value          # found directly from now on (this hook takes 0.3 us)
    return value
