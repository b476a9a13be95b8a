// Preloaded by tests/test_gpu_create_nomem.py: while armed, operator new
// refuses anything of 16 KB and more.
#include <cstdlib>
#include <new>

static bool armed = false;
extern "C" void new_fails(int on) { armed = on != 0; }

void* operator new(std::size_t n) {
  void* p = armed && n >= 16384 ? nullptr : std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
