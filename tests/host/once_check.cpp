// Calls of once_per_device from a script on standard input: "device result" per line; prints
// for each whether the setting was made, and the value that came back.
#include <cstdio>

#include "once.h"

enum Err { OK = 0, FAILED = 7 };

int main() {
  static gbmg::DeviceSet done{0};
  int device, result;
  while (std::scanf("%d %d", &device, &result) == 2) {
    bool made = false;
    const Err e = gbmg::once_per_device(done, device, [&]() {
      made = true;
      return (Err)result;
    });
    std::printf("%d %d\n", made ? 1 : 0, (int)e);
  }
  return 0;
}
